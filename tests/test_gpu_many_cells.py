"""Lattices of more cells than one grid dimension of 65,535 blocks spans.

Strips of identical 2 x 2-element cells, clamped along their long side: the reduced model of one principal
cell reproduces every cell, so the projection of each, the last columns of the trace contraction included,
is 1 up to the rounding of its traces (sums of at most 160 terms: far below 1e-9)."""
import numpy as np
import pytest

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _projections(ny, precision):
    from paper_2308_11371_gb300 import binding
    p = W.lattice_2d(100_000, ny, 2, r=0.3, n_rb=1)
    p.clamp_axis = 1
    s = binding.Solver(p, precision=precision, restart=2)
    _, alpha, pi, delta = s.rom_data()
    y = s.apply_F(torch.ones(1, s.L, dtype=torch.float64, device="cuda"))
    assert bool(torch.isfinite(y).all())
    s.close()
    return alpha, pi, delta


def test_fp64_traces_of_a_million_cells():
    from paper_2308_11371_gb300 import binding
    for a in _projections(11, binding.FETIDP_FP64):
        assert np.abs(a - 1.0).max() < 1e-9


def test_mixed_traces_of_two_million_cells():
    from paper_2308_11371_gb300 import binding
    for a in _projections(22, binding.FETIDP_MIXED_BF16):
        assert np.abs(a - 1.0).max() < 1e-9
