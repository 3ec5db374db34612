"""Algorithmic bytes that the profiler charges for the maps of the resident-operator path."""
import pytest

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_rb", [2, 3])
def test_resident_operator_maps_are_charged_as_fp32(n_rb):
    """M_D of a 2D mixed context: the gather writes FP32 columns, the principal groups (two each) leave FP32
    partial sums, their reduction FP32 results, which the scatter reads."""
    from paper_2308_11371_gb300 import binding
    s = binding.Solver(W.lattice_2d(6, 5, 8, a=0.2, r=0.12, r_grade=0.04, n_rb=n_rb),
                       precision=binding.FETIDP_MIXED_BF16)
    s.profile_enable(["maps"])
    s.precond(torch.ones(1, s.L, dtype=torch.float64, device="cuda"))
    p = s.profile_read()["maps"]
    cells, groups = s.N * s.n_d, (s.n_rb + 1) // 2
    gather = 8 * s.L + 4 * cells + 8 * cells
    reduce = 4 * cells * (groups + 1)
    scatter = 8 * s.L + 4 * cells + 8 * s.L
    assert p["launches"] == 3 and p["bytes"] == gather + reduce + scatter
