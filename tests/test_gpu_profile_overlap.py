"""Class times are the kernels' own: no launch's event pair covers another class's work."""
import numpy as np
import pytest

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_class_times_add_up_to_at_most_the_solve(prec):
    """The coarse correction runs beside the F_dd product and the local solve beside the inner PCG; timed
    like that, short kernels would count the time they wait for SMs and the sum would exceed the solve.
    2% are left for the resolution of the events (0.5 us each)."""
    from paper_2308_11371_gb300 import binding
    cells = (6, 4, 4) if prec == "fp64" else (16, 8, 8)
    rng = np.random.default_rng(3)
    loads = [W.Load(W.LOAD_BODY, tuple(rng.standard_normal(3))) for _ in range(6)]
    p = W.lattice_3d(*cells, e=6, r=0.2, r_spread=0.05, seed=3, n_rb=8, mask_kind=W.MASK_BCC_SIGMOID, loads=loads)
    s = binding.Solver(p, precision=binding.FETIDP_FP64 if prec == "fp64" else binding.FETIDP_MIXED_BF16)
    want, _, info0 = s.solve()
    s.profile_enable()
    t0, t1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
    t0.record()
    u, _, info = s.solve()
    t1.record()
    torch.cuda.synchronize()
    prof = s.profile_read()
    assert torch.equal(u, want) and info["inner_its_total"] == info0["inner_its_total"]
    assert sum(v["ms"] for v in prof.values()) <= 1.02 * t0.elapsed_time(t1)
