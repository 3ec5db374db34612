"""Operators called with the output buffer equal to the input buffer give the bits of the call into a
buffer of its own (the kernels of one call read a cell's input from several blocks)."""
import numpy as np
import pytest

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _problem(dim, n_rhs):
    """Cells of several 64-node blocks and 32-output tiles each; n_rhs body loads."""
    rng = np.random.default_rng(n_rhs)
    loads = [W.Load(W.LOAD_BODY, tuple(rng.standard_normal(dim))) for _ in range(n_rhs)]
    if dim == 2:
        p = W.lattice_2d(5, 3, 11, a=0.2, r=0.12, n_rb=2)
        p.loads = loads
        return p
    return W.lattice_3d(3, 2, 2, e=5, r=0.2, r_spread=0.05, seed=3, n_rb=3, mask_kind=W.MASK_BCC_SIGMOID, loads=loads)


def _vector(*shape):
    return torch.randn(*shape, generator=torch.Generator(device="cuda").manual_seed(7), dtype=torch.float64,
                       device="cuda")


@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n_rhs", [1, 9])
def test_cell_stiffness_in_place_and_overlapping(dim, n_rhs):
    from paper_2308_11371_gb300 import binding
    s = binding.Solver(_problem(dim, n_rhs))
    u = _vector(s.n_rhs, s.N, s.n_dof)
    want = s.apply_K(u)
    for _ in range(5):
        y = u.clone()
        assert torch.equal(s.apply_K(y, out=y), want)
    buf = torch.zeros(u.numel() + 3, dtype=torch.float64, device="cuda")   # output three entries further on
    buf[:-3] = u.ravel()
    s.apply_K(buf[:-3].view_as(u), out=buf[3:].view_as(u))
    assert torch.equal(buf[3:].view_as(u), want)


@pytest.mark.parametrize("options", [dict(method=1), dict(), dict(precision=1)], ids=["standard", "rom", "rom_mixed"])
@pytest.mark.parametrize("dim", [2, 3])
@pytest.mark.parametrize("n_rhs", [1, 9])
def test_local_solve_and_preconditioner_in_place(options, dim, n_rhs):
    """Standard FETI-DP (one inverse per cell, several output blocks) and the reduced-order local solve,
    alone and as part of the block preconditioner, whose local solve runs beside the inner PCG."""
    from paper_2308_11371_gb300 import binding
    s = binding.Solver(_problem(dim, n_rhs), **options)
    for name, x in (("local_rom_solve", _vector(s.n_rhs, s.N, s.n_r)), ("apply_P", _vector(s.n_rhs, s.n_tot))):
        want = getattr(s, name)(x)
        for _ in range(3):
            y = x.clone()
            assert torch.equal(getattr(s, name)(y, out=y), want), name


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("n_rhs", [1, 9])
@pytest.mark.parametrize("shift", [0, 1, 40])
def test_coarse_solve_in_place_and_overlapping(precision, n_rhs, shift):
    """The stored inverse (FP64) and the block factors (mixed), output `shift` entries after the input."""
    from paper_2308_11371_gb300 import binding
    s = binding.Solver(_problem(3, n_rhs), precision=precision)
    b = _vector(s.n_rhs, s.n_P)
    want = s.coarse_solve(b)
    for lo, hi in ((0, shift), (shift, 0)):
        buf = torch.zeros(b.numel() + shift, dtype=torch.float64, device="cuda")
        src, dst = (buf[o:o + b.numel()].view_as(b) for o in (lo, hi))
        src.copy_(b)
        s.coarse_solve(src, out=dst)
        assert torch.equal(dst, want)
