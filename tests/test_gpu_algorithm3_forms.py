"""The two FP64 forms of Algorithm 3's products with U_id_ring: assembled per cell up to 8 GiB
(N n_i n_d of 16 bytes), combined from the principal operators at every use above."""
import numpy as np
import pytest

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n_rhs", [1, 2])
def test_assembled_and_combined_forms_agree(n_rhs):
    """A lattice of 17 x 17 cells of 32^2 elements (n_i = 1,922, n_d = 248: 2.2 GB, assembled) against four
    copies of it in a batch (8.8 GB, combined).  The copies add no direction to the greedy basis and take
    the lattice's own coefficients, so every copy's part of P x is the lattice's P x, up to the inner
    tolerance (1e-11) and the traces' rounding behind the Gram solves (1e-9 in the projection tests)."""
    from paper_2308_11371_gb300 import binding
    rng = np.random.default_rng(n_rhs)
    p = W.lattice_2d(17, 17, 32, a=0.3, r=0.12, r_grade=0.04, n_rb=3)
    p.loads = [W.Load(W.LOAD_BODY, tuple(rng.standard_normal(2))) for _ in range(n_rhs)]
    one, four = binding.Solver(p, restart=2), binding.Solver([p] * 4, restart=2)
    assert list(one.rom_data()[0]) == list(four.rom_data()[0])
    x = torch.as_tensor(rng.standard_normal((n_rhs, one.n_tot)), device="cuda")
    parts = torch.split(x, [one.N * one.n_r, one.n_P, one.L], dim=1)
    launches, out = [], []
    for s, v in ((one, x), (four, torch.cat([q.repeat(1, 4) for q in parts], 1))):
        s.profile_enable(["grouped_gemm"])
        out.append(s.apply_P(v))
        launches.append(s.profile_read()["grouped_gemm"]["launches"])
    # the local bases of Eq. 46a, and in the combined form the two products with U_rd_ring
    assert launches == [1, 3]
    want = torch.split(out[0], [one.N * one.n_r, one.n_P, one.L], dim=1)
    got = torch.split(out[1], [4 * one.N * one.n_r, 4 * one.n_P, 4 * one.L], dim=1)
    for w, g in zip(want, got):
        g = g.view(n_rhs, 4, -1)
        assert float((g - w[:, None]).abs().max()) < 1e-8 * float(w.abs().max())
