"""Per-cell operator kernels at the sizes where their tilings change, against the FP64 CPU oracle.

Tolerances are those of the operator parity tests (quantities behind a dense factorisation 1e-9,
pure applications of a Dirichlet operator 1e-11): the kernels only order the sums differently.
"""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2308_11371_gb300 import workloads as W

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _rel(a, b):
    a, b = np.asarray(a), np.asarray(b)
    return np.abs(a - b).max() / max(np.abs(b).max(), 1e-300)


def _dev(x):
    return torch.as_tensor(np.ascontiguousarray(x), dtype=torch.float64, device="cuda")


def _loads(dim, count):
    rng = np.random.default_rng(count)
    return [W.Load(W.LOAD_BODY, tuple(rng.standard_normal(dim))) for _ in range(count)]


def _problem(kind, n_rhs):
    if kind == "2d_e3":     # n_d = 16: one narrow tile; n_p = 8
        p = W.lattice_2d(3, 2, 3, a=0.2, r=0.2, n_rb=2)
        p.loads = _loads(2, n_rhs)
    elif kind == "2d_e9":   # n_d = 64: two full tiles of 32 outputs
        p = W.lattice_2d(2, 2, 9, a=0.2, r=0.12, n_rb=2)
        p.loads = _loads(2, n_rhs)
    else:                   # n_d = 270, n_r = 351: a ragged last tile; n_p = 24
        p = W.lattice_3d(2, 2, 1, e=4, r=0.2, r_spread=0.05, seed=3, n_rb=3, mask_kind=W.MASK_BCC_SIGMOID,
                         map_kind=W.MAP_SHEAR_BEND_3D, map_params=(0.3, 2.0, 0.1, -0.15), loads=_loads(3, n_rhs))
    return p


_ORACLE = {}


def _oracle(kind):
    if kind not in _ORACLE:
        from oracle import feti_dp, ifeti_dp
        from oracle.discretization import Lattice
        lat = Lattice(_problem(kind, 1))
        blocks = [feti_dp.CellBlocks(lat, s) for s in range(lat.N)]
        _ORACLE[kind] = ifeti_dp.InexactFETIDP(lat, blocks=blocks)
    return _ORACLE[kind]


@pytest.mark.parametrize("kind", ["2d_e3", "2d_e9", "3d_e4"])
@pytest.mark.parametrize("n_rhs", [1, 2, 3, 4, 5, 6, 7, 8, 11])
def test_fp64_cell_operators_for_every_rhs_count(kind, n_rhs):
    from paper_2308_11371_gb300 import binding
    ref = _oracle(kind)
    s = binding.Solver(_problem(kind, n_rhs))
    rng = np.random.default_rng(n_rhs)
    lam = rng.standard_normal((s.n_rhs, s.L))
    y, z = s.apply_F(_dev(lam)).cpu().numpy(), s.precond(_dev(lam)).cpu().numpy()
    for r in range(n_rhs):
        assert _rel(y[r], ref.apply_F(lam[r])) < 1e-9
        assert _rel(z[r], ref.apply_MD(lam[r])) < 1e-11


@pytest.mark.parametrize("cells", [(4, 3), (8, 3), (11, 3), (13, 5)])
def test_fp64_principal_contractions_at_each_column_tile(cells):
    """12, 24, 33 and 65 columns: the 16-, 32- and 64-wide tiles and their remainders, the trace tiles
    and theirs.  Projections against the oracle, then Eq. 46a-b."""
    from oracle import feti_dp, ifeti_dp
    from oracle.discretization import Lattice
    from paper_2308_11371_gb300 import binding
    p = W.lattice_2d(cells[0], cells[1], 8, a=0.3, r=0.12, r_grade=0.03, n_rb=3)
    lat = Lattice(p)
    ref = ifeti_dp.InexactFETIDP(lat, blocks=[feti_dp.CellBlocks(lat, s) for s in range(lat.N)])
    s = binding.Solver(p)
    sigma, alpha, pi, delta = s.rom_data()
    assert list(sigma) == list(ref.rom.sigma)
    assert _rel(pi, ref.rom.pi) < 1e-9 and _rel(delta, ref.rom.delta) < 1e-9
    v = np.random.default_rng(1).standard_normal((s.n_rhs, s.N, s.n_r))
    x = s.local_rom_solve(_dev(v)).cpu().numpy()
    assert _rel(x[0], ref.rom.local_rom_solve(v[0])) < 1e-9


@pytest.mark.parametrize("cells", [(3, 2, 2), (13, 13, 13)])
def test_identical_cells_converge_in_one_outer_iteration_fp64(cells):
    """Identical cells make the reduced model exact, so the block preconditioner of Eq. 44 is the inverse
    and FGMRES needs one iteration (a second only to confirm).  2,197 cells of 6^3 elements are above the
    size up to which U_id_ring is assembled: both forms of Algorithm 3 are covered."""
    from paper_2308_11371_gb300 import binding
    p = W.lattice_3d(*cells, e=6, r=0.2, n_rb=1, mask_kind=W.MASK_BCC_SIGMOID)
    s = binding.Solver(p)
    u, lam, info = s.solve()
    assert info["n_rb"] == 1 and info["outer_its"] <= 2 and info["rel_residual"] < 1e-8


@pytest.mark.parametrize("kind", ["2d_e3", "2d_e9", "3d_e4"])
@pytest.mark.parametrize("n_rhs", [1, 4, 8, 9, 11])
def test_cell_stiffness_and_saddle_operator_for_every_vector_group(kind, n_rhs):
    """1-8 vectors per thread group; 9 and 11 make uneven groups.  Natural order (apply_K) and the split
    remaining / corner views (apply_A) against the oracle's assembled K_s: only the order of sums differs."""
    from paper_2308_11371_gb300 import binding
    ref = _oracle(kind)
    s = binding.Solver(_problem(kind, n_rhs))
    rng = np.random.default_rng(n_rhs)
    u = rng.standard_normal((s.n_rhs, s.N, s.n_dof))
    y = s.apply_K(_dev(u)).cpu().numpy()
    for c in range(s.N):
        assert _rel(y[:, c], u[:, c] @ ref.lat.stiffness(c).T) < 1e-12
    x = rng.standard_normal((s.n_rhs, s.n_tot))
    z = s.apply_A(_dev(x)).cpu().numpy()
    for r in range(n_rhs):
        assert _rel(z[r], ref.A(x[r])) < 1e-12


@pytest.mark.parametrize("kind,copies", [("3d_e4", 1), ("3d_e4", 3), ("3d_e4", 5)])
@pytest.mark.parametrize("n_rhs", [1, 2, 3, 4, 5, 6, 7, 8, 11])
def test_fp32_cell_operators_for_every_rhs_count_and_block_width(kind, copies, n_rhs):
    """Mixed path on 2 x 2 x 1 lattices batched 1, 3 and 5 times (4 to 20 cells with n_d = 270: lanes of 1,
    and lanes of 4 with a lattice of 216 cells below), every interleave of the right-hand sides.  The FP32
    operators carry ~6e-8 per entry and an FP32 sum of 270 terms: 1e-5 relative covers both."""
    from paper_2308_11371_gb300 import binding
    ref = _oracle(kind)
    probs = [_problem(kind, n_rhs) for _ in range(copies)]
    s = binding.Solver(probs, precision=binding.FETIDP_MIXED_BF16)
    f = binding.Solver(probs)
    rng = np.random.default_rng(n_rhs)
    lam = _dev(rng.standard_normal((s.n_rhs, s.L)))
    assert _rel(s.apply_F(lam).cpu(), f.apply_F(lam).cpu()) < 1e-5
    assert _rel(s.precond(lam).cpu(), f.precond(lam).cpu()) < 1e-5
    if copies == 1:
        y = s.apply_F(lam).cpu().numpy()
        assert max(_rel(y[r], ref.apply_F(lam[r].cpu().numpy())) for r in range(n_rhs)) < 1e-5


@pytest.mark.parametrize("cells,n_rhs", [((6, 6, 6), 3), ((7, 5, 4), 1), ((5, 3, 5), 6)])
def test_fp32_cell_operators_on_wider_blocks(cells, n_rhs):
    """216, 140 and 75 cells of n_d = 270: blocks of 4, 4 and 2 outputs per lane against the FP64 path."""
    from paper_2308_11371_gb300 import binding
    p = W.lattice_3d(*cells, e=4, r=0.2, r_spread=0.05, seed=3, n_rb=3, mask_kind=W.MASK_BCC_SIGMOID,
                     loads=_loads(3, n_rhs))
    s, f = binding.Solver(p, precision=binding.FETIDP_MIXED_BF16), binding.Solver(p)
    lam = _dev(np.random.default_rng(2).standard_normal((s.n_rhs, s.L)))
    assert _rel(s.apply_F(lam).cpu(), f.apply_F(lam).cpu()) < 1e-5
    assert _rel(s.precond(lam).cpu(), f.precond(lam).cpu()) < 1e-5


@pytest.mark.parametrize("precision", [0, 1])
def test_unsynchronised_calls_on_a_stream_and_in_a_graph_match_checked_calls(precision):
    """F_ring runs a branch on the context's own stream: back-to-back calls without input checks on a
    non-default stream, and the same calls captured into a graph and replayed, give the bits of checked
    calls one at a time."""
    from paper_2308_11371_gb300 import binding
    p = _problem("3d_e4", 3)
    s = binding.Solver(p, precision=precision)
    gen = torch.Generator(device="cuda").manual_seed(5)
    lams = [torch.randn(s.n_rhs, s.L, generator=gen, dtype=torch.float64, device="cuda") for _ in range(6)]
    want = [(s.apply_F(x).clone(), s.precond(x).clone()) for x in lams]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        a = binding.Solver(p, precision=precision, check_inputs=0)
        outs = [(torch.empty_like(x), torch.empty_like(x)) for x in lams]
        for _ in range(10):
            for x, (y, z) in zip(lams, outs):
                a.apply_F(x, y)
                a.precond(x, z)
        stream.synchronize()
        for (y, z), (yw, zw) in zip(outs, want):
            assert torch.equal(y, yw) and torch.equal(z, zw)
            y.zero_(), z.zero_()
        graph = torch.cuda.CUDAGraph()
        stream.synchronize()
        with torch.cuda.graph(graph, stream=stream):
            for x, (y, z) in zip(lams, outs):
                a.apply_F(x, y)
                a.precond(x, z)
        for _ in range(3):
            graph.replay()
    torch.cuda.synchronize()
    for (y, z), (yw, zw) in zip(outs, want):
        assert torch.equal(y, yw) and torch.equal(z, zw)


@pytest.mark.parametrize("n_rhs", [1, 3, 9])
@pytest.mark.parametrize("kind,copies", [("2d_e9", 1), ("3d_e4", 1), ("3d_e4", 3)])
def test_dense_and_block_coarse_solves_agree(kind, copies, n_rhs):
    """The FP64 context keeps S_PP^{-1} (n_P <= 1,024), the mixed one the FP64 block factors of the same
    matrix up to its own projections (pi agrees to 1e-7): both against each other, in place and not, and
    the dense one against the oracle."""
    from paper_2308_11371_gb300 import binding
    probs = [_problem(kind, n_rhs) for _ in range(copies)]
    f, s = binding.Solver(probs), binding.Solver(probs, precision=binding.FETIDP_MIXED_BF16)
    b = np.random.default_rng(4).standard_normal((f.n_rhs, f.n_P))
    x = f.coarse_solve(_dev(b))
    y = _dev(b)
    f.coarse_solve(y, y)
    assert torch.equal(x, y)
    assert _rel(s.coarse_solve(_dev(b)).cpu(), x.cpu()) < 1e-6
    if copies == 1:
        ref = _oracle(kind)
        for r in range(n_rhs):
            assert _rel(x[r].cpu(), ref.rom.coarse_solve(b[r])) < 1e-9


@pytest.mark.parametrize("cells,elems,clamp,load", [
    ((1, 1), 2, (0, 0), (1, 1)), ((5, 1), 3, (1, 1), (0, 0)), ((3, 7), 7, (0, 1), (0, 0)), ((40, 33), 8, (1, 0), (1, 1)),
    ((1, 1, 1), 2, (0, 0), (0, 1)), ((1, 3, 2), 3, (2, 1), (1, 0)), ((4, 2, 3), 4, (1, 0), (2, 1)),
    ((3, 3, 5), 5, (0, 1), (0, 0)),
])
def test_maps_and_loads_match_oracle(cells, elems, clamp, load):
    """B, B^T, the corner map and the loads are built per node: grids of one cell, several scan blocks
    (2048 nodes), each clamped face, a traction and a body force, alone and as the second lattice of a batch."""
    from oracle.discretization import Lattice
    from paper_2308_11371_gb300 import binding
    d = len(cells)
    make = W.lattice_2d if d == 2 else W.lattice_3d
    loads = [W.Load(W.LOAD_TRACTION, tuple(np.arange(1.0, d + 1)), axis=load[0], side=load[1]),
             W.Load(W.LOAD_BODY, tuple(np.arange(d, 0.0, -1.0)))]
    kw = dict(a=0.3) if d == 2 else dict(map_kind=W.MAP_SHEAR_BEND_3D, map_params=(0.2, 2.0, 0.1, -0.05))
    prob = make(*cells, e=elems, n_rb=1, **kw)
    prob.clamp_axis, prob.clamp_side = clamp
    first = make(*((2, 1) if d == 2 else (1, 2, 1)), e=elems, n_rb=1, **kw)
    first.loads, prob.loads = loads[::-1], loads
    rng = np.random.default_rng(11)
    for probs in ([prob], [first, prob]):
        lats = [Lattice(q) for q in probs]
        Bd = sp.block_diag([q.Bd for q in lats]).tocsr()
        f = np.concatenate([np.stack([q.load(c) for c in range(q.N)], 1) for q in lats], 1)
        s = binding.Solver(probs if len(probs) > 1 else prob)
        assert (s.L, s.n_P) == (Bd.shape[0], sum(q.n_P for q in lats))
        lam = rng.standard_normal((2, s.L))
        xd = s.gather_BT(_dev(lam)).cpu().numpy()
        yd = rng.standard_normal((2, s.N, s.n_d))
        z = s.scatter_B(_dev(yd)).cpu().numpy()
        u = rng.standard_normal(f.shape)
        c = s.compliance(_dev(u))
        for r in range(2):
            assert np.array_equal(xd[r].ravel(), Bd.T @ lam[r])
            assert np.array_equal(z[r], Bd @ yd[r].ravel())
            # sums of at most 2^d loads per node and n_dof N products, in another order
            assert abs(c[r] - (f[r] * u[r]).sum()) < 1e-12 * np.abs(f[r] * u[r]).sum()
        s.close()


@pytest.mark.parametrize("cells", [(1, 3), (2, 2), (13, 3), (40, 2), (3, 2, 2), (9, 2, 1)])
@pytest.mark.parametrize("n_rhs", [1, 3, 9])
def test_fp32_coarse_levels_repeat_and_converge(cells, n_rhs):
    """One to six levels of the cooperative coarse solve, one and two chunks of RHS: its barrier counters are
    cleared by the launch itself, so repeated applications give the same bits, and the solve that uses it
    reaches the monolithic displacement (1e-6 at outer residual 1e-8, as for the other mixed solves)."""
    from oracle import monolithic
    from oracle.discretization import Lattice
    from paper_2308_11371_gb300 import binding
    d = len(cells)
    make = W.lattice_2d if d == 2 else W.lattice_3d
    prob = make(*cells, e=4 if d == 2 else 3, n_rb=1)
    prob.loads = _loads(d, n_rhs)
    s = binding.Solver(prob, precision=binding.FETIDP_MIXED_BF16, tol_outer=1e-8)
    x = _dev(np.random.default_rng(5).standard_normal((n_rhs, s.L)))
    first = s.apply_F(x).clone()
    for _ in range(4):
        assert torch.equal(s.apply_F(x), first)
    u, _, info = s.solve()
    assert info["rel_residual"] <= 1e-8
    lat = Lattice(prob)
    assert _rel(u.cpu().numpy(), monolithic.to_cells(lat, monolithic.solve(lat))) < 1e-6
    s.close()
