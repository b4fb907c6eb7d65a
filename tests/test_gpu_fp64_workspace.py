"""GPU: the workspaces of the FP64 path's residue arithmetic. They only make calls
faster: a limit turns them off or makes the exchange take its moduli in several
passes (bit for bit the one-pass result, since every modulus' residues are the same), they
are given back when a buffer that a call needs does not fit, and what the integers
cannot hold is computed in double arithmetic, mesh point by mesh point."""
import numpy as np
import pytest

from oracle import fedvr_oracle as O
from paper_0911_4348_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-13  # residues against double arithmetic: the bound of the residue parity tests


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import Context
    c = Context()
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _sigma(ctx, V, G):
    S = torch.empty(G.shape, dtype=torch.float64, device="cuda")
    ctx.sigma2(_dev(V), _dev(G), S)
    torch.cuda.synchronize()
    return S.cpu().numpy()


@pytest.mark.parametrize("n,M", [(33, 40), (257, 2)])
def test_exchange_in_several_passes(ctx, n, M):
    rng = W.system_rng(105, n)
    G, V = W.random_symmetric_stack(rng, M, n), W.random_symmetric(rng, n)
    ctx.fp64_workspace(1 << 30)
    one = _sigma(ctx, V, G)
    st = ctx.fp64_workspace()
    assert st["exchange"] == 1 and st["passes"] == 1
    limit, seen = 1 << 30, set()
    while limit > 1 << 16:
        ctx.fp64_workspace(limit)
        got = _sigma(ctx, V, G)
        st = ctx.fp64_workspace()
        if st["exchange"] == 0:
            assert st["passes"] == 0
            assert np.max(np.abs(got - one)) < TOL * np.max(np.abs(one))
            break
        assert st["exchange"] == 1
        assert np.array_equal(got, one), st
        seen.add(st["passes"])
        limit = int(limit / 1.25)
    else:
        pytest.fail("a limit of 64 KB cannot hold the planes of a modulus")
    assert {1, 2, 3} <= seen and max(seen) > 10  # one modulus' planes do not fit below that
    ctx.fp64_workspace(1 << 30)
    assert np.array_equal(_sigma(ctx, V, G), one)


# every remainder of the 64-wide column slices, one and two column tiles, one and two
# buffers of gb, single and partial tile rows; by residues at every size
@pytest.mark.parametrize("n,M", [(12, 40), (16, 40), (17, 33), (33, 9), (48, 5), (63, 4), (64, 4),
                                 (65, 3), (79, 1), (97, 2), (112, 2), (130, 2), (255, 1), (272, 1)])
def test_exchange_at_the_edges_of_its_tiles(ctx, n, M):
    rng = W.system_rng(109, n)
    G, V = W.random_symmetric_stack(rng, M, n), W.random_symmetric(rng, n)
    ctx.fp64_workspace(8 << 30)
    got = _sigma(ctx, V, G)
    assert ctx.fp64_workspace()["exchange"] == 1
    for j in sorted({0, M // 2, M - 1}):
        want = O.sigma2_tau(G[j], G[M - 1 - j], V, 2.0)
        assert np.max(np.abs(got[j] - want)) < TOL * np.max(np.abs(want)), j


@pytest.mark.parametrize("n,u,p,order", [(12, 1, 3, 2), (12, 2, 6, 4), (16, 1, 4, 2), (33, 1, 3, 4),
                                         (63, 1, 2, 2), (65, 1, 2, 2)])
def test_small_convolutions_by_residues(ctx, n, u, p, order):
    M = 2 * u * p + 1
    rng = W.system_rng(110, n)
    A, G, d = rng.uniform(-1, 1, (M, n, n)), rng.uniform(-1, 1, (M, n, n)), rng.uniform(-1, 1, (n, n))
    mesh = O.power_mesh(40.0, u, p)
    want = O.conv1(d, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0),
                   **({"quad": "cubic4"} if order == 4 else {}))
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.fp64_workspace(8 << 30)
    ctx.set_quadrature(order)
    ctx.conv_sigma_g(40.0, u, p, _dev(d), _dev(A), _dev(G), I1)
    assert ctx.fp64_workspace()["conv"] == 1
    assert np.max(np.abs(I1.cpu().numpy() - want)) < TOL * np.max(np.abs(want))


# where the estimates of both sides cross: the call takes the side that measured faster
@pytest.mark.parametrize("n,M,residues", [(10, 4097, 0), (16, 700, 1), (24, 129, 1), (33, 40, 0),
                                          (39, 18, 0), (39, 129, 1), (74, 9, 1)])
def test_exchange_takes_the_faster_side(ctx, n, M, residues):
    G = torch.zeros((M, n, n), dtype=torch.float64, device="cuda")
    G[:] = torch.eye(n, dtype=torch.float64, device="cuda")
    ctx.sigma2(torch.ones((n, n), dtype=torch.float64, device="cuda"), G, torch.empty_like(G))
    assert ctx.fp64_workspace()["exchange"] == residues


def test_double_arithmetic_is_the_allocation_free_call(ctx):
    from paper_0911_4348_gb300 import sigma2_noalloc
    n, M = 74, 9  # by residues without a limit
    rng = W.system_rng(111, n)
    G, V = _dev(W.random_symmetric_stack(rng, M, n)), _dev(W.random_symmetric(rng, n))
    S, T = torch.empty_like(G), torch.empty_like(G)
    ctx.sigma2(V, G, S, 1.5)
    assert ctx.fp64_workspace()["exchange"] == 1
    ctx.fp64_workspace(0)
    ctx.sigma2(V, G, S, 1.5)
    sigma2_noalloc(V, G, T, 1.5)
    torch.cuda.synchronize()
    assert torch.equal(S, T)


def test_no_workspace_in_a_prepared_run(ctx):
    s = W.he_small()
    ctx.build_fedvr(s.n_elem, s.pts_per_elem, s.xmin, s.xmax, s.grid_kind)
    ctx.set_potential(s.Z, s.R, s.soft_en, s.soft_ee, s.n_elec)
    ctx.solve_hf(s.beta, tol=1e-12)
    out = []
    for limit in (-2, 0, -2):
        ctx.fp64_workspace(limit)
        ctx.prepare_2b(s.beta, s.u, s.p)
        r = [ctx.step_2b(0.5) for _ in range(3)]
        assert ctx.fp64_workspace()["conv"] == (0 if limit == 0 else 1)
        out.append(r[-1])
    assert out[0] == out[2]
    assert abs(out[0]["E0"] - out[1]["E0"]) < 1e-12 * abs(out[1]["E0"])
    # taken away under a prepared run: it goes on in double arithmetic
    ctx.prepare_2b(s.beta, s.u, s.p)
    ctx.step_2b(0.5)
    ctx.fp64_workspace(0)
    r = [ctx.step_2b(0.5) for _ in range(2)][-1]
    assert ctx.fp64_workspace()["conv"] == 0
    assert abs(r["E0"] - out[0]["E0"]) < 1e-12 * abs(out[0]["E0"])


def test_given_back_when_a_buffer_does_not_fit(ctx):
    rng = W.system_rng(106, 1)
    n, u, p = 96, 16, 16
    M = 2 * u * p + 1
    V = W.random_symmetric(rng, n)
    G = W.random_symmetric_stack(rng, M, n)
    d = 0.1 * W.random_symmetric(rng, n)
    Vd, Gd, dd = _dev(V), _dev(G), _dev(d)
    S, I1 = torch.empty_like(Gd), torch.empty_like(Gd)
    ctx.conv_sigma_g(40.0, u, p, dd, Gd, Gd, I1)
    ctx.sigma2(Vd, Gd, S)
    assert ctx.fp64_workspace() == dict(conv=1, exchange=1, passes=1)
    # a call whose own buffers (three stacks of 480 MB) fit only without the residues'
    m2 = 4097
    n2 = 120
    small = W.random_symmetric_stack(rng, 1, n2)
    G2 = torch.from_numpy(small).cuda().expand(m2, n2, n2).contiguous()
    V2 = _dev(W.random_symmetric(rng, n2))
    S2 = torch.empty_like(G2)
    torch.cuda.synchronize()
    need = 3 * G2.numel() * 8
    hog = []
    try:
        # leave a third of what the call needs, in pieces that the allocator can have
        while True:
            free = torch.cuda.mem_get_info()[0] - need // 3
            if free < 64 << 20:
                break
            try:
                hog.append(torch.empty(int(min(free, 32 << 30)) // (2 << 20) * (2 << 20),
                                       dtype=torch.uint8, device="cuda"))
            except torch.cuda.OutOfMemoryError:
                break
        ctx.sigma2(V2, G2, S2)
        torch.cuda.synchronize()
        got = S2[[0, m2 // 2, m2 - 1]].cpu().numpy()
    finally:
        hog.clear()
        torch.cuda.empty_cache()
    want = O.sigma2_tau(small[0], small[0], V2.cpu().numpy(), 2.0)
    for x in got:
        assert np.max(np.abs(x - want)) < TOL * np.max(np.abs(want))


def test_cancelling_mesh_points_in_double_arithmetic(ctx):
    # Sigma's column 0 is the negative of column 1 up to 2^-30 and g's rows 0 and 1 agree
    # on all but a few points, so most results cancel 2^-30 below their products
    n, u, p = 24, 2, 8
    M = 2 * u * p + 1
    rng = W.system_rng(107, n)
    A, G = 1e-9 * rng.uniform(-1, 1, (M, n, n)), 1e-9 * rng.uniform(-1, 1, (M, n, n))
    d = np.zeros((n, n))
    A[:, :, 0] = rng.uniform(0.5, 1, (n,))
    A[:, :, 1] = -A[:, :, 0] * (1 + 2.0 ** -30 * rng.uniform(0, 1, (n,)))
    G[:, 0, :] = G[:, 1, :] = rng.uniform(0.5, 1, (n,))
    dev = [_dev(x) for x in (d, A, G)]

    def run(limit):
        I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
        ctx.fp64_workspace(limit)
        ctx.conv_sigma_g(40.0, u, p, *dev, I1)
        return I1.cpu().numpy(), ctx.fp64_workspace()["conv"]

    got, st = run(8 << 30)
    double, st0 = run(0)
    assert st == 2 and st0 == 0
    mesh = O.power_mesh(40.0, u, p)
    want = O.conv1(d, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0))
    terms = O.conv1(np.abs(d), np.abs(A), np.abs(G), mesh, 40.0,
                    dict(O.lag_table(mesh["tau"], 40.0), s=np.ones((M, M))))
    # every point either double arithmetic's sum up to the order of the splits or, where it
    # does not cancel, as near
    assert np.max(np.abs(got - double)) < TOL * np.max(np.abs(terms))
    small = np.max(np.abs(want), axis=(1, 2)) < 2.0 ** -12 * np.max(np.abs(terms), axis=(1, 2))
    assert small.any()


def test_disjoint_blocks_of_the_exchange_in_double_arithmetic(ctx):
    # g and gb live on different halves, so that nothing meets (at j = 0 one entry does)
    n, M = 64, 4
    rng = W.system_rng(108, n)
    V = W.random_symmetric(rng, n)
    h = n // 2
    G = np.zeros((M, n, n))
    for j in range(M):
        a, b = (slice(0, h), slice(h, n)) if j < M // 2 else (slice(h, n), slice(0, h))
        G[j][a, a] = W.random_symmetric(rng, h)
        G[j][b, b] = 0.0
    G[0, 0, h] = G[0, h, 0] = 1e-3  # one entry that lets them meet
    ctx.fp64_workspace(8 << 30)
    got = _sigma(ctx, V, G)
    st = ctx.fp64_workspace()
    assert st["exchange"] == 2
    ctx.fp64_workspace(0)
    double = _sigma(ctx, V, G)
    want = O.sigma2(G, V, 2.0)
    for j in range(M):
        assert np.max(np.abs(got[j] - want[j])) <= TOL * np.max(np.abs(want[j]))
        if not want[j].any():
            assert np.array_equal(got[j], double[j])
