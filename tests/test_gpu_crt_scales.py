"""FP64 contractions by residue arithmetic: inputs whose entries differ in size
inside one matrix. Rows of the source, columns of g, single mesh points and the
contracted index are scaled by powers of two down to 2^-60 (10^-18); the result has
to be as accurate row by row and column by column as without the scales, which
power-of-two factors do not change in double arithmetic. The exchange is also held
entry by entry, on uncoupled blocks and on a Green's function that decays over 8 to 11
orders of magnitude.

Bounds. Relative to the products of its row's and column's scales an operand
entry is rounded to 2^-57 (convolution) or 2^-58 (exchange); K products add up to
sqrt(K) of such errors and K is below 1e5: 1e-13 as in the parity tests of the same
kernels. Against the sum of the magnitudes of an entry's own terms, the exchange of a
decaying g is held to 1e-13 too: the rounding of 2^-58 per factor leaves 2^10 for the
distance between the largest term of an entry and its row's and column's scales."""
import numpy as np
import pytest

from oracle import fedvr_oracle as O
from paper_0911_4348_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import Context
    c = Context()
    c.fp64_workspace(8 << 30)  # a limit of its own: residues at every size here
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _two(rng, n, span=60):
    e = rng.integers(-span, 1, n)
    e[rng.integers(n)] = 0
    return np.ldexp(1.0, e)


# (rows of the source, contracted index, columns of g) scaled or not
@pytest.mark.parametrize("which", ["row", "column", "inner", "all"])
@pytest.mark.parametrize("n,u,p,order", [(17, 2, 8, 2), (40, 2, 6, 2), (65, 1, 12, 4), (130, 1, 6, 2)])
def test_convolution_of_scaled_rows_and_columns(ctx, n, u, p, order, which):
    rng = W.system_rng(101, n)
    M = 2 * u * p + 1
    one = np.ones(n)
    r = _two(rng, n) if which in ("row", "all") else one
    t = _two(rng, n) if which in ("inner", "all") else one
    s = _two(rng, n) if which in ("column", "all") else one
    mag = 10.0 ** rng.uniform(-6, 1, size=(M, 1, 1))
    A, G = mag * rng.uniform(-1, 1, (M, n, n)), rng.uniform(-1, 1, (M, n, n))
    dHF = 0.1 * rng.uniform(-1, 1, (n, n))
    left, right = r[:, None] / t[None, :], t[:, None] * s[None, :]
    mesh = O.power_mesh(40.0, u, p)
    want = O.conv1(dHF, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0),
                   **({"quad": "cubic4"} if order == 4 else {}))
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.set_quadrature(order)
    ctx.conv_sigma_g(40.0, u, p, _dev(dHF * left), _dev(A * left), _dev(G * right), I1)
    torch.cuda.synchronize()
    ctx.set_quadrature(2)
    assert ctx.fp64_workspace()["conv"] in (1, 2)
    got = I1.cpu().numpy() / r[:, None] / s[None, :]
    assert np.max(np.abs(got - want)) < TOL * np.max(np.abs(want))
    # every row and every column by itself, relative to the stack's largest entry of it
    for ax in ((0, 2), (0, 1)):
        assert np.all(np.max(np.abs(got - want), axis=ax) < 10 * TOL * np.max(np.abs(want), axis=ax))


def test_convolution_of_empty_rows_and_columns(ctx):
    n, u, p = 40, 2, 6
    M = 2 * u * p + 1
    rng = W.system_rng(102, n)
    A, G, d = rng.uniform(-1, 1, (M, n, n)), rng.uniform(-1, 1, (M, n, n)), rng.uniform(-1, 1, (n, n))
    for x in (A, d):
        x[..., 3, :] = 0.0  # a row of the source
        x[..., :, 5] = 0.0  # a contracted column of the source
    G[:, 7, :] = 0.0        # a contracted row of g
    G[:, :, 9] = 0.0        # a column of g
    G[:, 5, :] *= 1e200     # meets the source's empty column only
    mesh = O.power_mesh(40.0, u, p)
    want = O.conv1(d, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0))
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.conv_sigma_g(40.0, u, p, _dev(d), _dev(A), _dev(G), I1)
    torch.cuda.synchronize()
    got = I1.cpu().numpy()
    assert np.max(np.abs(got - want)) < TOL * np.max(np.abs(want))
    assert not got[:, 3, :].any() and not got[:, :, 9].any()


def _exchange(ctx, V, G):
    S = torch.empty(G.shape, dtype=torch.float64, device="cuda")
    ctx.sigma2(_dev(V), _dev(G), S, 0.0)  # spin 0: the exchange alone
    torch.cuda.synchronize()
    assert ctx.fp64_workspace()["exchange"] in (1, 2)
    return S.cpu().numpy()


@pytest.mark.parametrize("n,M", [(33, 40), (65, 4), (130, 3), (257, 2)])
def test_exchange_of_scaled_matrices(ctx, n, M):
    # g_j -> D_j g_j D_j and V -> U V U: every mesh point with scales of its own
    rng = W.system_rng(103, n)
    G, V = W.random_symmetric_stack(rng, M, n), W.random_symmetric(rng, n)
    u = np.ldexp(1.0, rng.integers(-15, 1, n))
    D = np.stack([np.ldexp(1.0, rng.integers(-30, 1, n)) for _ in range(M)])
    # the pair (j, M - 1 - j) shares k and l: opposite scales there, none left over
    got = _exchange(ctx, V * u[:, None] * u[None, :],
                    G * D[:, :, None] * D[:, None, :])
    for j in sorted({0, M // 2, M - 1}):
        g, gb = G[j] * D[j][:, None] * D[j][None, :], None
        b = M - 1 - j
        gb = G[b] * D[b][:, None] * D[b][None, :]
        v = V * u[:, None] * u[None, :]
        want = O.sigma2_tau(g, gb, v, 0.0)
        f = u * D[j]
        w, x = want / f[:, None] / f[None, :], got[j] / f[:, None] / f[None, :]
        assert np.max(np.abs(x - w)) < TOL * np.max(np.abs(w)), j


@pytest.mark.parametrize("scale", [1e-9, 1e-18])
def test_exchange_of_uncoupled_blocks(ctx, scale):
    n, M = 48, 9
    rng = W.system_rng(104, n)
    V = W.random_symmetric(rng, n)
    G = np.zeros((M, n, n))
    h = n // 2
    G[:, :h, :h] = W.random_symmetric_stack(rng, M, h)
    G[:, h:, h:] = scale * W.random_symmetric_stack(rng, M, n - h)
    got = _exchange(ctx, V, G)
    for j in range(M):
        want = O.sigma2_tau(G[j], G[M - 1 - j], V, 0.0)
        for s in (slice(0, h), slice(h, n)):
            assert np.max(np.abs(got[j][s, s] - want[s, s])) < TOL * np.max(np.abs(want[s, s])), j


@pytest.mark.parametrize("n_elem,order,half", [(10, 4, 10.0), (13, 5, 12.0)])
def test_exchange_of_a_decaying_function_entry_by_entry(ctx, n_elem, order, half):
    b = O.fedvr_basis(n_elem, order, -half, half, 0)
    h = O.kinetic(b) + np.diag(O.potential(b["nodes"], [2.0], [0.0], 1.0))
    V = O.interaction(b["nodes"], 1.0)
    hf = O.hf_scf(h, V, 2.0, 1, 100.0, tol=1e-11)
    mesh = O.power_mesh(100.0, 3, 8)
    G = O.g0_mesh(hf["eps"], hf["C"], hf["mu"], mesh["tau"], 100.0)
    G = 0.5 * (G + G.transpose(0, 2, 1))
    M = G.shape[0]
    assert np.min(np.abs(G[-1])) < 1e-8 * np.max(np.abs(G[-1]))
    got = _exchange(ctx, V, G)
    for j in range(M):
        want = O.sigma2_tau(G[j], G[M - 1 - j], V, 0.0)
        terms = -O.sigma2_tau(np.abs(G[j]), np.abs(G[M - 1 - j]), np.abs(V), 0.0)
        assert np.all(np.abs(got[j] - want) <= TOL * np.abs(terms)), j


# Sparse and badly scaled in every index at once: no scales fit all products, so what the
# integers cannot hold has to be left to double arithmetic. Mesh points may lie 2^10
# below their largest products before that: 2^-47 sqrt(K) with K < 1e4 products, 1e-12.
@pytest.mark.parametrize("seed", range(12))
def test_sparse_and_badly_scaled_convolutions(ctx, seed):
    rng = W.system_rng(112, seed)
    n, u, p = int(rng.integers(12, 90)), int(rng.integers(1, 4)), int(rng.integers(2, 6))
    order, M = int(rng.choice([2, 4])), 2 * u * p + 1
    r, t, s = (np.ldexp(1.0, rng.integers(-200, 201, n)) for _ in range(3))
    mesh = lambda: np.ldexp(1.0, rng.integers(-30, 31, M))[:, None, None]
    A, G = rng.uniform(-1, 1, (M, n, n)) * mesh(), rng.uniform(-1, 1, (M, n, n)) * mesh()
    A *= rng.random(A.shape) < 0.1
    if seed % 2:
        G *= rng.random(G.shape) < 0.1
    A[rng.integers(M)] = 0.0
    d = rng.uniform(-1, 1, (n, n))
    left, right = r[:, None] / t[None, :], t[:, None] * s[None, :]
    dev = [_dev(x) for x in (d * left, A * left, G * right)]
    out, state = [], []
    ctx.set_quadrature(order)
    for limit in (0, 8 << 30):
        ctx.fp64_workspace(limit)
        I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
        ctx.conv_sigma_g(40.0, u, p, *dev, I1)
        out.append(I1.cpu().numpy())
        state.append(ctx.fp64_workspace()["conv"])
    ctx.set_quadrature(2)
    assert state[0] == 0 and state[1] in (1, 2)
    for i in range(M):
        assert np.max(np.abs(out[1][i] - out[0][i])) <= 1e-12 * np.max(np.abs(out[0][i])), i


@pytest.mark.parametrize("seed", range(12))
def test_sparse_and_badly_scaled_exchange(ctx, seed):
    rng = W.system_rng(113, seed)
    n, M = int(rng.integers(12, 120)), int(rng.integers(1, 7))
    G = W.random_symmetric_stack(rng, M, n)
    keep = rng.random((n, n)) < 0.1
    G = G * (keep | keep.T)
    D = np.ldexp(1.0, rng.integers(-60, 61, (M, n)))
    w = np.ldexp(1.0, rng.integers(-20, 21, n))
    G = G * D[:, :, None] * D[:, None, :]
    V = W.random_symmetric(rng, n) * w[:, None] * w[None, :]
    ctx.fp64_workspace(0)
    S = torch.empty(G.shape, dtype=torch.float64, device="cuda")
    ctx.sigma2(_dev(V), _dev(G), S, 0.0)
    want = S.cpu().numpy()
    ctx.fp64_workspace(8 << 30)
    got = _exchange(ctx, V, G)
    for j in range(M):
        assert np.max(np.abs(got[j] - want[j])) <= 1e-12 * np.max(np.abs(want[j])), j


def test_convolution_of_a_decaying_function(ctx):
    # what is kept of an entry is relative to the largest products of its row and column
    # over the mesh points, whatever the entry itself is: K = 2 M n roundings of 2^-57 each,
    # a factor of 16 for the rounding of the scales to powers of two
    b = O.fedvr_basis(13, 3, -25.0, 25.0, 0)
    h = O.kinetic(b) + np.diag(O.potential(b["nodes"], [2.0], [0.0], 1.0))
    V = O.interaction(b["nodes"], 1.0)
    beta, u, p = 60.0, 3, 8
    hf = O.hf_scf(h, V, 2.0, 1, beta, tol=1e-11)
    mesh = O.power_mesh(beta, u, p)
    lag = O.lag_table(mesh["tau"], beta)
    G = O.g0_mesh(hf["eps"], hf["C"], hf["mu"], mesh["tau"], beta)
    A = O.sigma2(G, V, 2.0)
    M, n, _ = G.shape
    d = 1e-3 * V * G[-1]
    want = O.conv1(d, A, G, mesh, beta, lag)
    assert np.min(np.abs(want[0])) < 1e-14 * np.max(np.abs(want[0]))
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.conv_sigma_g(beta, u, p, _dev(d), _dev(A), _dev(G), I1)
    assert ctx.fp64_workspace()["conv"] == 1
    got = I1.cpu().numpy()
    top = lambda X: np.max(np.abs(X), axis=(1, 2))
    diag = (mesh["wm"] + mesh["wp"])[:, None, None] * np.maximum(np.abs(A[0]), np.abs(A[-1])) + np.abs(d)
    src = np.concatenate([A, diag])
    R = np.max(np.max(np.abs(src), axis=2) / top(src)[:, None], axis=0)
    S = np.max(np.max(np.abs(G), axis=1) / top(G)[:, None], axis=0)
    for i in range(M):
        k = lag["k"][i]
        E = np.max(mesh["w"] * np.maximum(top(A)[k], top(A)[np.minimum(k + 1, M - 1)]) * top(G))
        E = max(E, top(src)[M + i] * top(G)[i])
        bound = 16 * 2.0 ** -57 * np.sqrt(2.0 * M * n) * E * R[:, None] * S[None, :]
        own = 1e-14 * np.abs(want[i])  # the double sums' own error
        assert np.all(np.abs(got[i] - want[i]) <= bound + own), i
        assert np.max(np.abs(got[i] - want[i])) < TOL * np.max(np.abs(want[i]))
