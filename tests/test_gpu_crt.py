"""FP64 contractions by residue arithmetic on the tensor cores against the FP64
oracle, at the edges of their tiles: every remainder of the 64-wide slices (32-
and 16-wide rests), one and two column tiles, full and partial 256-row tiles,
odd and even counts in the last chunk of a rest, the four-row table, and inputs
that the integers cannot hold (which the FP64 kernel computes).

Bounds: the residue path returns the exact sum of operands rounded to 2^-57 of
their largest entry, rounded once; the oracle's own FP64 sums of K = n M terms
carry about sqrt(K) 2^-53 of the largest partial sum. 1e-13 covers both for
K < 1e5 with the cancellation (up to 40) between the anti-periodic branches."""
import numpy as np
import pytest

from oracle import fedvr_oracle as O
from paper_0911_4348_gb300 import workloads as W
from tests._systems import maxrel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL = 1e-13


@pytest.fixture(scope="module")
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import Context
    c = Context()
    yield c
    c.close()


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _conv_case(n, M, seed, scale=1.0):
    rng = W.system_rng(94, seed)
    # a spread of magnitudes over the mesh points: every matrix has its own exponent
    mag = 10.0 ** rng.uniform(-6, 1, size=(M, 1, 1))
    A = scale * mag * rng.uniform(-1, 1, (M, n, n))  # not symmetric: index order matters
    G = rng.uniform(-1, 1, (M, n, n))
    return A, G, 0.1 * scale * rng.uniform(-1, 1, (n, n))


@pytest.mark.parametrize("n,u,p,order", [
    (12, 2, 6, 2), (16, 3, 4, 2), (17, 2, 8, 2), (33, 2, 6, 2), (48, 2, 6, 2), (63, 2, 6, 4),
    (64, 1, 12, 2), (65, 1, 12, 4), (97, 1, 6, 2), (256, 1, 2, 2), (257, 1, 2, 4), (272, 1, 2, 2)])
def test_first_convolution(ctx, n, u, p, order):
    M = 2 * u * p + 1
    A, G, dHF = _conv_case(n, M, n)
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.set_quadrature(order)
    ctx.conv_sigma_g(40.0, u, p, _dev(dHF), _dev(A), _dev(G), I1)
    torch.cuda.synchronize()
    ctx.set_quadrature(2)
    mesh = O.power_mesh(40.0, u, p)
    want = O.conv1(dHF, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0),
                   **({"quad": "cubic4"} if order == 4 else {}))
    assert maxrel(I1.cpu().numpy(), want) < TOL


@pytest.mark.parametrize("scale", [1e-300, 1e250])
def test_first_convolution_far_exponents(ctx, scale):
    n, u, p = 21, 2, 7
    M = 2 * u * p + 1
    A, G, dHF = _conv_case(n, M, 3)
    mesh = O.power_mesh(40.0, u, p)
    G[M // 2] = 0.0  # a zero matrix has no exponent
    want = O.conv1(dHF, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0))
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.conv_sigma_g(40.0, u, p, _dev(scale * dHF), _dev(scale * A), _dev(G), I1)
    torch.cuda.synchronize()
    assert maxrel(I1.cpu().numpy() / scale, want) < TOL


def test_first_convolution_not_finite_and_zero(ctx):
    n, u, p = 21, 2, 7
    M = 2 * u * p + 1
    A, G, dHF = _conv_case(n, M, 4)
    A[3, 2, 1] = np.inf
    I1 = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.conv_sigma_g(40.0, u, p, _dev(dHF), _dev(A), _dev(G), I1)
    torch.cuda.synchronize()
    got = I1.cpu().numpy()
    with np.errstate(invalid="ignore"):
        mesh = O.power_mesh(40.0, u, p)
        want = O.conv1(dHF, A, G, mesh, 40.0, O.lag_table(mesh["tau"], 40.0))
    ok = np.isfinite(want)
    assert ok.any() and not ok.all()
    assert np.array_equal(np.isfinite(got), ok)
    assert np.max(np.abs(got[ok] - want[ok])) < TOL * np.max(np.abs(want[ok]))
    # the next call starts with a clean flag; an all-zero G gives exact zeros
    A[3, 2, 1] = 0.5
    ctx.conv_sigma_g(40.0, u, p, _dev(dHF), _dev(A), _dev(0.0 * G), I1)
    torch.cuda.synchronize()
    assert not I1.cpu().numpy().any()


def _sigma_case(n, M, seed):
    rng = W.system_rng(95, seed)
    mag = 10.0 ** rng.uniform(-4, 1, size=(M, 1, 1))
    G = mag * W.random_symmetric_stack(rng, M, n)
    return G, W.random_symmetric(rng, n)


# n up to 64, 65 .. and above 256 (two column tiles), every remainder of the
# 64-wide slices, one and two buffers of gb, a single tile row and partial tiles
@pytest.mark.parametrize("n,M", [(16, 700), (17, 500), (33, 40), (39, 20), (48, 9), (63, 4), (64, 4),
                                 (65, 3), (97, 2), (130, 3), (199, 2), (240, 2), (255, 2), (256, 2),
                                 (257, 2), (299, 2)])
def test_second_born(ctx, n, M):
    G, V = _sigma_case(n, M, n)
    S = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.sigma2(_dev(V), _dev(G), S, 1.5)
    torch.cuda.synchronize()
    got = S.cpu().numpy()
    js = range(M) if n < 100 and M < 50 else [0, M // 2, M - 1]
    for j in js:  # against each mesh point's own largest entry
        want = O.sigma2_tau(G[j], G[M - 1 - j], V, 1.5)
        assert np.max(np.abs(got[j] - want)) < TOL * np.max(np.abs(want)), j
    assert np.array_equal(got, got.transpose(0, 2, 1))


def test_second_born_not_finite(ctx):
    n, M = 65, 3
    G, V = _sigma_case(n, M, 1)
    G[1, 2, 3] = G[1, 3, 2] = np.nan
    S = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx.sigma2(_dev(V), _dev(G), S)
    torch.cuda.synchronize()
    got = S.cpu().numpy()
    assert np.isnan(got[1]).all()  # every sum of that mesh point meets the entry
    for j in (0, 2):
        want = O.sigma2_tau(G[j], G[M - 1 - j], V, 2.0)
        assert np.max(np.abs(got[j] - want)) < TOL * np.max(np.abs(want))


def test_ladder_from_an_unsymmetric_start(ctx):
    # the ladder's convolution as a residue product of n^2 x n^2 matrices (n = 7,
    # M = 65), from a random t without the pair symmetries: rows, columns and the
    # transposed storage have to match the oracle's
    from paper_0911_4348_gb300 import FedvrError
    rng = W.system_rng(93, 7)
    n, u, p, beta = 7, 4, 8, 12.0
    h = W.random_symmetric(rng, n)
    V = 0.2 * np.abs(W.random_symmetric(rng, n))
    e, C = np.linalg.eigh(h)
    mesh = O.power_mesh(beta, u, p)
    G = O.g0_mesh(e, C, 0.5 * (e[2] + e[3]), mesh["tau"], beta)
    M = G.shape[0]
    t0 = 0.01 * rng.uniform(-1, 1, (M, n, n, n, n))  # t0[j][a][k][b][l]
    want = O.sigma_tmatrix(G, V, 2.0, mesh, O.bose_lag_table(mesh["tau"], beta), t0=t0, tol=1e-4)
    t = _dev(t0.transpose(0, 3, 4, 1, 2))
    S = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    it = ctx.sigma_tmatrix(beta, u, p, _dev(V), _dev(G), S, t=t, t_valid=True, t_tol=1e-4)
    torch.cuda.synchronize()
    assert it == want["iters"]
    assert maxrel(S.cpu().numpy(), want["Sigma"]) < TOL
    assert maxrel(t.cpu().numpy().transpose(0, 3, 4, 1, 2), want["t"]) < TOL
    G[3, 1, 1] = np.nan
    with pytest.raises(FedvrError) as err:
        ctx.sigma_tmatrix(beta, u, p, _dev(V), _dev(G), S)
    assert err.value.code == -6
