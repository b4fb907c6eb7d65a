"""The measured cases: the calls that programs built on this library make, over the range of
sizes that its workloads, tests and benchmark cover.

Every case is a plain dict. Common keys: ``kind`` (which call), ``n_elem`` and ``order`` (FE-DVR
grid, n_b = n_elem * order - 1), ``half`` (the box is [-half, half]), ``u`` and ``p`` (power mesh,
M = 2 u p + 1 points), ``beta`` and ``precision`` ("f64", "tf32" or "f16"). The seed draws the
physical system (nuclear charge of He, or the bond length of linear H3+), so another seed is
another molecule on the same grid.

Kinds:
  step       one iteration of the self-consistency on a given iterate (``step_2b`` with ``G_in``),
             then the new iterate and its self-energy read back on the device;
  sigma2     the second-Born self-energy of a whole tau-stack (``sigma2``);
  conv       the first Dyson convolution (``conv_sigma_g``);
  batch      a whole self-consistent solve of several uneven systems (``solve_2b_batched``);
  hf         a Hartree-Fock solve (``solve_hf``, ``get_hf``);
  kbe        a real-time Kadanoff-Baym propagation (``kbe_propagate``);
  gw         the GW self-energy (``sigma_gw``);
  tmatrix    the T-matrix self-energy (``sigma_tmatrix``);
  mlp        loss and gradient of the warm-start network on one mini-batch (``loss_grad``).

``exact`` is an independent plain numpy/torch float64 evaluation of the same formulas.
"""

from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_0911_4348_gb300 import Context, WarmStartNet, solve_2b_batched

PRECISION = {"f64": 0, "tf32": 1, "f16": 3}
SPIN = 2.0
MIXING = 0.5


# --------------------------------------------------------------------------------------------
# The cases
# --------------------------------------------------------------------------------------------
def listed():
    return [
        # The smallest iteration: the small He model (n_b = 15, M = 129) in the default
        # precision, where launches and latency count.
        dict(name="step f64 n15 M129", kind="step", species="he", n_elem=4, order=4, half=10.0,
             u=4, p=16, beta=100.0, precision="f64"),
        # An iteration of the plain (default-precision) solver on the 20 x 6 family (n_b = 119,
        # M = 257): both contractions of the method at an ordinary size.
        dict(name="step f64 n119 M257", kind="step", species="he", n_elem=20, order=6, half=50.0,
             u=8, p=16, beta=100.0, precision="f64"),
        # The benchmark's step: He, n_b = 199, M = 513, split FP16.
        dict(name="step f16 n199 M513", kind="step", species="he", n_elem=25, order=8, half=50.0,
             u=16, p=16, beta=100.0, precision="f16"),
        # The largest self-energy build: linear H3+, n_b = 299 (two column tiles), M = 1025.
        dict(name="sigma2 f16 n299 M1025", kind="sigma2", species="h3p", n_elem=30, order=10,
             half=60.0, u=32, p=16, beta=100.0, precision="f16"),
        # The first convolution on the binding-curve grid (n_b = 142, M = 1025).
        dict(name="conv f16 n142 M1025", kind="conv", species="h3p", n_elem=13, order=11,
             half=25.0, u=32, p=16, beta=100.0, precision="f16"),
        # A whole batched solve of four uneven systems in the call's default precision.
        dict(name="batch tf32 4 systems", kind="batch", systems=4, grids=3, u=8, p=16, beta=100.0,
             precision="tf32"),
        # The Hartree-Fock start of the benchmark's system.
        dict(name="hf n199", kind="hf", species="he", n_elem=25, order=8, half=50.0, beta=100.0),
        # Real-time propagation of driven He (n_b = 39), tensor-core and default precision.
        dict(name="kbe tf32 n39 T81", kind="kbe", species="he", n_elem=10, order=4, half=15.0,
             beta=100.0, steps=80, dt=0.04, precision="tf32"),
        dict(name="kbe f64 n39 T25", kind="kbe", species="he", n_elem=10, order=4, half=15.0,
             beta=100.0, steps=24, dt=0.04, precision="f64"),
        # The two self-energies beyond second Born (default precision is their only one).
        dict(name="gw f64 n39 M129", kind="gw", species="he", n_elem=10, order=4, half=15.0, u=4,
             p=16, beta=100.0),
        dict(name="tmatrix f64 n11 M65", kind="tmatrix", species="he", n_elem=4, order=3,
             half=8.0, u=4, p=8, beta=20.0),
        # One training mini-batch of the warm-start network (M = 257, two layers of 512).
        dict(name="mlp rows4096 M257", kind="mlp", rows=4096, M=257, hidden=512),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _grid(rng, lo, hi, order_lo=3, order_hi=10):
    order = rng.randint(order_lo, order_hi)
    n_elem = max(2, round((_log(rng, lo, hi) + 1) / order))
    while n_elem * order - 1 > hi:
        n_elem -= 1
    return dict(n_elem=n_elem, order=order)


def draw(rng):
    kind = rng.choice(["step", "step", "step", "sigma2", "conv", "batch", "hf", "kbe", "kbe",
                       "gw", "tmatrix", "mlp"])
    species = rng.choice(["he", "h3p"])
    half = round(rng.uniform(10.0, 60.0), 1)
    beta = round(rng.uniform(40.0, 100.0), 1)
    if kind in ("step", "sigma2", "conv"):
        precision = rng.choice(["f64", "f64", "tf32", "f16"])
        c = dict(kind=kind, species=species, half=half, beta=beta, precision=precision, p=16)
        top = 142 if precision == "f64" else 299 if kind != "step" else 203
        c.update(_grid(rng, 15, top))
        n = c["n_elem"] * c["order"] - 1
        u = int(round(_log(rng, 2, 32 if precision != "f64" else 12)))
        # no more work than the largest listed case of the precision
        most = 2.4e11 if precision == "f64" else 4.2e12 if kind == "step" else 6e12

        def work_at(u):
            m = 2 * u * 16 + 1
            return ((2.0 * m * m * n ** 3 if kind != "sigma2" else 0.0)
                    + (m * float(n) ** 4 if kind != "conv" else 0.0))

        while u > 2 and work_at(u) > most:
            u -= 1
        return dict(c, u=u)
    if kind == "batch":
        return dict(kind=kind, systems=rng.randint(2, 4), grids=rng.randint(4, 1 << 20), u=8, p=16,
                    beta=100.0, precision=rng.choice(["tf32", "f16"]))
    if kind == "hf":
        return dict(kind=kind, species=species, half=half, beta=beta, **_grid(rng, 15, 199, 3, 10))
    if kind == "kbe":
        precision = rng.choice(["f64", "tf32"])
        steps = rng.randint(8, 24) if precision == "f64" else rng.randint(16, 80)
        return dict(kind=kind, species=species, half=15.0, beta=beta, steps=steps, dt=0.03,
                    precision=precision, **_grid(rng, 11, 39, 3, 4))
    if kind == "gw":
        return dict(kind=kind, species="he", half=round(rng.uniform(10.0, 20.0), 1), u=rng.randint(3, 5),
                    p=16, beta=100.0, **_grid(rng, 14, 44, 3, 5))
    if kind == "tmatrix":
        return dict(kind=kind, species="he", half=round(rng.uniform(6.0, 9.0), 1),
                    u=rng.randint(2, 4), p=8, beta=20.0, **_grid(rng, 5, 11, 2, 4))
    return dict(kind=kind, rows=int(_log(rng, 500, 4096)), M=2 * 16 * rng.randint(4, 8) + 1,
                hidden=rng.choice([256, 512]))


# --------------------------------------------------------------------------------------------
# The method in plain numpy/torch (inputs, and the values of exact())
# --------------------------------------------------------------------------------------------
@functools.lru_cache(maxsize=None)
def _basis(n_elem, order, half):
    """Nodes, kinetic matrix and interaction of the uniform FE-DVR grid."""
    N = order
    c = np.zeros(N + 1)
    c[N] = 1.0
    xi = np.concatenate([[-1.0], np.sort(np.polynomial.legendre.legroots(
        np.polynomial.legendre.legder(c)).real), [1.0]])
    for _ in range(3):  # polish the inner roots of P'_N by Newton steps
        d1, d2 = np.polynomial.legendre.legder(c), np.polynomial.legendre.legder(c, 2)
        xi[1:-1] -= (np.polynomial.legendre.legval(xi[1:-1], d1)
                     / np.polynomial.legendre.legval(xi[1:-1], d2))
    om = 2.0 / (N * (N + 1) * np.polynomial.legendre.legval(xi, c) ** 2)
    D = np.zeros((N + 1, N + 1))  # D[m, k] = f'_m(xi_k)
    for m in range(N + 1):
        for k in range(N + 1):
            if k == m:
                D[m, k] = sum(1.0 / (xi[m] - xi[q]) for q in range(N + 1) if q != m)
            else:
                v = 1.0 / (xi[m] - xi[k])
                for q in range(N + 1):
                    if q != m and q != k:
                        v *= (xi[k] - xi[q]) / (xi[m] - xi[q])
                D[m, k] = v
    h = 2.0 * half / n_elem
    t = (2.0 / h) ** 2 * (D * (0.5 * h * om)) @ D.T
    total = n_elem * N + 1
    x, W, T = np.zeros(total), np.zeros(total), np.zeros((total, total))
    for i in range(n_elem):
        s = slice(i * N, i * N + N + 1)
        x[s] = -half + i * h + 0.5 * (xi + 1.0) * h
        W[s] += 0.5 * h * om
        T[s, s] += t
    x, W, T = x[1:-1], W[1:-1], T[1:-1, 1:-1]
    T = 0.5 * T / np.sqrt(np.outer(W, W))
    V = 1.0 / np.sqrt((x[:, None] - x[None, :]) ** 2 + 1.0)
    return x, T, V


def _nuclei(species, seed):
    r = np.random.Generator(np.random.PCG64([int(seed), 9114348]))
    if species == "he":
        return [float(r.uniform(1.6, 2.4))], [0.0]
    R = float(r.uniform(1.6, 2.4))
    return [1.0, 1.0, 1.0], [-R, float(r.uniform(-0.05, 0.05)), R]


def _hf_sigma(rho, V):
    return SPIN * np.diag(V @ np.diag(rho)) - V * rho


def _mu(eps, beta):
    """Holes below = particles above for one doubly occupied level (log-sum-exp form)."""
    lo, hi = eps[0], eps[1]

    def soft(z):
        return max(z, 0.0) + math.log1p(math.exp(-abs(z)))

    for _ in range(200):
        mu = 0.5 * (lo + hi)
        holes = -soft(beta * (mu - eps[0]))
        part = -np.array([soft(beta * (e - mu)) for e in eps[1:]])
        m = part.max()
        if m + math.log(np.exp(part - m).sum()) < holes:
            lo = mu
        else:
            hi = mu
    return 0.5 * (lo + hi)


def _hf(species, n_elem, order, half, beta, seed, iterations=400, tol=1e-13):
    x, T, V = _basis(n_elem, order, half)
    Z, R = _nuclei(species, seed)
    h = T + np.diag(-sum(z / np.sqrt((x - r) ** 2 + 1.0) for z, r in zip(Z, R)))
    _, C = np.linalg.eigh(h)
    rho = np.outer(C[:, 0], C[:, 0])
    for _ in range(iterations):
        S0 = _hf_sigma(rho, V)
        eps, C = np.linalg.eigh(h + S0)
        mu = _mu(eps, beta)
        f = 1.0 / (1.0 + np.exp(np.clip(beta * (eps - mu), -700.0, 700.0)))
        new = (C * f) @ C.T
        if np.abs(new - rho).max() < tol:
            break
        rho = 0.5 * (rho + new)
    E = SPIN * np.sum(h * new) + 0.5 * SPIN * np.sum(_hf_sigma(new, V) * new)
    return dict(x=x, h=h, V=V, eps=eps, C=C, mu=mu, rho=new, Sigma0=S0, E=E)


def _mesh(beta, u, p):
    B = [0.0] + [0.5 * beta * 0.5 ** (p - k) for k in range(1, p + 1)]
    s = [0.0]
    for k in range(1, p + 1):
        width = B[1] if k == 1 else B[k - 1]
        s += [B[k - 1] + width * r / u for r in range(1, u + 1)]
    s = np.array(s)
    tau = np.concatenate([-beta + s[:-1], -s[::-1]])
    d = 0.5 * np.diff(tau)
    wm, wp = np.concatenate([[0.0], d]), np.concatenate([d, [0.0]])
    return tau, wm + wp, wm, wp


def _phi(tau, eps, mu, beta):
    """g^0 of the levels at each tau in [-beta, 0]: [len(tau)][n]."""
    y, t = (eps - mu)[None, :], tau[:, None]
    up = np.exp(-(beta + t) * np.maximum(y, 0.0)) / (1.0 + np.exp(-beta * np.maximum(y, 0.0)))
    dn = np.exp(-t * np.minimum(y, 0.0)) / (1.0 + np.exp(beta * np.minimum(y, 0.0)))
    return np.where(y >= 0.0, up, dn)


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _g0(hf, tau, beta):
    C = _dev(hf["C"])
    return (C[None] * _dev(_phi(tau, hf["eps"], hf["mu"], beta))[:, None, :]) @ C.T


def _direct(G, V):
    return SPIN * G * (V @ (G * G.flip(0)) @ V)


def _sigma2_exact(G, V):
    S = _direct(G, V)
    Gb = G.flip(0)
    n = V.shape[0]
    step = max(1, int(2e8 // (G.shape[0] * n * n)))
    for b0 in range(0, n, step):  # P^(b) = g diag(V_b) gb; X_ab = sum_k V_ak g_kb P^(b)_ak
        b = slice(b0, min(n, b0 + step))
        P = (G[None] * V[b, None, None, :]) @ Gb[None]           # [b][j][a][k]
        gb = G[:, :, b].permute(2, 0, 1)                          # [b][j][k]
        S[:, :, b] -= torch.einsum("ak,bjk,bjak->jab", V, gb, P)
    return S


def _lags(tau, beta, bose=False):
    """Bracket, weight and sign of tau_i - tau_j mapped into [-beta, 0]."""
    x = tau[:, None] - tau[None, :]
    i, j = np.indices(x.shape)
    keep = j >= i if bose else j > i
    y = np.where(keep, x, x - beta)
    k = np.clip(np.searchsorted(tau, y, side="right") - 1, 0, len(tau) - 2)
    t = (y - tau[k]) / (tau[k + 1] - tau[k])
    return k, t, np.where(keep | bose, 1.0, -1.0)


def _conv1_exact(dHF, S, G, beta, u, p):
    tau, w, wm, wp = _mesh(beta, u, p)
    M, n = len(tau), G.shape[1]
    k, t, sg = _lags(tau, beta)
    out = torch.empty_like(G)
    flat = G.reshape(M * n, n)
    for i in range(M):
        c1, c2 = sg[i] * w * (1.0 - t[i]), sg[i] * w * t[i]
        kk = torch.from_numpy(k[i]).cuda()
        B = _dev(c1)[:, None, None] * S[kk] + _dev(c2)[:, None, None] * S[kk + 1]
        B[i] = dHF - wm[i] * S[0] + wp[i] * S[M - 1]
        out[i] = B.permute(1, 0, 2).reshape(n, M * n) @ flat
    return out


def _conv2_exact(I1, hf, beta, u, p):
    tau, w, wm, wp = _mesh(beta, u, p)
    M = len(tau)
    C = _dev(hf["C"])
    X = C.T @ I1
    out = torch.empty_like(I1)
    ends = _phi(np.array([-beta, 0.0]), hf["eps"], hf["mu"], beta)
    lag = tau[:, None] - tau[None, :]
    i, j = np.indices(lag.shape)
    sign = np.where(j > i, 1.0, -1.0)
    lag = np.where(j > i, lag, lag - beta)
    lag[np.arange(M), np.arange(M)] = 0.0
    for a in range(len(hf["eps"])):
        K = sign * w[None, :] * _phi(lag.reshape(-1), hf["eps"][a:a + 1], hf["mu"], beta).reshape(M, M)
        K[np.arange(M), np.arange(M)] = -wm * ends[0, a] + wp * ends[1, a]
        out[:, a] = _dev(K) @ X[:, a]
    return C @ out


def _bose_conv(Q, W, tau, w, lags):
    k, t, _ = lags
    M, n = len(tau), Q.shape[1]
    out = torch.empty_like(W)
    flat = W.reshape(M * n, n)
    for i in range(M):
        kk = torch.from_numpy(k[i]).cuda()
        A = _dev(w * (1.0 - t[i]))[:, None, None] * Q[kk] + _dev(w * t[i])[:, None, None] * Q[kk + 1]
        out[i] = A.permute(1, 0, 2).reshape(n, M * n) @ flat
    return out


def _gw_exact(G, V, beta, u, p):
    tau, w, _, _ = _mesh(beta, u, p)
    lags = _lags(tau, beta, bose=True)
    Q = G * G.flip(0)
    src = V @ Q @ V
    W = src.clone()
    for _ in range(500):
        new = src - SPIN * (V @ _bose_conv(Q, W, tau, w, lags))
        r = float((new - W).abs().max())
        W = 0.7 * W + 0.3 * new
        if r < 1e-12:
            break
    return SPIN * G * W


def _tmatrix_exact(G, V, beta, u, p):
    tau, w, _, _ = _mesh(beta, u, p)
    k, t, _ = _lags(tau, beta, bose=True)
    M, n = len(tau), G.shape[1]
    # t[j][b][l][a][k] = t_j(ak; bl)
    src = torch.einsum("ak,jab,jkl,bl->jblak", V, G, G, V)
    T = src.clone()
    GT = G.transpose(1, 2)
    for _ in range(500):
        Y = torch.empty_like(T)
        for i in range(M):
            # sum of c X_j over the j of each mesh point r, then g_r (sum) g_r^T
            c = np.zeros((M, M))
            np.add.at(c, (k[i], np.arange(M)), w * (1.0 - t[i]))
            np.add.at(c, (k[i] + 1, np.arange(M)), w * t[i])
            r = np.nonzero(np.abs(c).sum(1))[0]
            X = (_dev(c[r]) @ T.reshape(M, -1)).reshape(len(r), n * n, n, n)
            rr = torch.from_numpy(r).cuda()
            Y[i] = (G[rr][:, None] @ X @ GT[rr][:, None]).sum(0).reshape(n, n, n, n)
        new = src - V[None, None, None] * Y
        res = float((new - T).abs().max())
        T = 0.7 * T + 0.3 * new
        if res < 1e-12:
            break
    Gb = G.flip(0)
    return (SPIN * torch.einsum("jblak,jlk->jab", T, Gb) - torch.einsum("jlbak,jlk->jab", T, Gb))


def _kbe_exact(hf, dt, steps, dv):
    n, Tn = len(hf["eps"]), steps + 1
    z = torch.complex128
    h, V = _dev(hf["h"]).to(z), _dev(hf["V"]).to(z)
    L = torch.zeros((Tn, Tn, n, n), dtype=z, device="cuda")
    Gt = torch.zeros_like(L)
    eye = torch.eye(n, dtype=z, device="cuda")
    L[0, 0] = _dev(hf["rho"]).to(z)
    Gt[0, 0] = L[0, 0] - eye
    S = torch.zeros((2, Tn, n, n), dtype=z, device="cuda")
    rho, E, N = [], [], []

    def hhf(i):
        r = L[i, i]
        s = SPIN * torch.diag(V @ torch.diagonal(r)) - V * r
        return h + torch.diag(_dev(dv[i]).to(z)) + s, s

    def weights(m):
        w = np.full(m + 1, dt)
        w[0] *= 0.5
        w[-1] *= 0.5
        return _dev(w if m else np.zeros(1)).to(z)

    def sigma(i):
        for w, (A, B) in enumerate(((L, Gt), (Gt, L))):
            g, gb = A[i, :i + 1], -B[i, :i + 1].conj().transpose(1, 2)
            out = SPIN * g * (V @ (g * gb.transpose(1, 2)) @ V)
            for b in range(n):
                P = (g * V[b][None, None, :]) @ gb
                out[:, :, b] -= torch.einsum("ak,jak,jk->ja", V, P, g[:, :, b])
            S[w, :i + 1] = out

    def collide(i, j):
        wi, wj = weights(i), weights(j)
        d = (S[1, :i + 1] - S[0, :i + 1]) * wi[:, None, None]
        D = (L[:j + 1, j] - Gt[:j + 1, j]) * wj[:, None, None]
        return ((d @ L[:i + 1, j]).sum(0) + (S[0, :j + 1] @ D).sum(0),
                (d @ Gt[:i + 1, j]).sum(0) + (S[1, :j + 1] @ D).sum(0))

    def rhs(i):
        hi, _ = hhf(i)
        both = [collide(i, j) for j in range(i + 1)]
        return [[-1j * hi @ F[i, j] + both[j][q] for j in range(i + 1)] for q, F in enumerate((L, Gt))]

    def advance(i, R0, R1=None):
        f = dt if R1 is None else 0.5 * dt
        for q, F in enumerate((L, Gt)):
            for j in range(i + 1):
                F[i + 1, j] = F[i, j] + f * (R0[q][j] if R1 is None else R0[q][j] + R1[q][j])
                F[j, i + 1] = F[i + 1, j].conj().T
        X = R0[0][i] + R0[0][i].conj().T
        if R1 is not None:
            X = X + R1[0][i + 1] + R1[0][i + 1].conj().T
        L[i + 1, i + 1] = L[i, i] + f * X
        Gt[i + 1, i + 1] = L[i + 1, i + 1] - eye

    def observe(i):
        r = L[i, i]
        _, s = hhf(i)
        K, _ = collide(i, i)
        e = (torch.trace(h @ r) + (_dev(dv[i]).to(z) * torch.diagonal(r)).sum()).real
        E.append(float(SPIN * e + 0.5 * SPIN * torch.trace(s @ r).real
                       + 0.5 * SPIN * torch.trace(1j * K).real))
        N.append(float(SPIN * torch.trace(r).real))
        rho.append(r.cpu().numpy().copy())

    sigma(0)
    observe(0)
    for i in range(steps):
        R0 = rhs(i)
        advance(i, R0)
        sigma(i + 1)
        advance(i, R0, rhs(i + 1))
        sigma(i + 1)
        observe(i + 1)
    return dict(rho=np.array(rho), E=np.array(E), N=np.array(N))


def _field(c, seed):
    """A dipole field x_a E(t): E(t) = amp sin(omega t) sin^2(pi t / t_end)."""
    r = np.random.Generator(np.random.PCG64([int(seed), 17]))
    t = np.arange(c["steps"] + 1) * c["dt"]
    e = r.uniform(0.05, 0.15) * np.sin(r.uniform(0.6, 1.2) * t) * np.sin(np.pi * t / t[-1]) ** 2
    x, _, _ = _basis(c["n_elem"], c["order"], c["half"])
    return e[:, None] * x[None, :]


def _hf_of(c, seed, **kw):
    return _hf(c["species"], c["n_elem"], c["order"], c["half"], c["beta"], seed, **kw)


def _stacks(c, seed):
    """g on the mesh (the HF Green's function), V, and for the convolution the direct term of the
    self-energy and the change of the HF self-energy a first iteration brings."""
    hf = _hf_of(c, seed, iterations=12)  # inputs only: a few HF iterations give their shape
    tau, _, _, _ = _mesh(c["beta"], c["u"], c["p"])
    G, V = _g0(hf, tau, c["beta"]).contiguous(), _dev(hf["V"])
    s = dict(V=V, G=G)
    if c["kind"] == "conv":
        s["Sigma"] = _direct(G, V).contiguous()
        s["Sigma"] = (0.5 * (s["Sigma"] + s["Sigma"].transpose(1, 2))).contiguous()
        r = np.random.Generator(np.random.PCG64([int(seed), 5]))
        d = r.uniform(-1e-3, 1e-3, hf["V"].shape) * hf["V"]
        s["dHF"] = _dev(0.5 * (d + d.T))
    return s


def _mlp_data(c, seed):
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    M, H, rows = c["M"], c["hidden"], c["rows"]
    din = 2 * M + 3
    # feature rows fall off along tau like the self-energy and g do
    fall = torch.exp(-torch.linspace(0.0, 6.0, din, device="cuda"))
    X = torch.randn(rows, din, generator=g, device="cuda") * fall
    T = 0.1 * torch.randn(rows, M, generator=g, device="cuda")
    par = []
    for a, b in ((din, H), (H, H), (H, M)):
        par.append(torch.randn(a * b, generator=g, device="cuda") * math.sqrt(2.0 / a))
        par.append(0.01 * torch.randn(b, generator=g, device="cuda"))
    return X, T, torch.cat(par).cpu().numpy()


def _mlp_exact(c, seed):
    X, T, params = _mlp_data(c, seed)
    M, H = c["M"], c["hidden"]
    w, at, leaves = torch.from_numpy(params).cuda().double(), 0, []
    for shape in ((2 * M + 3, H), (H,), (H, H), (H,), (H, M), (M,)):
        size = math.prod(shape)
        leaves.append(w[at:at + size].reshape(shape).requires_grad_())
        at += size
    W1, b1, W2, b2, W3, b3 = leaves
    y = torch.relu(torch.relu(X.double() @ W1 + b1) @ W2 + b2) @ W3 + b3
    loss = ((y - T.double()) ** 2).sum() / (2.0 * T.numel())
    g = torch.autograd.grad(loss, leaves)
    return dict(loss=float(loss.detach()), grad=torch.cat([v.reshape(-1) for v in g]).float().cpu().numpy())


def _batch_grids(c):
    r = np.random.Generator(np.random.PCG64([int(c["grids"]), 4]))
    out = []
    for k in range(c["systems"]):
        order = int(r.integers(4, 9))
        out.append(dict(species="he" if k % 2 == 0 else "h3p", order=order,
                        n_elem=int(r.integers(-(-60 // order), 130 // order + 1)),
                        half=50.0 if k % 2 == 0 else 60.0))
    return out


def _context(c, seed):
    ctx = Context()
    ctx.build_fedvr(c["n_elem"], c["order"] + 1, -c["half"], c["half"], 0)
    Z, R = _nuclei(c["species"], seed)
    ctx.set_potential(Z, R, 1.0, 1.0, 2)
    return ctx


# --------------------------------------------------------------------------------------------
# The measured interface
# --------------------------------------------------------------------------------------------
def prepare(case, seed):
    c, k = case, case["kind"]
    if k == "mlp":
        net = WarmStartNet(c["M"], c["hidden"])
        X, T, params = _mlp_data(c, seed)
        net.set_params(params)
        return dict(case=c, net=net, X=X.contiguous(), T=T.contiguous())
    if k == "batch":
        ctxs = []
        for q, g in enumerate(_batch_grids(c)):
            ctx = _context(g, seed + 1000 * q)
            ctx.solve_hf(c["beta"], tol=1e-11)
            ctxs.append(ctx)
        M = 2 * c["u"] * c["p"] + 1
        out = [[torch.empty((M, x.n_b, x.n_b), dtype=torch.float64, device="cuda")
                for _ in range(2)] for x in ctxs]
        return dict(case=c, ctxs=ctxs, out=out)
    if k in ("sigma2", "conv", "gw", "tmatrix"):
        s = _stacks(c, seed)
        return dict(s, case=c, ctx=Context(), out=torch.empty_like(s["G"]))
    ctx = _context(c, seed)
    s = dict(case=c, ctx=ctx)
    if k == "hf":
        return s
    ctx.solve_hf(c["beta"], tol=1e-12)
    if k == "kbe":
        return dict(s, dv=_field(c, seed))
    ctx.prepare_2b(c["beta"], c["u"], c["p"], PRECISION[c["precision"]])
    G = torch.empty((2 * c["u"] * c["p"] + 1, ctx.n_b, ctx.n_b), dtype=torch.float64, device="cuda")
    ctx.read_2b(G_out=G)
    return dict(s, G=G, G_out=torch.empty_like(G), S_out=torch.empty_like(G))


def run(state):
    c = state["case"]
    k = c["kind"]
    if k == "mlp":
        loss, grad = state["net"].loss_grad(state["X"], state["T"])
        return dict(loss=loss, grad=grad)
    if k == "batch":
        r = solve_2b_batched(state["ctxs"], c["beta"], c["u"], c["p"], MIXING, 1e-6, 60,
                             PRECISION[c["precision"]], check=False)
        for ctx, (G, S) in zip(state["ctxs"], state["out"]):
            ctx.read_2b(G_out=G, Sigma_out=S)
        return dict(E0=r["E0"], N=r["N"], iters=r["iters"], stacks=state["out"])
    ctx = state["ctx"]
    if k == "hf":
        E, mu = ctx.solve_hf(c["beta"], tol=1e-12)
        d = ctx.get_hf()
        # the eigenvectors C are defined up to their signs; rho0 and Sigma0 are built from them
        return dict(E=E, mu=mu, eps=d["eps"], rho0=d["rho0"], Sigma0=d["Sigma0"])
    if k == "kbe":
        r = ctx.kbe_propagate(c["dt"], c["steps"], True, dv=state["dv"],
                              precision=PRECISION[c["precision"]])
        return dict(rho=r["rho"], E=r["E"], N=r["N"])
    if k == "step":
        r = ctx.step_2b(MIXING, G_in=state["G"])
        ctx.read_2b(G_out=state["G_out"], Sigma_out=state["S_out"])
        return dict(res=r["res"], E0=r["E0"], N=r["N"], G=state["G_out"], Sigma=state["S_out"])
    if k == "sigma2":
        ctx.sigma2(state["V"], state["G"], state["out"], SPIN, PRECISION[c["precision"]])
    elif k == "conv":
        ctx.conv_sigma_g(c["beta"], c["u"], c["p"], state["dHF"], state["Sigma"], state["G"],
                         state["out"], PRECISION[c["precision"]])
    elif k == "gw":
        ctx.sigma_gw(c["beta"], c["u"], c["p"], state["V"], state["G"], state["out"], SPIN)
    else:
        ctx.sigma_tmatrix(c["beta"], c["u"], c["p"], state["V"], state["G"], state["out"], SPIN)
    return state["out"]


def work(case):
    c, k = case, case["kind"]
    if k == "mlp":
        M, H, rows = c["M"], c["hidden"], c["rows"]
        par = (2 * M + 3) * H + H * H + H * M + 2 * H + M
        # forward, the weight gradients, and the input gradients of layers 2 and 3
        flops = 2.0 * rows * (2 * ((2 * M + 3) * H) + 3 * (H * H + H * M))
        return dict(bytes=4.0 * (rows * (3 * M + 3) + 2 * par), flops=flops)
    if k == "batch":
        M = 2 * c["u"] * c["p"] + 1
        f = b = 0.0
        for g in _batch_grids(c):
            n = g["n_elem"] * g["order"] - 1
            f += 20 * (2.0 * M * M * n ** 3 + M * (float(n) ** 4 + 4.0 * n ** 3))  # about 20 iterations
            b += 8.0 * (2.0 * M * n * n + 4.0 * n * n)
        return dict(bytes=b, flops=f)
    n = float(c["n_elem"] * c["order"] - 1)
    if k == "hf":  # about 20 iterations of a symmetric eigenproblem
        return dict(bytes=8.0 * 5 * n * n, flops=20 * 9.0 * n ** 3)
    if k == "kbe":
        T = c["steps"] + 1
        coll = sum(2.0 * 8.0 * 2.0 * (i + 1) * (1.5 * i + 3) * n ** 3 for i in range(T))
        sig = sum(2.0 * 8.0 * 2 * (i + 1) * (n ** 4 + 2 * n ** 3) for i in range(T))
        return dict(bytes=8.0 * (T * n + 2.0 * T * n * n), flops=coll + sig)
    M = 2.0 * c["u"] * c["p"] + 1
    stack = M * n * n
    if k == "sigma2":
        return dict(bytes=8.0 * (2 * stack + n * n), flops=M * (n ** 4 + 4 * n ** 3))
    if k == "conv":
        return dict(bytes=8.0 * (3 * stack + n * n), flops=2.0 * M * M * n ** 3)
    if k == "gw":  # about 40 inner iterations of the periodic convolution
        return dict(bytes=8.0 * (2 * stack + n * n), flops=40 * 2.0 * M * M * n ** 3)
    if k == "tmatrix":  # about 40 inner iterations of the ladder
        return dict(bytes=8.0 * (2 * stack + n * n), flops=40 * 4.0 * M * M * n ** 5)
    return dict(bytes=8.0 * (4 * stack + 3 * n * n),
                flops=2.0 * M * M * n ** 3 + M * (n ** 4 + 8 * n ** 3) + 2.0 * M * M * n * n)


def exact(case, seed):
    c, k = case, case["kind"]
    if k == "batch":
        return None  # twenty float64 iterations of every system
    if k == "mlp":
        return _mlp_exact(c, seed)
    if k == "hf":
        hf = _hf_of(c, seed)
        return dict(E=float(hf["E"]), mu=float(hf["mu"]), eps=hf["eps"], rho0=hf["rho"],
                    Sigma0=hf["Sigma0"])
    if k == "kbe":
        if c["steps"] > 30:
            return None  # minutes of small float64 products
        return _kbe_exact(_hf_of(c, seed), c["dt"], c["steps"], _field(c, seed))
    if k != "step":
        s = _stacks(c, seed)
        n, M = s["G"].shape[1], s["G"].shape[0]
        if k == "sigma2":
            return _sigma2_exact(s["G"], s["V"]) if 2.0 * M * n ** 4 < 6e12 else None
        if k == "conv":
            return _conv1_exact(s["dHF"], s["Sigma"], s["G"], c["beta"], c["u"], c["p"])
        if k == "gw":
            return _gw_exact(s["G"], s["V"], c["beta"], c["u"], c["p"])
        return _tmatrix_exact(s["G"], s["V"], c["beta"], c["u"], c["p"])
    hf = _hf_of(c, seed)
    tau, w, _, _ = _mesh(c["beta"], c["u"], c["p"])
    V = _dev(hf["V"])
    G = _g0(hf, tau, c["beta"])
    S = _sigma2_exact(G, V)
    rho = G[-1].cpu().numpy()
    shf = _hf_sigma(rho, hf["V"])
    corr = float((_dev(w) * (S.flip(0) * G).sum((1, 2))).sum())
    E0 = SPIN * np.sum(hf["h"] * rho) + 0.5 * SPIN * np.sum(shf * rho) - 0.5 * SPIN * corr
    I1 = _conv1_exact(_dev(shf - hf["Sigma0"]), S, G, c["beta"], c["u"], c["p"])
    new = G + _conv2_exact(I1, hf, c["beta"], c["u"], c["p"])
    new = (1.0 - MIXING) * G + MIXING * 0.5 * (new + new.transpose(1, 2))
    return dict(res=float((new - G).abs().max()), E0=float(E0), N=float(SPIN * np.trace(rho)), G=new,
                Sigma=S)
