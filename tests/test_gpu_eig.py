"""GPU vs oracle: the Hartree-Fock eigenproblem at the edges of its kernels
(tiles of 16 rotation pairs, products in tiles of 8), with clusters of levels
closer than any coupling (two far atoms), and the Fermi level where one level
counts and where all do. Tolerances are those of the Hartree-Fock parity test:
energies 1e-12 relative, levels 1e-10 of the largest."""
import numpy as np
import pytest

from oracle import fedvr_oracle as O
from tests._systems import maxrel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_elem,order,half,Z,R,n_elec,beta", [
    (1, 3, 3.0, [2.0], [0.0], 2, 10.0),
    (8, 4, 8.0, [2.0], [0.1], 2, 100.0),
    (11, 3, 8.0, [1.0, 1.0], [-0.9, 0.9], 2, 40.0),
    (17, 2, 8.0, [2.0], [0.0], 2, 2.0),
    (13, 5, 20.0, [2.0, 2.0], [-9.0, 9.0], 4, 100.0),
    (11, 6, 30.0, [2.0], [0.0], 2, 100.0),
    (26, 5, 60.0, [1.0, 1.0, 1.0], [-1.7, 0.0, 1.7], 2, 60.0),
])
def test_hf_eigenproblem_edges(n_elem, order, half, Z, R, n_elec, beta):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import Context
    b = O.fedvr_basis(n_elem, order, -half, half, 0)
    h = O.kinetic(b) + np.diag(O.potential(b["nodes"], Z, R, 1.0))
    V = O.interaction(b["nodes"], 1.0)
    want = O.hf_scf(h, V, 2.0, n_elec // 2, beta, tol=1e-13)
    ctx = Context()
    try:
        ctx.build_fedvr(n_elem, order + 1, -half, half, 0)
        ctx.set_potential(Z, R, 1.0, 1.0, n_elec)
        E, mu = ctx.solve_hf(beta, tol=1e-13, max_iter=500)
        got = ctx.get_hf()
    finally:
        ctx.close()
    big = max(1.0, np.max(np.abs(want["eps"])))
    assert abs(E - want["E_hf"]) < 1e-12 * max(1.0, abs(want["E_hf"]))
    assert abs(mu - want["mu"]) < 1e-10 * max(1.0, abs(want["mu"]))
    assert np.max(np.abs(got["eps"] - want["eps"])) < 1e-10 * big
    assert maxrel(got["rho0"], want["rho0"]) < 1e-11
    C = got["C"]
    assert np.max(np.abs(C.T @ C - np.eye(len(C)))) < 1e-12
    F = h + got["Sigma0"]
    assert np.max(np.abs(F @ C - C * got["eps"])) < 1e-10 * big
