"""GPU: the split exchange of a launch that mixes systems on both sides of n = 256.
Every CTA goes through several tiles of each system, largest first, so that the
halves of the columns pass from one system to the next at different times. The
self-energy of the first iteration is a function of the starting g alone and every
sum is taken in the order of the system's own launch, so it equals the one-system
run's bit for bit."""
import numpy as np
import pytest

from paper_0911_4348_gb300 import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# n = 304 (19 chunks of 16 columns), 272, 160: widths 304, 272 and 160
GRIDS = [(61, 5), (39, 7), (23, 7)]


def _ctx(n_elem, order):
    from paper_0911_4348_gb300 import Context
    c = Context()
    c.build_fedvr(n_elem, order + 1, -40.0, 40.0, 0)
    c.set_potential([2.0], [0.0], 1.0, 1.0, 2)
    c.solve_hf(20.0, tol=1e-10)
    c.conv1_splits(1)
    return c


@pytest.mark.parametrize("precision", ["SPLIT_TF32", "SPLIT_F16"])
def test_mixed_launch_equals_single(precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0911_4348_gb300 as P
    prec = getattr(P, precision)
    u, p, beta = 2, 8, 20.0
    M = 2 * u * p + 1
    single = []
    ctxs = [_ctx(*g) for g in GRIDS]
    try:
        for c, (n_elem, order) in zip(ctxs, GRIDS):
            n = n_elem * order - 1
            S = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
            c.solve_2b(beta, u, p, 0.5, 1e-30, 1, precision=prec, Sigma_out=S, check=False)
            single.append(S.cpu().numpy())
        # the order of the systems is the order of the work: large ones first, and back
        for order in ([0, 1, 2], [0, 2, 1]):
            P.solve_2b_batched([ctxs[k] for k in order], [beta] * 3, [u] * 3, [p] * 3, 0.5, 1e-30, 1,
                               prec, check=False)
            for k in order:
                S = torch.empty_like(torch.from_numpy(single[k])).cuda()
                ctxs[k].read_2b(Sigma_out=S)
                assert np.array_equal(S.cpu().numpy(), single[k]), (order, k)
    finally:
        for c in ctxs:
            c.close()
