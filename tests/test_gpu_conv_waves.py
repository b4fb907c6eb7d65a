"""GPU: the stage-level first convolution's own choice of its work split. 161 row
tiles are one full wave of a 152-SM GPU and nine CTAs more, so the call splits
the mesh range; above n = 256 a row tile is two items. The block sums are those of
one split: only the order of their FP64 additions differs (1e-13, as for requested
splits)."""
import numpy as np
import pytest

from paper_0911_4348_gb300 import workloads as W
from tests._systems import maxrel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["SPLIT_TF32", "SPLIT_F16"])
@pytest.mark.parametrize("n,u", [(64, 10), (257, 2)])
def test_chosen_split_agrees_with_one(n, u, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0911_4348_gb300 as P
    p, beta = 16, 10.0
    M = 2 * u * p + 1
    rng = W.system_rng(98, n)
    G = torch.from_numpy(W.random_symmetric_stack(rng, M, n)).cuda()
    S = torch.from_numpy(W.random_symmetric_stack(rng, M, n)).cuda()
    d = torch.from_numpy(W.random_symmetric(rng, n)).cuda()
    out, used = [], []
    ctx = P.Context()
    try:
        for request in (0, 1):
            ctx.conv1_splits(request)
            I1 = torch.empty_like(G)
            ctx.conv_sigma_g(beta, u, p, d, S, G, I1, getattr(P, precision))
            torch.cuda.synchronize()
            out.append(I1.cpu().numpy())
            used.append(ctx.conv1_splits())
    finally:
        ctx.close()
    assert used[1] == 1
    if n == 64 and torch.cuda.get_device_properties(0).multi_processor_count == 152:
        assert used[0] > 1
    assert np.all(np.isfinite(out[0]))
    assert maxrel(out[0], out[1]) < 1e-13
