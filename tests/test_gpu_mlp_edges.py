"""Loss, gradients and inference of the warm-start network at the edges of the
product kernels' tiles (128 x 64 outputs, 16-wide slices, the mini-batch cut
into slices of at least 64 rows) against the FP64 reference. FP32 sums of up to
1000 terms carry 1000 x 2^-24 = 6e-5 of their largest partial sum at most."""
import numpy as np
import pytest

from oracle import mlp_oracle as N
from paper_0911_4348_gb300 import workloads as W
from tests.test_gpu_mlp import _flat, _unflat

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,M,H", [(1, 17, 32), (63, 17, 33), (65, 31, 64), (127, 63, 65),
                                      (129, 65, 128), (1000, 33, 129), (513, 129, 63)])
def test_gradient_and_forward(rows, M, H):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import WarmStartNet
    din = 2 * M + 3
    rng = W.system_rng(83, rows)
    P = N.init_params(din, H, M, rng)
    for k in ("b1", "b2", "b3"):
        P[k] = rng.normal(0.0, 0.05, P[k].shape)
    X = rng.normal(size=(rows, din)).astype(np.float32)
    T = rng.normal(size=(rows, M)).astype(np.float32)
    net = WarmStartNet(M, H, seed=1)
    net.set_params(_flat(P).astype(np.float32))
    P32 = _unflat(_flat(P).astype(np.float32).astype(np.float64), din, H, M)
    y, cache = N.forward(P32, X.astype(np.float64))
    want = N.backward(P32, cache, y, T.astype(np.float64))
    loss, grad = net.loss_grad(torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda())
    want_loss = N.loss(y, T.astype(np.float64))
    assert abs(loss - want_loss) < 1e-5 * want_loss
    got = _unflat(grad.astype(np.float64), din, H, M)
    for k in want:
        assert np.max(np.abs(got[k] - want[k])) < 1e-4 * np.max(np.abs(want[k])), k
    Y = torch.empty((rows, M), dtype=torch.float32, device="cuda")
    net.forward(torch.from_numpy(X).cuda(), Y)
    torch.cuda.synchronize()
    assert np.max(np.abs(Y.cpu().numpy() - y)) < 1e-5 * np.max(np.abs(y))
    net.close()
