"""GPU: the scratch of the warm-start network's weight gradients is what the slices of
the mini-batch take, not sixteen copies of the largest layer, and inference takes none."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _free():
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_scratch_of_the_largest_network():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import WarmStartNet
    M, H, rows = 4097, 4096, 64
    net = WarmStartNet(M, H, seed=1)
    try:
        X = torch.zeros((rows, 2 * M + 3), dtype=torch.float32, device="cuda")
        X[:, 0] = 1.0
        T = torch.zeros((rows, M), dtype=torch.float32, device="cuda")
        before = _free()
        loss, grad = net.loss_grad(X, T)
        used = before - _free()
    finally:
        net.close()
    assert np.isfinite(loss) and np.all(np.isfinite(grad))
    # activations, outputs and deltas of 64 rows are below 10 MB; allocations come in
    # pieces of 2 MB; one layer's partial result alone would be 134 MB
    assert used < 64 << 20


def test_inference_takes_no_slices():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import WarmStartNet
    M, H, rows = 1025, 2048, 64  # 16 slices of the widest layer were 268 MB
    net = WarmStartNet(M, H, seed=1)
    try:
        X = torch.zeros((rows, 2 * M + 3), dtype=torch.float32, device="cuda")
        Y = torch.empty((rows, M), dtype=torch.float32, device="cuda")
        before = _free()
        net.forward(X, Y)
        used = before - _free()
    finally:
        net.close()
    assert used < 64 << 20
