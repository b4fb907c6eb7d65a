"""GPU vs oracle: the tensor-core exchange where its epilogue has no room to stage
rows (n > 224): two accumulators up to n = 256, one above with products waiting in
tensor memory; both halves of the columns at their smallest and largest. The
tolerance is that of the split exchange elsewhere: three products of operands
with 22 significant bits and sums of n^2 terms in FP32, 1e-5 of the largest entry."""
import numpy as np
import pytest

from oracle import fedvr_oracle as O
from paper_0911_4348_gb300 import workloads as W
from tests._systems import maxrel

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["SPLIT_TF32", "SPLIT_F16"])
@pytest.mark.parametrize("n,M", [(224, 3), (225, 3), (256, 2), (257, 3), (273, 2), (304, 3)])
def test_exchange_of_large_systems(n, M, precision):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_0911_4348_gb300 as P
    rng = W.system_rng(97, n)
    G = W.random_symmetric_stack(rng, M, n)
    V = W.random_symmetric(rng, n)
    S = torch.empty((M, n, n), dtype=torch.float64, device="cuda")
    ctx = P.Context()
    try:
        ctx.sigma2(torch.from_numpy(V).cuda(), torch.from_numpy(G).cuda(), S, spin=2.0,
                   precision=getattr(P, precision))
        torch.cuda.synchronize()
    finally:
        ctx.close()
    got = S.cpu().numpy()
    assert maxrel(got, O.sigma2(G, V, 2.0)) < 1e-5
    assert np.array_equal(got, got.transpose(0, 2, 1))
