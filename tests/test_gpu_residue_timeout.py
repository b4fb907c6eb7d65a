"""GPU: a bounded wait of the FP64 path's residue kernels that gives up. Their result
is computed again in double arithmetic, but the timeout must not pass unseen: it
reaches the host without a copy and is returned by the next call that
synchronises, or by the next call at all. The wait runs out on a barrier that
nothing releases (1 ms)."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture()
def ctx():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_0911_4348_gb300 import Context
    c = Context()
    c.build_fedvr(4, 5, -10.0, 10.0)
    yield c
    c.close()


def test_the_next_call_returns_it(ctx):
    from paper_0911_4348_gb300 import FedvrError
    ctx.selftest_wait(2, 1e-3)
    torch.cuda.synchronize()
    with pytest.raises(FedvrError) as e:
        ctx.conv1_splits()  # a call that does not touch the GPU
    assert e.value.code == -5 and "residue" in str(e.value)
    with pytest.raises(FedvrError) as e:
        ctx.conv1_splits()
    assert e.value.code == -7  # failed, as after every timeout


def test_a_call_that_synchronises_returns_it(ctx):
    from paper_0911_4348_gb300 import FedvrError
    ctx.selftest_wait(2, 0.2)  # recorded while the next call is under way
    with pytest.raises(FedvrError) as e:
        ctx.set_potential([2.0], [0.0], 1.0, 1.0, 2)
    assert e.value.code == -5


def test_another_context_is_not_affected(ctx):
    from paper_0911_4348_gb300 import Context
    ctx.selftest_wait(2, 1e-3)
    torch.cuda.synchronize()
    other = Context()
    try:
        assert other.build_fedvr(4, 5, -10.0, 10.0) == 15
    finally:
        other.close()
