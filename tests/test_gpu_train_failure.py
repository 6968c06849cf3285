"""GPU test of a training step that gives up waiting for its weights: a limit of
no polls makes the first wait run out.  The calls that synchronise report it,
no parameter and no Adam moment changes in that step or a later one, and after
set_params the network trains as a new one does, bit for bit."""
import numpy as np
import pytest

from test_gpu_mlp import _random_net, _raw_inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
ETIMEDOUT = -4


def _batch(M):
    rng = np.random.default_rng(M)
    x = _raw_inputs(rng, M).astype(np.float32)
    t = np.stack([rng.normal(0.1, 0.2, M), rng.normal(-3.0, 1.5, M)], axis=1).astype(np.float32)
    return torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda()


def _raises(call, *args, **kw):
    from paper_1409_4923_gb300 import engine
    with pytest.raises(engine.SdeError) as e:
        call(*args, **kw)
    assert e.value.code == ETIMEDOUT


@pytest.mark.parametrize("M", [33, 600, 2433])          # one, several and 32-row blocks of the chain
def test_a_step_that_gives_up_changes_nothing_and_is_reported(M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import surrogate as S
    x, t = _batch(M)
    net, p, _ = _random_net(S, 31)
    ref, _, _ = _random_net(S, 31)
    try:
        fit = dict(steps=3, batch=min(M, 512), lr=1e-3, lr_final=1e-4, seed=2)
        net.train_step(x, t, 1e-3)
        before = net.get_params()
        net.set_wait_polls(0)
        net.train_step(x, t, 1e-3)
        _raises(net.sync)
        _raises(net.get_params)
        net.set_wait_polls(1 << 24)
        net.train_step(x, t, 1e-3)                        # a later step, its waits in order
        _raises(net.fit, x, t, **fit)
        _raises(net.gradients, x, t)
        after = np.zeros_like(before)
        assert net._L.sde_mlp_get_params(net._net, after.ctypes.data) == ETIMEDOUT
        np.testing.assert_array_equal(after, before)
        # a new start: the same losses and parameters as a network that never failed
        for n in (net, ref):
            n.set_params(p)
        losses = [n.fit(x, t, **fit) for n in (net, ref)]
        np.testing.assert_array_equal(losses[0], losses[1])
        np.testing.assert_array_equal(net.get_params(), ref.get_params())
    finally:
        net.close()
        ref.close()
