"""GPU test of one network's forward buffer over calls of different sizes: the
buffer and its tensor maps are those of the largest call so far, the last tile
of a call reaches past its rows, and more than 2^20 rows go through it in two
chunks.  A row's outputs do not depend on the call that it is in, so every call
gives, bit for bit, the outputs of a network that has seen no other call."""
import numpy as np
import pytest

from test_gpu_mlp import _random_net, _raw_inputs

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

ROWS = 2 ** 20 + 777


@pytest.mark.parametrize("sizes", [(70001, 300, 1, 129, 128), (5, 4097, ROWS, 200, 152 * 128 + 33)])
def test_calls_of_different_sizes_over_one_buffer(sizes):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import surrogate as S
    x = torch.from_numpy(_raw_inputs(np.random.default_rng(3), max(sizes)).astype(np.float32)).cuda()
    net = _random_net(S, 12)[0]
    try:
        for M in sizes:
            part = x[x.shape[0] - M:].contiguous()           # other rows in each call
            y = net.forward(part)
            net.sync()
            new = _random_net(S, 12)[0]
            try:
                want = new.forward(part)
                new.sync()
            finally:
                new.close()
            assert torch.isfinite(y).all() and torch.equal(y, want), M
            # the same rows as calls of their own
            for a in (0, M // 2, M - 1):
                assert torch.equal(net.forward(part[a:a + 1].contiguous()), y[a:a + 1]), (M, a)
    finally:
        net.close()
