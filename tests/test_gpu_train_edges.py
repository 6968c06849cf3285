"""GPU test of the training kernels at the edges of their tiles: one row, a row
short of and past a 16-row tile, past a 256-row split of the weight gradients,
past two and four splits side by side, and both sides of the change from 16 to
32 rows per block.  The bar is that of test_gpu_mlp's gradient test: every
gradient entry within 8 standard deviations of its propagated BF16 rounding
error around the FP64 oracle on the same BF16 weights and FP32 biases."""
import numpy as np
import pytest

from oracle import mlp as omlp
from test_gpu_mlp import K_SIGMA, _grad_error_sigma, _random_net, _raw_inputs, bf16_round

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M", [1, 15, 17, 257, 513, 1025, 2432, 2433, 4999])
def test_gradients_at_tile_edges(M):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import surrogate as S
    net, p, (shift, scale, mask, osh, osc) = _random_net(S, 31)
    rng = np.random.default_rng(M)
    x = _raw_inputs(rng, M).astype(np.float32)
    t = np.stack([rng.normal(0.1, 0.2, M), rng.normal(-3.0, 1.5, M)], axis=1).astype(np.float32)
    try:
        g, L = net.gradients(torch.from_numpy(x).cuda(), torch.from_numpy(t).cuda())
    finally:
        net.close()
    P = omlp.unflatten(p)
    for name in P:
        w = P[name].astype(np.float32)
        P[name] = bf16_round(w) if name[0] == "W" else w.astype(np.float64)
    pm = omlp.flatten(P)
    xp = omlp.input_map(x.astype(np.float64), shift.astype(np.float32), scale.astype(np.float32), mask)
    tp = (t - osh) / osc
    L0, g0 = omlp.loss_and_grad(pm, xp, tp)
    assert abs(L - L0) <= 0.03 * L0
    G, G0, sigma = omlp.unflatten(g.astype(np.float64)), omlp.unflatten(g0), _grad_error_sigma(pm, xp, tp, M)
    live = {"W1": np.s_[:, :7], "W4": np.s_[:2], "b4": np.s_[:2]}
    for name, _ in omlp.SHAPES:
        s = live.get(name, np.s_[:])
        assert np.all(np.abs(G[name][s] - G0[name][s]) <= K_SIGMA * sigma[name][s] + 1e-12), name
    assert not G["W1"][:, 7:].any() and not G["W4"][2:].any() and not G["b4"][2:].any()
