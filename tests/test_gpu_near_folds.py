"""GPU test of the folds that round by adding 1.5 2^23 (near folds): where
coordinates lie beyond their range, runs of few paths and two paths per lane
keep the conversions and agree with the persistent kernel (a grid set by hand,
one path per lane) bit for bit.  An FP32 emulation of both roundings asserts
that the coordinates used are ones where they differ."""
import numpy as np
import pytest

from test_gpu_split import _outputs, _params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")
F32 = np.float32
TWO_PI, INV = F32(6.2831853071795865), F32(0.15915494309189535)
SHIFT = F32(12582912.0)


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import engine
    return engine


def _roundings(model, c):
    """Whole periods that the conversion and the shifted sum take off FP32 coordinates c."""
    c = np.asarray(c, dtype=F32)
    if model == 2:
        half = (c + F32(1)).astype(np.float64) * 0.5           # exact
        up = (half + float(SHIFT)).astype(F32)                 # the sum is exact in FP64
        down = np.where(up > half + float(SHIFT), np.nextafter(up, F32(-np.inf)), up)
        return np.floor(half).astype(F32), down - SHIFT
    t = c * INV
    return np.rint(t), (t + SHIFT) - SHIFT


def _all_outputs(E, model, prm, ppt, grid, run):
    eng = E.Engine(model, prm, seed=9)
    try:
        eng.set_tuning(64, grid)
        eng.set_paths_per_thread(ppt)
        out = _outputs(64)
        run(eng, out)
        return [eng.stats()["sums"]] + [v.cpu().numpy() for v in out.values()]
    finally:
        eng.close()


def _same(E, model, prm, run):
    want = _all_outputs(E, model, prm, 1, 3, run)
    for ppt, grid in ((1, 0), (2, 3)):
        for a, b in zip(_all_outputs(E, model, prm, ppt, grid, run), want):
            np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("x0", [1e13, 1e15, -1e15])
def test_far_initial_coordinates(E, model, x0):
    """The first fold of a huge x0 leaves an FP32 residual beyond the near folds' range."""
    phi = np.arange(64) / 64.0
    c = (F32(x0) + F32(x0) * phi.astype(F32)) * TWO_PI
    left = (c.astype(np.float64) - np.rint(c * INV).astype(np.float64) * float(TWO_PI)).astype(F32)
    if model != 2 and abs(x0) > 1e14:
        near = _roundings(model, left)
        assert np.any(near[0] != near[1])
    prm = E.make_params(**dict(_params(model, 3), x0_lo=min(x0, 2 * x0), x0_hi=max(x0, 2 * x0)))
    _same(E, model, prm, lambda eng, out: eng.run(64, 0.01, 40, 200, path_out=out))


@pytest.mark.parametrize("model", [0, 1, 2])
def test_far_coordinates_of_a_checkpoint_where_the_roundings_differ(E, model):
    """A checkpoint (its checksum valid) whose coordinates the two roundings fold differently."""
    eng = E.Engine(model, E.make_params(**_params(model, 3)), seed=9)
    eng.begin(64, 0.01, 40, 200)
    eng.advance(33)
    blob = bytearray(eng.checkpoint())
    eng.close()
    odd = 2.0 * np.arange(2300000, 2300064) + 1.0             # whole periods, between 2^22 and 2^23
    c = ((odd * float(TWO_PI)) if model != 2 else 2.0 * odd - 0.5).astype(F32) * np.where(np.arange(64) % 2, 1, -1)
    c = c.astype(F32)
    near = _roundings(model, c)
    assert np.mean(near[0] != near[1]) > 0.25
    header, stride = 224, 64
    blob[header + 16 * stride:header + 20 * stride] = c.tobytes()
    h = 0xcbf29ce484222325
    for byte in blob[header:]:
        h = ((h ^ byte) * 0x100000001b3) & 0xFFFFFFFFFFFFFFFF
    blob[216:224] = h.to_bytes(8, "little")

    def run(eng, out):
        eng.restore(bytes(blob))
        eng.advance(0, path_out=out)
    _same(E, model, E.make_params(**_params(model, 3)), run)


@pytest.mark.parametrize("dt", [0.6, 0.9, 1.6, 2.2, 2.5])
def test_strong_damping_per_step(E, dt):
    """gamma dt from 0.54 to 2.25, up to and past the stability limit of a step
    (where paths may run off to infinities): packed pairs and few-path kernels
    against the persistent kernel, in runs and in a scan whose other points are
    ordinary ones or far beyond the near folds' range."""
    prm = E.make_params(**_params(0, 3))
    _same(E, 0, prm, lambda eng, out: eng.run(64, dt, 40, 200, path_out=out))
    points = [dict(params=p, dt=d, paths=100, n_transient=10, n_avg=200)
              for p, d in ((prm, dt), (prm, 0.01), (E.make_params(**dict(_params(0, 3), zeta=1e9)), 0.01), (prm, dt))]
    sums = []
    for mode in (1, 2):
        eng = E.Engine(0, prm, seed=9)
        eng.set_tuning(64, 3)
        eng.set_scan_mode(mode)
        sums.append([r["sums"] for r in eng.scan(points)])
        eng.close()
    np.testing.assert_array_equal(sums[0], sums[1])
