"""GPU test of the runs that draw their noise in warps of their own (few paths)
against the persistent kernels (a grid set by hand): every noise combination
of every model, path counts and step counts off the 32-step blocks, whole runs,
runs cut into launches and segments cut anywhere.  The two take the same
operations, so every output is equal bit for bit."""
import numpy as np
import pytest

import gpu_common as gc

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

# Gaussian, Poisson, dichotomous, Box-Muller (8), compensated (16), dichotomous drift (32)
FLAGS = [1, 2, 4, 3, 5, 6, 7, 4 | 32, 7 | 32, 1 | 8, 3 | 8 | 16, 5 | 8, 7 | 8, 7 | 8 | 32]
MODELS = {0: dict(gamma=0.9, a=4.2, omega=4.9, F=0.1, V0=1.0, Q=0.01, v0_lo=-2.0, v0_hi=2.0),
          1: dict(a=0.5, omega=4.9, F=0.1, V0=0.2, Q=0.05),
          2: dict(a=0.3, omega=4.9, F=0.1, V0=1.0, Q=0.01, x0_lo=-1.0)}


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import engine
    return engine


def _params(model, flags):
    return dict(MODELS[model], x0_hi=1.0, zeta=0.1, Fa=0.5, Fb=0.8, mua=2.0, mub=3.0, noise_flags=flags,
                **{"lambda": 4.0})


def _outputs(paths):
    return {k: torch.zeros(paths, dtype=t, device="cuda") for k, t in (
        ("X_f", torch.float64), ("v_f", torch.float32), ("vbar", torch.float64), ("jP", torch.int32),
        ("jD", torch.int32))}


def _run(E, model, flags, paths, n_tr, n_avg, grid, how):
    eng = E.Engine(model, E.make_params(**_params(model, flags)), seed=9)
    try:
        eng.set_tuning(64, grid)
        out, dt = _outputs(paths), 0.01
        if how == "cuts":
            eng.begin(paths, dt, n_tr, n_avg)
            for n in (17, 47, 64, 0):
                eng.advance(n, path_out=out)
        else:
            eng.set_steps_per_launch(how)
            eng.run(paths, dt, n_tr, n_avg, path_out=out)
        st = eng.stats()
    finally:
        eng.close()
    return st["sums"], {k: v.cpu().numpy() for k, v in out.items()}


@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("flags", FLAGS)
def test_split_runs_equal_persistent_runs(E, model, flags):
    for paths, n_tr, n_avg, how in ((33, 0, 1, 0), (70, 37, 400, 0), (64, 64, 320, 32), (33, 300, 291, 96),
                                    (65, 64, 200, "cuts"), (32, 0, 150, "cuts")):
        a = _run(E, model, flags, paths, n_tr, n_avg, 0, how)
        b = _run(E, model, flags, paths, n_tr, n_avg, 3, how)
        assert a[0] == b[0], (paths, n_tr, n_avg, how)
        for k in a[1]:
            np.testing.assert_array_equal(a[1][k], b[1][k], err_msg="%s %s" % (k, (paths, n_tr, n_avg, how)))


def test_far_coordinates_keep_the_conversions(E):
    """Kicks so large that folds leave the range of near_folds: the run takes the
    persistent kernel and both calls agree."""
    for model in (0, 1, 2):
        r = []
        for grid in (0, 3):
            eng = E.Engine(model, E.make_params(**dict(_params(model, 2), zeta=1e9)), seed=9)
            eng.set_tuning(64, grid)
            out = _outputs(40)
            eng.run(40, 0.01, 10, 200, path_out=out)
            r.append((eng.stats()["sums"], out["X_f"].cpu().numpy()))
            eng.close()
        np.testing.assert_array_equal(r[0][0], r[1][0])
        np.testing.assert_array_equal(r[0][1], r[1][1])


def test_far_coordinates_with_two_paths_per_lane(E):
    """The same kicks with two paths per lane asked for, in a run and in a scan of
    one launch per point: both take one path per lane and agree."""
    r = []
    for ppt, mode in ((1, 1), (2, 2)):
        prm = E.make_params(**dict(_params(0, 3), zeta=1e9))
        eng = E.Engine(0, prm, seed=9)
        eng.set_tuning(64, 3)
        eng.set_paths_per_thread(ppt)
        eng.set_scan_mode(mode)
        out = _outputs(100)
        eng.run(100, 0.01, 10, 200, path_out=out)
        scan = eng.scan([dict(params=prm, dt=0.01, paths=100, n_transient=10, n_avg=200)])
        r.append((eng.stats()["sums"], scan[0]["sums"], out["X_f"].cpu().numpy()))
        eng.close()
    for a, b in zip(*r):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("model", [0, 1, 2])
def test_far_coordinates_in_a_checkpoint(E, model):
    """A checkpoint whose coordinates and velocities lie beyond the near folds'
    range (its checksum valid): a restored run keeps the conversions."""
    eng = E.Engine(model, E.make_params(**_params(model, 3)), seed=9)
    eng.begin(64, 0.01, 40, 200)
    eng.advance(33)
    blob = bytearray(eng.checkpoint())
    eng.close()
    header, stride = 224, 64
    far = np.frombuffer(blob, dtype=np.float32, offset=header + 16 * stride, count=2 * stride).copy()
    far[3], far[stride + 7] = 3.0e8, -2.5e9
    blob[header + 16 * stride:header + 24 * stride] = far.tobytes()
    h = 0xcbf29ce484222325
    for byte in blob[header:]:
        h = ((h ^ byte) * 0x100000001b3) & 0xFFFFFFFFFFFFFFFF
    blob[216:224] = h.to_bytes(8, "little")
    r = []
    for grid in (0, 3):
        eng = E.Engine(model, E.make_params(**_params(model, 3)), seed=9)
        eng.set_tuning(64, grid)
        eng.restore(bytes(blob))
        out = _outputs(64)
        eng.advance(0, path_out=out)
        r.append([eng.stats()["sums"]] + [v.cpu().numpy() for v in out.values()])
        eng.close()
    for a, b in zip(*r):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("model", [0, 1, 2])
@pytest.mark.parametrize("flags", FLAGS)
def test_split_probes_equal_persistent_probes(E, model, flags):
    """Step-size probes (local_error) of few paths against the one-warp kernel."""
    for paths, steps in ((33, 1), (70, 45), (64, 288), (32, 600)):
        r = []
        for grid in (0, 3):
            eng = E.Engine(model, E.make_params(**_params(model, flags)), seed=9)
            eng.set_tuning(64, grid)
            r.append(eng.local_error(paths, 0.01, steps))
            eng.close()
        assert r[0] == r[1], (paths, steps)
