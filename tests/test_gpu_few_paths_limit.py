"""GPU test of the line between the few-path kernels and the others: it lies at
the measured number of 32-path blocks per SM for each noise combination, and
runs, cut runs and step-size probes at the line and one path past it are those
of the persistent kernels (a grid set by hand) bit for bit."""
import numpy as np
import pytest

from test_gpu_split import _outputs, _params

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def E():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import engine
    return engine


def _sms():
    return torch.cuda.get_device_properties(torch.cuda.current_device()).multi_processor_count


# noise flags as in test_gpu_split; 32-path blocks per SM by model
@pytest.mark.parametrize("flags,blocks", [
    (0, (0, 0, 0)), (1, (6, 8, 8)), (2, (8, 8, 8)), (4, (8, 8, 8)), (7, (8, 8, 8)), (6 | 32, (8, 8, 8)),
    (7 | 32, (6, 6, 6)), (1 | 8, (24, 24, 24)), (3 | 8, (24, 24, 24)), (5 | 8, (24, 14, 14)),
    (5 | 8 | 32, (24, 14, 14)), (7 | 8 | 32, (24, 24, 24)), (4 | 8, (8, 8, 8))])
def test_limit_by_noise(E, flags, blocks):
    for model in (0, 1, 2):
        prm = E.make_params(**_params(model, flags))
        assert E.few_paths_limit(model, prm) == 32 * blocks[model] * _sms(), model


def test_limit_refuses_bad_parameters(E):
    with pytest.raises(E.SdeError):
        E.few_paths_limit(0, E.make_params(gamma=0.0))


@pytest.mark.parametrize("model,flags", [(0, 1), (0, 7 | 32), (1, 5 | 8)])
def test_both_sides_of_the_line_agree_with_the_persistent_kernels(E, model, flags):
    prm = E.make_params(**_params(model, flags))
    limit = E.few_paths_limit(model, prm)
    for paths in (limit, limit + 1):
        r = []
        for grid in (0, 2 * _sms()):
            eng = E.Engine(model, prm, seed=9)
            eng.set_tuning(64, grid)
            got = []
            for steps in (0, 32):
                out = _outputs(paths)
                eng.set_steps_per_launch(steps)
                eng.run(paths, 0.01, 8, 60, path_out=out)
                got += [eng.stats()["sums"]] + [v.cpu().numpy() for v in out.values()]
            got.append(list(eng.local_error(paths, 0.01, 20).values()))
            eng.close()
            r.append(got)
        for a, b in zip(*r):
            np.testing.assert_array_equal(a, b)
