"""The launch autotuner and the kernels for runs of few paths: a tuning on one
side of their limit, or with kernels of another generation, never serves the
other, and no grid is chosen that would keep such a run from them."""
import pytest

from paper_1409_4923_gb300 import autotune as AT, engine as E


def test_the_few_path_limit_parts_a_size_class():
    assert AT.size_class(20000) == AT.size_class(60000)
    assert AT.key("GB300", 0, 3, 20000, True) != AT.key("GB300", 0, 3, 60000, False)


def test_tunings_of_other_kernel_generations_are_not_used(monkeypatch):
    now = AT.key("GB300", 0, 3, 1024)
    assert now != "GB300|model=0|flags=3|paths~4^5"
    monkeypatch.setattr(AT, "KERNEL_GENERATION", AT.KERNEL_GENERATION + 1)
    assert AT.key("GB300", 0, 3, 1024) != now


@pytest.mark.gpu
def test_few_paths_keep_the_default_shape(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1409_4923_gb300 import workloads as W
    spec = W.run_spec("poisson_1024")
    prm = E.make_params(**spec["params"])
    cache = str(tmp_path / "tune.json")
    t = AT.tune(spec["model"], prm, spec["dt"], 1024, n_probe_steps=512, cache=cache)
    assert list(t["seconds"]) == [(128, 0, 1)] and (t["block"], t["grid"], t["ppt"]) == (128, 0, 1)
    assert AT.tune(spec["model"], prm, spec["dt"], 1024, cache=cache) == {f: t[f] for f in AT.DEFAULT}
