"""Packing of a scan's points: the same records, and the same refusals, as
assigning them to ScanPoint structures field by field."""
import ctypes

import pytest

from paper_1409_4923_gb300 import engine as E


class WithMore(E.Params):
    _fields_ = [("label", ctypes.c_double)]


def _by_field(points):
    arr = (E.ScanPoint * len(points))()
    for i, pt in enumerate(points):
        arr[i].p = pt["params"]
        arr[i].dt = float(pt["dt"])
        for k in ("paths", "n_transient", "n_avg"):
            setattr(arr[i], k, int(pt[k]))
    return arr


def _points(params):
    return [dict(params=p, dt=0.01 * (i + 1), paths=100 + i, n_transient=i, n_avg=7 - 9 * i)
            for i, p in enumerate(params)]


def test_points_are_packed_as_by_field():
    p = E.make_params(gamma=0.9, F=0.25, x0_hi=1.0, noise_flags=3, point=5, **{"lambda": 4.0})
    more = WithMore(*[getattr(p, name) for name, _ in E.Params._fields_])
    more.label = 17.0
    as_tuple = tuple(getattr(p, name) for name, _ in E.Params._fields_)
    for points in ([], _points([p]), _points([p, more, as_tuple, p])):
        assert bytes(E._scan_array(points)) == bytes(_by_field(points))


@pytest.mark.parametrize("bad", [{"gamma": 0.9}, None, 1.0, [0.9], ("x",)])
def test_other_params_are_refused(bad):
    for pack in (E._scan_array, _by_field):
        with pytest.raises((TypeError, RuntimeError)):
            pack(_points([bad]))
