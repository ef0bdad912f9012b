"""The packed camera structs hold what ctypes would store field by field, and
what does not fit the packed form behaves as ctypes does.  Host code only."""
import ctypes as ct
import types

import numpy as np
import pytest

from paper_2110_06635_gb300 import _abi as A


def _cam(**kw):
    rng = np.random.default_rng(2)
    d = dict(w=1237, h=821, fx=901.5, fy=902.25, cx=600.1, cy=400.2, k1=-0.05, k2=0.01, k3=0.002, p1=1e-3, p2=-2e-3,
             model=1, R=rng.normal(size=(3, 3)), t=rng.normal(size=3), ev=0.7, wb=(0.9, 1.0, 1.2), vig_c=(0.4, 0.6),
             vig_a=(-0.1, 0.02, 0.003), epilogue=True)
    d.update(kw)
    return types.SimpleNamespace(**d)


def test_every_field():
    cam = _cam()
    s = A.camera_struct(cam)
    f = np.float32
    assert (s.K.w, s.K.h, s.K.model) == (1237, 821, 1)
    for n in ("fx", "fy", "cx", "cy", "k1", "k2", "k3", "p1", "p2"):
        assert getattr(s.K, n) == f(getattr(cam, n))
    assert np.array_equal(s.T.R[:], cam.R.astype(f).reshape(9)) and np.array_equal(s.T.t[:], cam.t.astype(f))
    assert s.ph.ev == f(0.7) and s.ph.enabled == 1 and s.ph.crf_n == 0 and not s.ph.crf_lut
    assert np.array_equal(s.ph.wb[:], f(cam.wb)) and np.array_equal(s.ph.vig_c[:], f(cam.vig_c))
    assert np.array_equal(s.ph.vig_a[:], f(cam.vig_a))
    bare = A.camera_struct(types.SimpleNamespace(w=4, h=3, fx=1, fy=1, cx=0, cy=0, k1=0, k2=0, R=np.eye(3), t=[0, 0, 1]))
    assert bare.K.model == 0 and bare.ph.enabled == 0 and list(bare.ph.wb) == [1, 1, 1] and bare.T.t[2] == 1


@pytest.mark.parametrize("kw", [dict(fx=1e39), dict(ev=-1e300), dict(w=(1 << 32) + 5)])
def test_out_of_range_as_ctypes(kw):
    s = A.camera_struct(_cam(**kw))
    (name, v), = kw.items()
    got = s.ph.ev if name == "ev" else getattr(s.K, name)
    assert got == (ct.c_int32(v).value if name == "w" else ct.c_float(v).value)


def test_wrong_lengths_are_refused():
    with pytest.raises((IndexError, RuntimeError)):
        A.camera_struct(_cam(wb=(1.0, 1.0), vig_c=(0.5, 0.5, 0.5)))
    with pytest.raises(ValueError):
        A.camera_struct(_cam(R=np.eye(4)))
