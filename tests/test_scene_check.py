"""Scene creation refuses invalid primitives with the same error whether the
host checks them (few) or the device does (many; the host where there is none).
"""
import numpy as np
import pytest

from paper_1702_01530_gb300 import capi, scenegen as sg

MANY = 9000          # more than the host checks itself


def _create(ns, nt, change):
    rng = np.random.default_rng(ns + nt)
    s = sg.config_small(1)
    sp, tr = np.zeros(ns, sg.SPHERE_DT), np.zeros(nt, sg.TRIANGLE_DT)
    sp["center"], sp["radius"] = rng.uniform(-5, 5, (ns, 3)), 0.1
    for v in ("v0", "v1", "v2"):
        tr[v] = rng.uniform(-5, 5, (nt, 3))
    li = s.lights.copy()
    change(sp, tr, li, len(s.materials))
    with pytest.raises(capi.RtError) as e:
        capi.rt_scene_create(sp, tr, s.materials, li, stream=0)
    return e.value


def _sphere(i, field, value):
    def f(sp, tr, li, nm):
        sp[field][i] = nm if value is None else value
    return f


def _tri(i, field, value):
    def f(sp, tr, li, nm):
        tr[field][i] = nm if value is None else value
    return f


def _two(sp, tr, li, nm):
    li["intensity"] = 1e9
    tr["v1"][7] = np.nan
    sp["radius"][-1] = 0.0


@pytest.mark.parametrize("ns,nt,change,frag", [
    (MANY, 5, _sphere(0, "center", (0, np.inf, 0)), "sphere 0 invalid"),
    (MANY, 0, _sphere(MANY - 1, "radius", -0.0), f"sphere {MANY - 1} invalid"),
    (MANY, 0, _sphere(4, "radius", np.nan), "sphere 4 invalid"),
    (MANY, 3, _sphere(17, "material", None), "sphere 17 material out of range"),
    (0, MANY, _tri(0, "v0", (np.nan, 0, 0)), "triangle 0 has a non-finite vertex"),
    (3, MANY, _tri(MANY - 1, "v2", (0, 0, -np.inf)), f"triangle {MANY - 1} has a non-finite vertex"),
    (1, MANY, _tri(MANY - 1, "material", None), f"triangle {MANY - 1} material out of range"),
    (8, MANY, _two, "sphere 7 invalid"),
])
def test_invalid_primitives_are_refused(ns, nt, change, frag):
    e = _create(ns, nt, change)
    assert e.code == capi.RT_ERR_INVALID_ARG and frag in str(e)


@pytest.mark.gpu
@pytest.mark.parametrize("ns,nt,change,frag", [
    (MANY, 0, _sphere(MANY - 1, "center", (0, 0, np.nan)), f"sphere {MANY - 1} invalid"),
    (MANY, 0, _sphere(0, "radius", 0.0), "sphere 0 invalid"),
    (MANY, 1, _sphere(MANY - 1, "material", None), f"sphere {MANY - 1} material out of range"),
    (0, MANY, _tri(MANY - 1, "v2", (0, 0, np.inf)), f"triangle {MANY - 1} has a non-finite vertex"),
    (1, MANY, _tri(0, "material", None), "triangle 0 material out of range"),
])
def test_the_device_finds_them(ns, nt, change, frag):
    e = _create(ns, nt, change)
    assert e.code == capi.RT_ERR_INVALID_ARG and frag in str(e)


@pytest.mark.gpu
def test_extreme_values_are_accepted():
    s = sg.config_small(1)
    tr = np.zeros(MANY, sg.TRIANGLE_DT)
    for v in ("v0", "v1", "v2"):
        tr[v] = np.random.default_rng(1).uniform(-5, 5, (MANY, 3))
    tr["v1"][3] = np.finfo(np.float32).max
    sp = np.zeros(1, sg.SPHERE_DT)
    sp["radius"] = np.float32(1e-45)
    for t in ("material",):
        tr[t][-1] = len(s.materials) - 1
    capi.rt_scene_destroy(capi.rt_scene_create(sp, tr, s.materials, s.lights, stream=0))
