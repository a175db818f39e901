"""The FP64 kernel's lane groups: a ray's record does not depend on how many
rays its warp holds (which decides the lanes per ray, and changes as rays
end), and agrees with the CPU oracle.

Sizes: one ray (32 lanes) to past the eight a warp starts with; both modes in
one warp, so that groups of one warp take different Appleton-Hartree branches.
Tolerances as for every FP64 fan: 1e-6 km, identical step and attempt counts.
"""
import dataclasses

import numpy as np
import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def lib():
    rtbuild.build()
    return rt.load()


@pytest.mark.parametrize("n_el", [1, 2, 3, 5, 9, 130, 700])
@pytest.mark.parametrize("interp,integrator,field", [("gd", wl.RKF45, True), ("cr", wl.RK4, True), ("gd", wl.RK4, False)])
def test_records_do_not_depend_on_the_warp(orc, n_el, interp, integrator, field):
    w = wl.config2()
    spec = w.grid if field else dataclasses.replace(w.grid, b0_tesla=0.0)
    g = rt.Grid(spec, w.ne, interp=interp)
    fan = w.fan.replace(freq_mhz=[9.0], el_deg=np.linspace(6.0, 75.0, n_el), az_deg=[40.0], integrator=integrator,
                        h_km=2.0, max_steps=2000)
    res = rt.rt_trace(g, rt.Fan(fan, rt.RT_FP64))
    # the canonical claim order puts neighbouring elevations, elevation-fastest (the default) as well; a
    # two-azimuth fan puts other rays beside each ray
    two = fan.replace(az_deg=[40.0, 200.0])
    other = rt.rt_trace(g, rt.Fan(two, rt.RT_FP64), cfg=rt.launch_config(order=rt.RT_ORDER_CANONICAL))
    assert np.array_equal(res, other.reshape(-1, 2)[:, 0])
    pick = sorted({0, n_el // 2, n_el - 1})
    for e in pick:
        for m, mode in enumerate((wl.MODE_O, wl.MODE_X)):
            one = rt.rt_trace(g, rt.Fan(fan.replace(el_deg=[fan.el_deg[e]], modes=mode), rt.RT_FP64))[0]
            assert one == res[m * n_el + e], (e, m)
    sub = fan.replace(el_deg=fan.el_deg[pick])
    ref = orc.trace_fan(orc.Grid(spec, w.ne, interp=interp), sub)
    got = res.reshape(2, n_el)[:, pick].reshape(-1)
    for f in ("status", "n_steps", "n_attempts"):
        assert np.array_equal(got[f], ref[f]), f
    for f in ("group_path_km", "ground_range_km", "apogee_km"):
        assert np.abs(got[f] - ref[f]).max() <= 1e-6, f
