"""FP64 rays beside others in a warp, at every number of rays a warp starts
with: rays next to the boundary between the modes (groups of one warp then take
different Appleton-Hartree branches), in the first and in a partly filled last
block (idle groups follow group 0's ray), against the same rays traced alone
with all 32 lanes, bit for bit.  The sizes are odd multiples so that the mode
boundary falls inside a warp and the last block is not full."""
import ctypes
import dataclasses

import numpy as np
import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _rays_per_warp(n):
    import torch
    f = ctypes.CDLL(rtbuild.LIB)["_ZN4rtgd18fp64_rays_per_warpExi"]  # rtgd::fp64_rays_per_warp(long long, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_longlong, ctypes.c_int]
    return f(n, torch.cuda.get_device_properties(0).multi_processor_count)


@pytest.mark.parametrize("rays,n_el,modes", [(2, 301, 3), (2, 601, 1), (4, 701, 3), (4, 1403, 2), (8, 1301, 3), (8, 2603, 1)])
@pytest.mark.parametrize("interp,integrator,field", [("gd", wl.RKF45, True), ("cr", wl.RK4, True), ("gd", wl.RK4, False)])
def test_records_equal_the_lone_rays(rays, n_el, modes, interp, integrator, field):
    rtbuild.build()
    w = wl.config2()
    spec = w.grid if field else dataclasses.replace(w.grid, b0_tesla=0.0)
    g = rt.Grid(spec, w.ne, interp=interp)
    fan = w.fan.replace(freq_mhz=[9.0], el_deg=np.linspace(6.0, 75.0, n_el), az_deg=[40.0], modes=modes,
                        integrator=integrator, h_km=4.0, max_steps=600)
    n = fan.n_rays
    assert _rays_per_warp(n) == rays and _rays_per_warp(1) == 1
    assert n % rays or modes == 3 and n_el % rays
    res = rt.rt_trace(g, rt.Fan(fan, rt.RT_FP64))
    last = n - (n % rays or rays)
    pick = {0, 1, rays - 1, n // 3, n_el - 2, n_el - 1, n_el, n_el + 1, last, n - 1}
    for i in sorted(p for p in pick if p < n):
        mode = modes if modes != 3 else (wl.MODE_O, wl.MODE_X)[i // n_el]
        one = rt.rt_trace(g, rt.Fan(fan.replace(el_deg=[fan.el_deg[i % n_el]], modes=mode), rt.RT_FP64))
        assert one.tobytes() == res[i:i + 1].tobytes(), i
