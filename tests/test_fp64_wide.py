"""FP64 fans that fill the GPU many times over start with 32 rays a warp, one
per lane: the dispatch line, and the records, which are those of the smaller
fans' lane groups bit for bit.

Sizes: just past the line, with an odd number of elevations (the boundary
between the modes falls inside a warp) and a partly filled last block; every
status a ray can end with is met while a lane holds a ray of its own.
"""
import ctypes
import dataclasses

import numpy as np
import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl


def _rays_per_warp(n, sms):
    rtbuild.build()
    rt.load()
    f = ctypes.CDLL(rtbuild.LIB)["_ZN4rtgd18fp64_rays_per_warpExi"]  # rtgd::fp64_rays_per_warp(long long, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_longlong, ctypes.c_int]
    return f(n, sms)


@pytest.mark.parametrize("n,wide", [(24840, False), (51098, False), (58367, False), (58368, True), (61830, True),
                                    (98928, True), (495122, True)])
def test_dispatch_line(n, wide):
    """On 152 SMs the faster of both measured starts, see fp64_rays_per_warp."""
    assert (_rays_per_warp(n, 152) == 32) == wide


_VARIANTS = {
    "field": dict(),
    "no field, path limit": dict(field=False, max_group_path_km=1800.0),
    "rk4, step limit": dict(integrator=wl.RK4, h_km=3.0, max_steps=500),
    "catmull-rom, from inside the layer": dict(interp="cr", tx_alt_km=180.0),
}


@pytest.mark.gpu
@pytest.mark.parametrize("variant", list(_VARIANTS))
def test_records_equal_the_lane_groups(variant):
    import torch
    kw = dict(_VARIANTS[variant])
    field, interp = kw.pop("field", True), kw.pop("interp", "gd")
    w = wl.config2()
    spec = w.grid if field else dataclasses.replace(w.grid, b0_tesla=0.0)
    g = rt.Grid(spec, w.ne, interp=interp)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_el = 229
    n_az = 2 * 32 * 6 * sms // (4 * n_el) + 2
    fan = w.fan.replace(freq_mhz=[9.0, 21.0], el_deg=np.linspace(4.0, 80.0, n_el), rtol=1e-7,
                        az_deg=np.linspace(0.0, 355.0, n_az), **kw)
    assert _rays_per_warp(fan.n_rays, sms) == 32 and fan.n_rays % 32
    res = rt.rt_trace(g, rt.Fan(fan, rt.RT_FP64)).reshape(-1, n_az)
    for part in np.array_split(np.arange(n_az), 3):
        sub = fan.replace(az_deg=fan.az_deg[part])
        assert _rays_per_warp(sub.n_rays, sms) == 8
        assert rt.rt_trace(g, rt.Fan(sub, rt.RT_FP64)).reshape(-1, len(part)).tobytes() == \
            np.ascontiguousarray(res[:, part]).tobytes()


@pytest.mark.gpu
def test_captured_plan_and_noalloc_call():
    """The same fan from a captured graph of a plan and through the entry point
    that allocates nothing: the records of the plain call."""
    import torch
    w = wl.config2()
    g = rt.Grid(w.grid, w.ne)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n_az = 2 * 32 * 6 * sms // (2 * 229) + 2
    fan = rt.Fan(w.fan.replace(freq_mhz=[24.0], el_deg=np.linspace(4.0, 80.0, 229), rtol=1e-7,
                               az_deg=np.linspace(0.0, 355.0, n_az)), rt.RT_FP64)
    n = fan.n_rays
    assert _rays_per_warp(n, sms) == 32
    out, side, graph = torch.zeros((2, n * 64), dtype=torch.uint8, device="cuda"), torch.cuda.Stream(), torch.cuda.CUDAGraph()
    plan = rt.Plan(g, fan)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        with torch.cuda.graph(graph, stream=side):
            plan.execute(out[0].data_ptr(), n, stream=side.cuda_stream)
    graph.replay()
    rt.rt_trace_device_noalloc(g, fan, out[1].data_ptr(), n, stream=torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    ref = rt.rt_trace(g, fan).tobytes()
    assert out[0].cpu().numpy().tobytes() == ref and out[1].cpu().numpy().tobytes() == ref
