"""GATHER in the plain and fused kernels reads the quad layout: the same
samples, so the same records as QUAD, bit for bit; an ordered persistent
GATHER plan's four-lane share takes that route too."""
import numpy as np
import pytest
import torch

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def small():
    rtbuild.build()
    w = wl.config2(elev_step=6.0, az_step=60.0)
    return w, {i: rt.Grid(w.grid, w.ne, interp=i) for i in ("gd", "cr")}


@pytest.mark.parametrize("interp", ["gd", "cr"])
@pytest.mark.parametrize("lanes", [0, 1, 2, 4])
def test_plain_gather_equals_quad(small, interp, lanes):
    w, grids = small
    fan = rt.Fan(w.fan, rt.RT_MIXED)
    a, b = (rt.rt_trace(grids[interp], fan, cfg=rt.launch_config(kernel=rt.RT_KERNEL_PLAIN, stencil=s, lanes_per_ray=lanes))
            for s in (rt.RT_STENCIL_GATHER, rt.RT_STENCIL_QUAD))
    assert a.tobytes() == b.tobytes()


def _device(n):
    return torch.zeros(n * 64, dtype=torch.uint8, device="cuda")


def test_fused_gather_equals_quad(small):
    w, grids = small
    fans = [rt.Fan(w.fan.replace(el_deg=w.fan.el_deg[k::3]), rt.RT_MIXED) for k in range(3)]
    n = sum(f.n_rays for f in fans)
    outs = [_device(n) for _ in range(2)]
    for o, s in zip(outs, (rt.RT_STENCIL_GATHER, rt.RT_STENCIL_QUAD)):
        rt.rt_trace_fans_device(grids["gd"], fans, o.data_ptr(), n, cfg=rt.launch_config(stencil=s))
    torch.cuda.synchronize()
    assert torch.equal(*outs)


def test_ordered_persistent_gather_plan(small):
    w, grids = small
    fan = rt.Fan(w.fan, rt.RT_MIXED)
    n = fan.n_rays
    plan = rt.Plan(grids["gd"], fan, rt.launch_config(kernel=rt.RT_KERNEL_PERSISTENT, stencil=rt.RT_STENCIL_GATHER,
                                                      lanes_per_ray=1))
    first, again = _device(n), _device(n)
    plan.execute(first.data_ptr(), n)
    for exclusive in (False, True):
        n_long = plan.order(first.data_ptr(), spread=0, long_factor=1.2, long_exclusive=exclusive)
        assert n_long > 0
        plan.execute(again.data_ptr(), n)
        torch.cuda.synchronize()
        a, b = (x.cpu().numpy().view(rt.RESULT_DTYPE) for x in (first, again))
        four = rt.rt_trace(grids["gd"], fan, cfg=rt.launch_config(kernel=rt.RT_KERNEL_PLAIN, stencil=rt.RT_STENCIL_QUAD,
                                                                  lanes_per_ray=4))
        same = np.array([x.tobytes() == y.tobytes() for x, y in zip(a, b)])
        share = np.array([x.tobytes() == y.tobytes() for x, y in zip(four, b)])
        assert np.all(same | share) and (~same).sum() <= n_long
