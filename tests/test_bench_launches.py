"""The launches that bench.py counts per step are the kernels that one trace
queues: the kernel nodes of a captured plan execution, in both precisions."""
import ctypes
import os
import sys

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
if ROOT not in sys.path:
    sys.path.insert(0, ROOT)

import bench  # noqa: E402
from paper_2506_18579_gb300 import build as rtbuild  # noqa: E402
from paper_2506_18579_gb300 import rtgd as rt  # noqa: E402
from paper_2506_18579_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_launches_per_step(precision):
    import torch
    rtbuild.build()
    w = wl.config2(elev_step=6.0, az_step=60.0)
    grid = rt.Grid(w.grid, w.ne)
    fan = rt.Fan(w.fan, rt.RT_MIXED if precision == "mixed" else rt.RT_FP64)
    plan = rt.Plan(grid, fan, rt.launch_config(kernel=rt.RT_KERNEL_PLAIN))
    out = torch.zeros(fan.n_rays * 64, dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    cu = ctypes.CDLL("libcuda.so.1")
    stream, graph, n = ctypes.c_void_p(side.cuda_stream), ctypes.c_void_p(), ctypes.c_size_t(0)
    assert cu.cuStreamBeginCapture_v2(stream, 1) == 0  # this thread's calls only
    plan.execute(out.data_ptr(), fan.n_rays, stream=side.cuda_stream)
    assert cu.cuStreamEndCapture(stream, ctypes.byref(graph)) == 0
    assert cu.cuGraphGetNodes(graph, None, ctypes.byref(n)) == 0
    nodes = (ctypes.c_void_p * n.value)()
    assert cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)) == 0
    kernels = 0
    for node in nodes:
        kind = ctypes.c_int(-1)
        assert cu.cuGraphNodeGetType(ctypes.c_void_p(node), ctypes.byref(kind)) == 0
        kernels += kind.value == 0
    assert cu.cuGraphDestroy(graph) == 0
    assert kernels == bench.LAUNCHES_PER_STEP
