"""Rays that a warp of the FP64 kernel starts with on 152 SMs: at either end of
each start's range, and at sizes that the table at fp64_rays_per_warp gives."""
import ctypes

import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt


@pytest.mark.parametrize("n,rays", [(1, 1), (522, 1), (555, 1), (556, 2), (1104, 2), (1105, 4), (2256, 4), (2257, 8),
                                    (24840, 8), (58367, 8), (58368, 32), (495122, 32), (2 ** 31 - 1, 32)])
def test_start(n, rays):
    rtbuild.build()
    rt.load()
    f = ctypes.CDLL(rtbuild.LIB)["_ZN4rtgd18fp64_rays_per_warpExi"]  # rtgd::fp64_rays_per_warp(long long, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_longlong, ctypes.c_int]
    assert f(n, 152) == rays
