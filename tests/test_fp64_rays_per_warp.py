"""Rays that a warp of the FP64 kernel starts with: on 152 SMs the fastest of the
measured starts at the sizes where one is faster than its neighbours (the
table at fp64_rays_per_warp)."""
import ctypes

import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt


@pytest.mark.parametrize("n,rays", [(1, 1), (184, 1), (460, 1), (522, 2), (640, 2), (1000, 2), (2000, 4), (4968, 8),
                                    (24840, 8), (51098, 8), (61830, 32), (98928, 32), (495122, 32)])
def test_measured_best(n, rays):
    rtbuild.build()
    rt.load()
    f = ctypes.CDLL(rtbuild.LIB)["_ZN4rtgd18fp64_rays_per_warpExi"]  # rtgd::fp64_rays_per_warp(long long, int)
    f.restype, f.argtypes = ctypes.c_int, [ctypes.c_longlong, ctypes.c_int]
    assert f(n, 152) == rays
