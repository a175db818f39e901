"""Mixed precision on a grid axis of more than 10^6 nodes, and on cells so fine
that one step crosses millions of them.

The cells beyond the 10^6th are read as such (right-hand sides within the
mixed path's 2e-4 of the FP64 path's, records within its 0.05 km).  On such an
axis a stage offset of 2^22 cells or more, which float cannot place in a cell,
is retried with a smaller step by the adaptive integrator and ends a fixed-step
ray as not finite instead of reading another cell.
"""
import dataclasses

import numpy as np
import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def _grid(n_alt, dalt, alt0, hm, h, fo):
    base = wl.config2().grid
    spec = dataclasses.replace(base, n_lat=4, n_lon=4, n_alt=n_alt, lat0_deg=wl.TX[0] - 30.0, lon0_deg=wl.TX[1] - 30.0,
                               alt0_km=alt0, dlat_deg=20.0, dlon_deg=20.0, dalt_km=dalt)
    z = (alt0 + dalt * np.arange(n_alt) - hm) / h
    col = (fo * 1e6) ** 2 / 80.6 * np.exp(0.5 * (1.0 - z - np.exp(-z)))
    return spec, np.array(np.broadcast_to(col.astype(np.float32), (4, 4, n_alt)))


@pytest.fixture(scope="module")
def long_grid():
    rtbuild.build()
    spec, ne = _grid(1_500_000, 4e-4, 60.0, 520.0, 60.0, 9.0)  # cell 10^6 lies at 460 km
    return rt.Grid(spec, ne)


def test_right_hand_side_beyond_a_million_cells(long_grid):
    rng = np.random.default_rng(3)
    n = 300
    k = rng.normal(size=(n, 3))
    k *= (rng.uniform(0.3, 1.0, n) / np.linalg.norm(k, axis=1))[:, None]
    lat, lon = wl.TX[0] + rng.uniform(-25, 25, n), wl.TX[1] + rng.uniform(-25, 25, n)
    ys = np.column_stack([wl.EARTH_RADIUS_KM + rng.uniform(300.0, 659.0, n), np.radians(90 - lat), np.radians(lon), k])
    for mode in (1, -1):
        ref, _ = rt.rt_eval_rhs(long_grid, 14.0, mode, ys, rt.RT_FP64)
        scale = np.abs(ref).max(axis=0)
        for st in (rt.RT_STENCIL_GATHER, rt.RT_STENCIL_QUAD):
            got, _ = rt.rt_eval_rhs(long_grid, 14.0, mode, ys, rt.RT_MIXED, st)
            assert np.max(np.abs(got - ref) / scale) < 2e-4


@pytest.mark.parametrize("lanes", [1, 2, 4])
def test_rays_beyond_a_million_cells(lanes):
    # a linear layer of whole multiples of 2^19 el/m^3, exact in float: at 0.4 m a cell the rounding of samples
    # would be nearly a percent of the gradient, another one in every cell
    spec, ne = _grid(1_500_000, 4e-4, 60.0, 520.0, 60.0, 9.0)
    ne[:] = np.arange(spec.n_alt, dtype=np.float32) * np.float32(2.0 ** 19)  # 8 MHz at the top, 660 km
    g = rt.Grid(spec, ne)
    fan = wl.config2().fan.replace(freq_mhz=[12.0], el_deg=[20.0, 28.0, 33.0, 36.0, 50.0, 65.0, 80.0], az_deg=[20.0, 200.0],
                                   integrator=wl.RK4, h_km=2.0, max_steps=3000)
    ref = rt.rt_trace(g, rt.Fan(fan, rt.RT_FP64))
    got = rt.rt_trace(g, rt.Fan(fan, rt.RT_MIXED), cfg=rt.launch_config(lanes_per_ray=lanes))
    landed = ref["status"] == rt.RT_RAY_LANDED
    assert landed.any() and not landed.all() and ref["apogee_km"][landed].max() > 470.0
    assert np.array_equal(got["status"], ref["status"])
    for f in ("group_path_km", "ground_range_km", "apogee_km"):
        assert np.abs(got[f] - ref[f]).max() <= 0.05, f


@pytest.mark.parametrize("n_alt", [64, 1_500_000])
def test_steps_across_millions_of_cells(n_alt):
    spec, ne = _grid(n_alt, 1e-6, 100.0, 100.0, 60.0, 1.0)  # 1 mm cells: 2^22 of them are 4.2 km
    g = rt.Grid(spec, ne)
    fan = wl.config2().fan.replace(freq_mhz=[20.0], el_deg=[30.0, 60.0, 85.0], az_deg=[75.0], h_km=15.0, h_max_km=15.0)
    for integrator in (wl.RKF45, wl.RK4):
        ref = rt.rt_trace(g, rt.Fan(fan.replace(integrator=integrator), rt.RT_FP64))
        got = rt.rt_trace(g, rt.Fan(fan.replace(integrator=integrator), rt.RT_MIXED))
        assert np.all(ref["status"] == rt.RT_RAY_ESCAPED)
        if n_alt > 1 << 20 and integrator == wl.RK4:  # no smaller step to go over to
            assert np.all(got["status"] == rt.RT_RAY_NONFINITE)
            continue
        assert np.array_equal(got["status"], ref["status"])
        assert np.abs(got["group_path_km"] - ref["group_path_km"]).max() <= 0.05
