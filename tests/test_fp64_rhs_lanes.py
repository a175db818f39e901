"""rt_eval_rhs in FP64 evaluates what the tracer runs: a state's derivative by
1, 4, 8, 16 or 32 lanes, as many as a trace of that many rays starts with, is
the same bit for bit, and the oracle's to 1e-10 of its scale (the bound of the
one-thread evaluation: rounding of a few hundred FP64 operations)."""
import dataclasses

import numpy as np
import pytest

from paper_2506_18579_gb300 import build as rtbuild
from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SIZES = (1, 3, 601, 1403, 2603, 60001)  # on 152 SMs 1, 1, 2, 4, 8 and 32 states a warp, last blocks not full


@pytest.mark.parametrize("interp,field", [("gd", True), ("cr", True), ("gd", False)])
def test_derivatives_do_not_depend_on_the_lanes(orc, interp, field):
    rtbuild.build()
    w = wl.config2()
    spec = w.grid if field else dataclasses.replace(w.grid, b0_tesla=0.0)
    g, og = rt.Grid(spec, w.ne, interp=interp), orc.Grid(spec, w.ne, interp=interp)
    rng = np.random.default_rng(11)
    n = SIZES[-1]
    lat = rng.uniform(spec.lat0_deg - 0.5, spec.lat0_deg + (spec.n_lat - 1) * spec.dlat_deg + 0.5, n)
    lon = rng.uniform(spec.lon0_deg - 0.5, spec.lon0_deg + (spec.n_lon - 1) * spec.dlon_deg + 0.5, n)
    alt = rng.uniform(spec.alt0_km - 20, spec.alt0_km + (spec.n_alt - 1) * spec.dalt_km + 20, n)
    k = rng.normal(size=(n, 3))
    k *= (rng.uniform(0.3, 1.0, n) / np.linalg.norm(k, axis=1))[:, None]
    ys = np.column_stack([spec.earth_radius_km + alt, np.radians(90 - lat), np.radians(lon), k])
    for mode in (1, -1):
        whole, mu2 = rt.rt_eval_rhs(g, 10.0, mode, ys, rt.RT_FP64)
        for size in SIZES[:-1]:
            dy, m = rt.rt_eval_rhs(g, 10.0, mode, ys[n - size:], rt.RT_FP64)
            assert dy.tobytes() == whole[n - size:].tobytes() and m.tobytes() == mu2[n - size:].tobytes(), size
        ref = np.array([orc.rhs(og, 10.0, mode, y) for y in ys[-600:]])
        assert np.max(np.abs(whole[-600:] - ref) / (np.abs(ref).max(axis=0) + 1e-300)) < 1e-10
