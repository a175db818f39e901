"""The tracer's timed cases: ray fans through the public entry points.

A case is a dict of plain values: the grid, the fan, the precision and
integrator, the entry point and its launch options.  ``prepare`` makes the
ionosphere and the transmitter from a seed and holds what a program keeps
between calls (the resident grid, the fan descriptor, a plan, output
buffers); ``run`` is one call; its outputs are the whole records, one array
per field.  ``exact`` traces small fans in 64-bit numpy.

The ionospheres are the workloads' stand-ins (E + F2 Chapman layers, a
latitude gradient of foF2, a travelling disturbance), evaluated on the GPU.
"""
import math

import numpy as np
import torch

from paper_2506_18579_gb300 import rtgd as rt
from paper_2506_18579_gb300 import workloads as wl

FIELDS = ("group_path_km", "ground_range_km", "az_dev_deg", "apogee_km", "land_lat_deg", "land_lon_deg")
COUNTS = ("status", "n_steps", "n_attempts", "n_evals")

_BASE = dict(
    entry="device",                                  # host, device, plan, fans, ionogram, snapshot
    n_lat=91, n_lon=181, n_alt=151, dlat=1.0, dlon=1.0, dalt=4.0,
    field=True, interp="gd", samples="f32", table=False,
    precision="mixed", integrator="rkf45", rtol=1e-8, h_km=1.0,
    n_freq=3, f_lo=8.0, f_hi=16.0, n_el=115, el_lo=3.0, el_hi=60.0, n_az=36, az_lo=0.0, az_span=350.0, modes=3,
    tuned=False, stencil="auto", lanes=0, threads=0, kernel="auto", order="elevation",
    n_fans=1, rx_km=1500.0)


def _case(**kw):
    assert not set(kw) - set(_BASE) - {"name"}
    return {**_BASE, **kw}


def listed():
    return [
        # One ray of a point-to-point link, as a homing loop asks for them one
        # after the other: the smallest call, host records.
        _case(name="one_ray", entry="host", n_lat=61, n_lon=121, n_alt=101, dlat=1.5, dlon=1.5, dalt=6.0, n_freq=1,
              f_lo=11.0, f_hi=11.0, n_el=1, el_lo=17.0, el_hi=17.0, n_az=1, az_lo=71.0, az_span=0.0, modes=1),
        # The paper's elevation scan of one frequency (16 rays, no field,
        # fixed-step RK4 at 1 km), all in double, host records.
        _case(name="scan_rk4_fp64", entry="host", n_lat=21, n_lon=21, n_alt=61, dlat=2.0, dlon=2.0, dalt=10.0,
              field=False, samples="f64", precision="fp64", integrator="rk4", n_freq=1, f_lo=10.0, f_hi=10.0, n_el=16,
              el_lo=5.0, el_hi=50.0, n_az=1, az_lo=30.0, az_span=0.0, modes=1),
        # The same scan over several frequencies and both modes, mixed precision.
        _case(name="scan_rk4_mixed", n_lat=21, n_lon=21, n_alt=61, dlat=2.0, dlon=2.0, dalt=10.0, integrator="rk4",
              n_freq=5, f_lo=6.0, f_hi=14.0, n_el=37, el_lo=5.0, el_hi=77.0, n_az=1, az_lo=30.0, az_span=0.0),
        # A coordinate-registration fan (one frequency, elevation x azimuth),
        # in double, adaptive: the precision a result is checked with.
        _case(name="sector_fp64", precision="fp64", n_freq=1, f_lo=12.0, f_hi=12.0, n_el=29, el_lo=3.0, el_hi=59.0,
              n_az=9, az_lo=20.0, az_span=64.0),
        # The paper's comparison interpolant (Catmull-Rom) at rtol 1e-9, in double.
        _case(name="catmull_rom_fp64", n_lat=31, n_lon=31, n_alt=121, dalt=5.0, interp="cr", samples="f64",
              precision="fp64", rtol=1e-9, n_freq=2, f_lo=8.0, f_hi=12.0, n_el=101, el_lo=5.0, el_hi=55.0, n_az=8,
              az_span=315.0),
        # The whole anisotropic fan (24,840 rays) in double.
        _case(name="fan_fp64", entry="device", precision="fp64"),
        # The same fan in mixed precision with the library's default launch,
        # host records: what a first call does.
        _case(name="fan_mixed_host", entry="host"),
        # The same fan as a plan in the launch configuration the autotuner
        # takes for it: a scan repeated on a resident grid.
        _case(name="fan_mixed_plan", entry="plan", table=True, tuned=True, stencil="table", lanes=4, threads=96,
              kernel="plain"),
        # The 495,122-ray ionogram-synthesis batch as a plan, likewise.
        _case(name="batch_plan", entry="plan", n_lat=181, n_lon=361, n_alt=301, dlat=0.5, dlon=0.5, dalt=2.0, table=True,
              tuned=True, stencil="table", lanes=1, threads=32, kernel="plain", n_freq=281, f_lo=2.0, f_hi=30.0,
              n_el=881, el_lo=1.0, el_hi=89.0, n_az=1, az_lo=45.0, az_span=0.0),
        # Many small requests fused into one launch, as the request server
        # makes it (an odd size of fan, one mode each).
        _case(name="small_fans", entry="fans", n_fans=48, n_freq=1, f_lo=13.0, f_hi=13.0, n_el=41, el_lo=4.0, el_hi=54.0,
              n_az=7, az_lo=-30.0, az_span=60.0, modes=1),
        # An oblique ionogram towards a receiver 1,500 km away.
        _case(name="ionogram", entry="ionogram", n_lat=61, n_lon=121, n_alt=101, dlat=1.5, dlon=1.5, dalt=6.0, n_freq=57,
              f_lo=2.0, f_hi=30.0, n_el=177, el_lo=1.0, el_hi=89.0, n_az=1, az_lo=45.0, az_span=0.0),
        # A new ionosphere snapshot on the host: grid preparation (per-cell
        # table included), one small fan, grid released.
        _case(name="snapshot", entry="snapshot", table=True, n_freq=1, f_lo=9.5, f_hi=9.5, n_el=23, el_lo=5.0, el_hi=49.0,
              n_az=5, az_lo=0.0, az_span=80.0, modes=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    entry = rng.choice(("host", "device", "device", "plan", "fans", "ionogram", "snapshot"))
    precision = "mixed" if entry in ("fans", "plan") else rng.choice(("mixed", "mixed", "fp64"))
    rk4 = entry != "ionogram" and rng.random() < 0.25
    n_lat, n_lon, n_alt = int(_log(rng, 15, 140)), int(_log(rng, 15, 260)), int(_log(rng, 41, 260))
    c = dict(entry=entry, precision=precision, integrator="rk4" if rk4 else "rkf45",
             n_lat=n_lat, n_lon=n_lon, n_alt=n_alt, dlat=round(rng.uniform(24.0, 80.0) / (n_lat - 1), 3),
             dlon=round(rng.uniform(24.0, 100.0) / (n_lon - 1), 3), dalt=round(rng.uniform(480.0, 640.0) / (n_alt - 1), 3),
             field=rng.random() < 0.8, interp="cr" if rng.random() < 0.2 else "gd",
             samples="f64" if rng.random() < 0.25 else "f32", table=entry != "fans" and rng.random() < 0.4,
             rtol=1e-8 if precision == "fp64" else 10.0 ** rng.uniform(-9.0, -6.5), h_km=round(rng.uniform(1.0, 3.0), 2),
             modes=rng.choice((1, 2, 3)))
    rays = _log(rng, 1, 3000 if precision == "fp64" else 60000) / (2 if c["modes"] == 3 else 1)
    if entry == "fans":
        c["n_fans"] = int(_log(rng, 2, 80))
        rays = min(rays, 20000) / c["n_fans"]
    c["n_freq"] = max(1, min(int(_log(rng, 1, 60)), int(rays)))
    c["n_az"] = 1 if entry == "ionogram" or rng.random() < 0.4 else max(1, min(int(_log(rng, 1, 36)), int(rays / c["n_freq"])))
    c["n_el"] = max(1, round(rays / (c["n_freq"] * c["n_az"])))
    if entry == "ionogram":  # a scan wide enough to meet the receiver
        c["n_el"], c["n_freq"] = max(c["n_el"], rng.randrange(60, 140)), min(max(c["n_freq"], 3), 40)
    c["f_lo"] = round(rng.uniform(3.0, 5.0 if entry == "ionogram" else 14.0), 2)
    c["f_hi"] = round(c["f_lo"] + (rng.uniform(1.0, 14.0) if c["n_freq"] > 1 else 0.0), 2)
    c["el_lo"] = round(rng.uniform(2.0, 25.0), 2)
    c["el_hi"] = round(c["el_lo"] + (rng.uniform(40.0 if entry == "ionogram" else 5.0, 60.0) if c["n_el"] > 1 else 0.0), 2)
    c["az_lo"] = round(rng.uniform(0.0, 360.0), 2)
    c["az_span"] = round(rng.uniform(10.0, 180.0), 2) if c["n_az"] > 1 else 0.0
    if entry == "ionogram":
        c["rx_km"] = round(rng.uniform(300.0, 900.0), 1)
    if precision == "mixed" and entry in ("host", "device", "plan") and rng.random() < 0.6:
        c.update(tuned=True, stencil=rng.choice(("gather", "quad") + (("table",) if c["table"] else ())),
                 lanes=rng.choice((0, 1, 2, 4)), threads=rng.choice((0, 32, 64, 96, 128)),
                 kernel=rng.choice(("plain", "plain", "plain", "persistent")), order=rng.choice(("canonical", "elevation")))
    return _case(**c)


# ------------------------------------------------------------------ inputs
def _n_rays(c):
    return c["n_freq"] * (2 if c["modes"] == 3 else 1) * c["n_el"] * c["n_az"] * c["n_fans"]


def _spec(c, seed):
    """Grid, analytic ionosphere and fans of a case, from the seed alone."""
    rng = np.random.default_rng([seed, 2506])
    lat_tx, lon_tx = wl.TX[0], wl.TX[1]
    g = wl.centred_grid(lat_tx, lon_tx, c["n_lat"], c["n_lon"], c["n_alt"], c["dlat"], c["dlon"], c["dalt"],
                        **(wl.dipole_field(lon_tx) if c["field"] else {}))
    iono = dict(foe=rng.uniform(2.8, 3.2), hme=rng.uniform(106.0, 114.0), fof2_lo=rng.uniform(5.7, 6.3),
                fof2_hi=rng.uniform(9.5, 10.5), hmf2=rng.uniform(285.0, 315.0), lat_c=lat_tx + rng.uniform(-5.0, 5.0),
                lon_c=lon_tx + rng.uniform(-5.0, 5.0), direction=rng.uniform(0.0, 2 * np.pi), phase=rng.uniform(0.0, 2 * np.pi))
    # (end points included; a full circle of azimuths is stated by its last one)
    axis = lambda lo, hi, n: np.linspace(lo, hi, n) if n > 1 else np.array([lo])  # noqa: E731
    fans = []
    for _ in range(c["n_fans"]):
        fans.append(wl.FanSpec(
            lat_tx + rng.uniform(-2.0, 2.0), lon_tx + rng.uniform(-2.0, 2.0), 0.0,
            freq_mhz=axis(c["f_lo"], c["f_hi"], c["n_freq"]), el_deg=axis(c["el_lo"], c["el_hi"], c["n_el"]),
            az_deg=np.mod(axis(c["az_lo"], c["az_lo"] + c["az_span"], c["n_az"]), 360.0), modes=c["modes"],
            integrator=wl.RK4 if c["integrator"] == "rk4" else wl.RKF45, h_km=c["h_km"], rtol=c["rtol"], atol_km=1e-6,
            h_min_km=1e-6, h_max_km=20.0, max_steps=20000 if c["integrator"] == "rk4" else 200000,
            precision=wl.FP64 if c["precision"] == "fp64" else wl.MIXED))
    return g, iono, fans


def _density(c, g, iono):
    """The grid's samples on the host (what an ionosphere model hands over)."""
    lat, lon, alt = (torch.as_tensor(x, device="cuda") for x in g.axes())

    def chapman(hm, h):
        z = (alt - hm) / h
        return torch.exp(0.5 * (1.0 - z - torch.exp(-z)))

    nm = lambda fo: (fo * 1e6) ** 2 / 80.6  # noqa: E731
    fof2 = iono["fof2_lo"] + (iono["fof2_hi"] - iono["fof2_lo"]) * (lat - lat[0]) / (lat[-1] - lat[0])
    p, q = torch.deg2rad(lat)[:, None], torch.deg2rad(lon)[None, :]
    p0, q0 = math.radians(iono["lat_c"]), math.radians(iono["lon_c"])
    cosr = torch.clamp(math.sin(p0) * torch.sin(p) + math.cos(p0) * torch.cos(p) * torch.cos(q - q0), -1.0, 1.0)
    rho = wl.EARTH_RADIUS_KM * torch.arccos(cosr)
    s = wl.EARTH_RADIUS_KM * ((p - p0) * math.cos(iono["direction"]) + (q - q0) * math.cos(p0) * math.sin(iono["direction"]))
    tid = 1.0 + 0.05 * torch.exp(-rho ** 2 / (2 * 600.0 ** 2)) * torch.cos(2 * math.pi * s / 200.0 + iono["phase"])
    ne = (nm(iono["foe"]) * chapman(iono["hme"], 10.0) + nm(fof2)[:, None] * chapman(iono["hmf2"], 50.0))[:, None, :] * tid[:, :, None]
    return ne.to(torch.float64 if c["samples"] == "f64" else torch.float32).cpu().numpy()


def _config(c):
    if not c["tuned"]:
        return None
    return rt.launch_config(kernel={"auto": 0, "plain": 1, "persistent": 2}[c["kernel"]],
                            stencil={"auto": 0, "gather": 1, "quad": 2, "table": 3}[c["stencil"]], block_threads=c["threads"],
                            order={"canonical": 0, "elevation": 1}[c["order"]], lanes_per_ray=c["lanes"])


def _receiver(c, f):
    """The point rx_km away on azimuth az_lo (spherical Earth)."""
    a, d = math.radians(c["az_lo"]), c["rx_km"] / wl.EARTH_RADIUS_KM
    p = math.radians(f.tx_lat_deg)
    p2 = math.asin(math.sin(p) * math.cos(d) + math.cos(p) * math.sin(d) * math.cos(a))
    dl = math.atan2(math.sin(a) * math.sin(d) * math.cos(p), math.cos(d) - math.sin(p) * math.sin(p2))
    return math.degrees(p2), f.tx_lon_deg + math.degrees(dl)


class _State:
    pass


def prepare(case, seed):
    s = _State()
    s.case, s.cfg = case, _config(case)
    s.spec, iono, specs = _spec(case, seed)
    ne = _density(case, s.spec, iono)
    s.fans = [rt.Fan(f) for f in specs]
    s.n = _n_rays(case)
    if case["entry"] == "snapshot":
        s.ne = ne
    else:
        s.grid = rt.Grid(s.spec, ne, table=case["table"], interp=case["interp"])
    if case["entry"] in ("host", "snapshot"):
        s.out = np.zeros(s.n, dtype=rt.RESULT_DTYPE)
    elif case["entry"] == "ionogram":
        s.rx = _receiver(case, specs[0])
    else:
        s.out = torch.zeros((s.n, 8), dtype=torch.float64, device="cuda")
    if case["entry"] == "plan":
        s.plan = rt.Plan(s.grid, s.fans[0], s.cfg)
    return s


def _fields(out):
    if isinstance(out, np.ndarray):
        return {k: out[k] for k in FIELDS + COUNTS}
    whole = out.view(torch.int32)  # the last 16 bytes of a record hold its four counts
    return {**{k: out[:, i] for i, k in enumerate(FIELDS)}, **{k: whole[:, 12 + i] for i, k in enumerate(COUNTS)}}


def run(s):
    entry, fan = s.case["entry"], s.fans[0]
    stream = torch.cuda.current_stream().cuda_stream
    if entry == "host":
        return _fields(rt.rt_trace(s.grid, fan, out=s.out, cfg=s.cfg, stream=stream))
    if entry == "snapshot":
        grid = rt.Grid(s.spec, s.ne, table=s.case["table"], interp=s.case["interp"])
        rt.rt_trace(grid, fan, out=s.out, cfg=s.cfg, stream=stream)
        grid.close()
        return _fields(s.out)
    if entry == "ionogram":
        f = fan.spec
        pts, _ = rt.rt_ionogram(s.grid, (f.tx_lat_deg, f.tx_lon_deg, f.tx_alt_km), s.rx, fan.freq, fan.el, modes=f.modes,
                                integrator=f.integrator, precision=f.precision, h_km=f.h_km, rtol=f.rtol, atol_km=f.atol_km,
                                h_min_km=f.h_min_km, h_max_km=f.h_max_km, max_steps=f.max_steps, cfg=s.cfg, stream=stream)
        whole = pts.base  # the buffer behind the points found, zeros after them
        return {"n_points": len(pts), **{k: whole[k] for k in whole.dtype.names}}
    if entry == "plan":
        s.plan.execute(s.out.data_ptr(), s.n, stream)
    elif entry == "fans":
        rt.rt_trace_fans_device(s.grid, s.fans, s.out.data_ptr(), s.n, cfg=s.cfg, stream=stream)
    else:
        rt.rt_trace_device(s.grid, fan, s.out.data_ptr(), s.n, cfg=s.cfg, stream=stream)
    return _fields(s.out)


# Right-hand-side evaluations of a ray: about 2,000 adaptive ones at rtol 1e-8
# (a fourth-order method: rtol^-1/5), or the steps of a 1,500 km path.
def _evals(c):
    return 4 * 1500.0 / c["h_km"] if c["integrator"] == "rk4" else 2000.0 * (1e-8 / c["rtol"]) ** 0.2


def work(case):
    n, wide = _n_rays(case), 8 if case["samples"] == "f64" else 4
    nodes = case["n_lat"] * case["n_lon"] * case["n_alt"]
    # the samples around a ray's path (some 300 cells of 64), at most the grid; a snapshot reads all of it
    touched = nodes if case["entry"] == "snapshot" else min(nodes, n * 300 * 64)
    # operations of an evaluation: 64-point contraction with gradients, weights, dipole, Appleton-Hartree, ray equations
    return {"bytes": touched * wide + 64.0 * n, "flops": n * _evals(case) * 900.0}


# ------------------------------------------------------- 64-bit statement
# Fixed-step RK4 or Fehlberg 4(5) with quantised, face-aligned steps and the
# last step solved for the ground or the grid's top, over arrays of rays.
_RKF = [[1 / 4], [3 / 32, 9 / 32], [1932 / 2197, -7200 / 2197, 7296 / 2197], [439 / 216, -8.0, 3680 / 513, -845 / 4104],
        [-8 / 27, 2.0, -3544 / 2565, 1859 / 4104, -11 / 40]]
_B4 = [25 / 216, 0.0, 1408 / 2565, 2197 / 4104, -1 / 5, 0.0]
_B5 = [16 / 135, 0.0, 6656 / 12825, 28561 / 56430, -9 / 50, 2 / 55]
_RK4 = [[1 / 2], [0.0, 1 / 2], [0.0, 0.0, 1.0]]


class _Exact:
    def __init__(self, g, ne, interp):
        self.g, self.interp = g, interp
        p = np.asarray(ne, dtype=np.float64)
        for ax in range(3):  # one ghost layer per face, quadratic extrapolation
            t = lambda i: np.take(p, [i], axis=ax)  # noqa: B023, E731
            p = np.concatenate([3 * t(0) - 3 * t(1) + t(2), p, 3 * t(-1) - 3 * t(-2) + t(-3)], axis=ax)
        self.p = p
        self.top = g.alt0_km + (g.n_alt - 1) * g.dalt_km
        la, lo = math.radians(g.pole_lat_deg), math.radians(g.pole_lon_deg)
        self.m = (math.cos(la) * math.cos(lo), math.cos(la) * math.sin(lo), math.sin(la))

    def coords(self, y):
        g = self.g
        lon = np.degrees(y[2]) - g.lon0_deg
        lon -= 360.0 * np.floor(lon / 360.0)
        return np.stack([(90.0 - np.degrees(y[1]) - g.lat0_deg) / g.dlat_deg, lon / g.dlon_deg,
                         (y[0] - g.earth_radius_km - g.alt0_km) / g.dalt_km])

    def weights(self, t):
        def half(s):
            if self.interp == "cr":
                return (s * (-0.5 + s * (1 - s * 0.5)), 1 + s * s * (-2.5 + s * 1.5), -0.5 + s * (2 - s * 1.5), s * (-5 + s * 4.5))
            return (s * (-0.5 + s * (11 / 12 + s * (-1 / 6 + s * (-5 / 12 + s / 6)))),
                    1 + s * s * (-2.25 + s * (0.5 + s * (1.25 - s * 0.5))),
                    -0.5 + s * (11 / 6 + s * (-0.5 + s * (-5 / 3 + s * 5 / 6))), s * (-4.5 + s * (1.5 + s * (5 - s * 2.5))))
        a, b, da, db = half(t)
        d, c, dd, dc = half(1 - t)
        return np.stack([a, b, c, d]), np.stack([da, db, -dc, -dd])

    def rhs(self, y, f_hz, sign):
        g = self.g
        n = np.array([g.n_lat, g.n_lon, g.n_alt])[:, None]
        x = self.coords(y)
        inside = np.all((x >= 0) & (x <= n - 1), axis=0)
        x = np.where(inside, x, 0.0)
        i = np.minimum(np.floor(x).astype(np.int64), n - 2)
        (wa, da), (wb, db), (wc, dc) = (self.weights(t) for t in x - i)
        o = np.arange(4)
        u = self.p[(i[0] + o[:, None])[:, None, None], (i[1] + o[:, None])[None, :, None], (i[2] + o[:, None])[None, None, :]]
        v, dv = (u * wc).sum(2), (u * dc).sum(2)
        s, sb, sc = (v * wb).sum(1), (v * db).sum(1), (dv * wb).sum(1)
        k = 80.6 / f_hz ** 2 * inside
        X, dX = k * (s * wa).sum(0), (k * (sc * wa).sum(0) / g.dalt_km, -k * np.degrees((s * da).sum(0)) / g.dlat_deg,
                                      k * np.degrees((sb * wa).sum(0)) / g.dlon_deg)
        r, st, ct, sp, cp, kr, kt, kp = y[0], np.sin(y[1]), np.cos(y[1]), np.sin(y[2]), np.cos(y[2]), y[3], y[4], y[5]
        kk = kr * kr + kt * kt + kp * kp
        if g.b0_tesla == 0.0:
            mu2, H, K, G = 1 - X, [0.5 * d for d in dX], (kr, kt, kp), -kk - X
        else:
            mx, my, mz = self.m
            mr, mt, mp = mx * st * cp + my * st * sp + mz * ct, mx * ct * cp + my * ct * sp - mz * st, -mx * sp + my * cp
            A = 2.7992489872e10 / f_hz * g.b0_tesla * (g.earth_radius_km / r) ** 3
            Y = (-2 * A * mr, A * mt, A * mp)
            YY, kY = A * A * (1 + 3 * mr * mr), kr * Y[0] + kt * Y[1] + kp * Y[2]
            gYY = (-6 * YY / r, 6 * A * A * mr * mt, 6 * A * A * mr * st * mp)
            gkY = (-3 * kY / r, A * (-2 * kr * mt - kt * mr),
                   A * (-2 * kr * st * mp + kt * ct * mp - kp * (st * mr + ct * mt)))
            L = kY * kY / kk
            T = np.maximum(YY - L, 0.0)
            a = 1 - X
            S = np.sqrt(T * T + 4 * L * a * a)
            # ordinary: mu^2 = 1 - X / (1 + q), q = 2 L a / (S + T); extraordinary: 1 - 2 X a / D, D = 2 a - T - S
            with np.errstate(all="ignore"):
                W, D = S + T, 2 * a - T - S
                q = 2 * L * a / W
                qX, qL, qT = 2 * L * (4 * L * a * a / S - W) / W ** 2, 2 * a / W - 4 * L * a ** 3 / (S * W * W), -q / S
                o2, N = (1 + q) ** 2, 2 * X * a
                up = sign > 0
                mu2 = np.where(up, 1 - X / (1 + q), 1 - N / D)
                FX = np.where(up, (X * qX - (1 + q)) / o2, (N * (-2 + 4 * L * a / S) - (2 - 4 * X) * D) / D ** 2)
                FL = np.where(up, X * qL / o2, -N * 2 * a * a / S / D ** 2)
                FT = np.where(up, X * qT / o2, N * (-1 - T / S) / D ** 2)
            c = (FL - FT) * 2 * kY / kk
            H = [-0.5 * (FX * dX[j] + FT * gYY[j] + c * gkY[j]) for j in range(3)]
            K = [kj - 0.5 * c * (Yj - kY / kk * kj) for kj, Yj in zip((kr, kt, kp), Y)]
            G = -kk + X * FX + L * FL + T * FT
        dr, dt, dp = -K[0] / G, -K[1] / (G * r), -K[2] / (G * r * st)
        return np.stack([dr, dt, dp, H[0] / G + kt * dt + kp * st * dp, (H[1] / G - kt * dr + kp * r * ct * dp) / r,
                         (H[2] / G - kp * st * dr - kp * r * ct * dt) / (r * st)]), mu2

    def step(self, y, k1, h, f, sign, adaptive):
        ks = [k1]
        for row in _RKF if adaptive else _RK4:
            ks.append(self.rhs(y + h * sum(a * k for a, k in zip(row, ks) if a), f, sign)[0])
        if not adaptive:
            return y + h / 6 * (ks[0] + 2 * ks[1] + 2 * ks[2] + ks[3]), None
        return (y + h * sum(b * k for b, k in zip(_B4, ks) if b), h * sum((b5 - b4) * k for b5, b4, k in zip(_B5, _B4, ks)))

    def face(self, y, k1):
        g, x = self.g, self.coords(y)
        v = np.stack([-np.degrees(k1[1]) / g.dlat_deg, np.degrees(k1[2]) / g.dlon_deg, k1[0] / g.dalt_km])
        last = np.array([g.n_lat, g.n_lon, g.n_alt])[:, None] - 1.0
        F = np.where(v > 0, np.maximum(np.floor(x) + 1, 0), np.minimum(np.ceil(x) - 1, last))
        ok = (v != 0) & (F >= 0) & (F <= last)
        ok[:2] &= (x[2] >= 0) & (x[2] <= last[2])
        with np.errstate(all="ignore"):
            return np.where(ok, (F - x) / v, np.inf).min(0)

    def trace(self, fan):
        g, RE, adaptive = self.g, self.g.earth_radius_km, fan.integrator == wl.RKF45
        n = fan.n_rays
        f, sign, el, az = (np.array(v) for v in zip(*(fan.ray_params(i) for i in range(n))))
        f, el, az = f * 1e6, np.radians(el), np.radians(az)
        th0, ph0 = math.radians(90.0 - fan.tx_lat_deg), math.radians(fan.tx_lon_deg)
        y = np.stack([np.full(n, RE + fan.tx_alt_km), np.full(n, th0), np.full(n, ph0),
                      np.sin(el), -np.cos(el) * np.cos(az), np.cos(el) * np.sin(az)])
        y[3:] *= np.sqrt(self.rhs(y, f, sign)[1])
        P, apo, status, steps, tries, evals = (np.zeros(n), y[0] - RE, *(np.zeros(n, np.int64) for _ in range(3)), np.ones(n, np.int64))
        h, k1, known = np.full(n, fan.h_km), np.zeros((6, n)), np.zeros(n, bool)
        prev, solving, side = np.full((3, n), np.nan), np.zeros(n, np.int64), np.zeros(n, np.int64)  # solving: 1 ground, 2 top
        br = np.zeros((4, n))  # bracket a, fa, b, fb of the last step's solve
        rounds = np.zeros(n, np.int64)
        live = np.arange(n)
        while live.size:
            over = tries[live] >= fan.max_steps
            status[live[over & (solving[live] == 0)]] = 4
            live = live[~(over & (solving[live] == 0))]
            need = live[~known[live]]
            if need.size:
                k1[:, need] = self.rhs(y[:, need], f[need], sign[need])[0]
                known[need], evals[need] = True, evals[need] + 1
                turn = need[(prev[1, need] > 0) & (k1[0, need] <= 0)]
                for i in turn:  # the turning point of the cubic through both ends
                    m0, m1, d = prev[2, i] * prev[1, i], prev[2, i] * k1[0, i], y[0, i] - prev[0, i]
                    A, B = m0 + m1 - 2 * d, 3 * d - 2 * m0 - m1
                    lo, hi = 0.0, 1.0
                    for _ in range(60):
                        mid = 0.5 * (lo + hi)
                        lo, hi = (mid, hi) if m0 + 2 * B * mid + 3 * A * mid * mid > 0 else (lo, mid)
                    s = 0.5 * (lo + hi)
                    apo[i] = max(apo[i], prev[0, i] + s * (m0 + s * (B + s * A)) - RE)
                prev[1, need] = np.nan
            if not live.size:
                break
            hs, at_face = h[live].copy(), np.zeros(live.size, bool)
            if adaptive:
                hf = self.face(y[:, live], k1[:, live])
                at_face = (hf > 1e-3 * hs) & (hf < hs)
                hs = np.where(at_face, hf * (1 + 1e-4), hs)
            sol = solving[live] > 0
            a, fa, b, fb = br[:, live]
            with np.errstate(all="ignore"):
                hs = np.where(sol, b - fb * (b - a) / (fb - fa), hs)
            yn, e = self.step(y[:, live], k1[:, live], hs, f[live], sign[live], adaptive)
            tries[live] += 1
            evals[live] += 5 if adaptive else 3
            keep = np.ones(live.size, bool)
            for j in np.flatnonzero(sol):
                i = live[j]
                sg, target = (1.0, RE) if solving[i] == 1 else (-1.0, RE + self.top)
                fc = sg * (yn[0, j] - target)
                rounds[i] += 1
                if abs(fc) < 1e-9 or rounds[i] >= 60:
                    P[i], y[:, i], status[i], keep[j] = P[i] + hs[j], yn[:, j], solving[i], False
                    steps[i] += 1
                    if solving[i] == 2:
                        apo[i] = max(apo[i], y[0, i] - RE)
                elif fc < 0:
                    br[2:, i] = hs[j], fc
                    br[1, i] *= 0.5 if side[i] == -1 else 1.0
                    side[i] = -1
                else:
                    br[:2, i] = hs[j], fc
                    br[3, i] *= 0.5 if side[i] == 1 else 1.0
                    side[i] = 1
            good, nxt = ~sol, h[live].copy()
            if adaptive:
                yl = y[:, live]
                pos = np.maximum(np.abs(e[0]), np.maximum(yl[0] * np.abs(e[1]), yl[0] * np.sin(yl[1]) * np.abs(e[2])))
                kmag = np.maximum(np.sqrt((yl[3:] ** 2).sum(0)), 1e-3)
                err = np.maximum(pos / (fan.atol_km + fan.rtol * yl[0]), np.abs(e[3:]).max(0) / (fan.rtol * kmag))
                with np.errstate(all="ignore"):
                    fac = np.where(err == 0, 5.0, np.minimum(5.0, np.maximum(0.2, 0.9 * err ** -0.2)))
                fac = np.exp2(np.floor(4 * np.log2(fac)) * 0.25)
                bad = ~sol & ~(err <= 1)
                h[live[bad]] *= fac[bad]
                low = bad & (h[live] < fan.h_min_km)
                status[live[low]], keep[low] = 5, False
                good &= ~bad
                nxt = np.clip(nxt * np.where(at_face, np.minimum(fac, 1.0), fac), fan.h_min_km, fan.h_max_km)
            odd = good & ~np.isfinite(yn).all(0)
            status[live[odd]], keep[odd], good = 6, False, good & ~odd
            lands = good & (yn[0] < RE)
            exits = good & ~lands & (yn[0] - RE > self.top)
            for j in np.flatnonzero(lands | exits):
                i = live[j]
                sg, target = (1.0, RE) if lands[j] else (-1.0, RE + self.top)
                solving[i], side[i], rounds[i] = 1 if lands[j] else 2, 0, 0
                br[:, i] = 0.0, sg * (y[0, i] - target), hs[j], sg * (yn[0, j] - target)
            go = good & ~lands & ~exits
            at = live[go]
            prev[:, at] = y[0, at], k1[0, at], hs[go]
            P[at] += hs[go]
            steps[at] += 1
            y[:, at], known[at], h[at] = yn[:, go], False, nxt[go]
            apo[at] = np.maximum(apo[at], y[0, at] - RE)
            x = self.coords(y[:, at])
            out = (y[0, at] - RE >= g.alt0_km) & ((x[0] < 0) | (x[0] > g.n_lat - 1) | (x[1] < 0) | (x[1] > g.n_lon - 1))
            status[at[out]] = 3
            keep[np.flatnonzero(go)[out]] = False
            live = live[keep]
        th, dl = y[1], y[2] - ph0
        east, north = np.sin(th) * np.sin(dl), np.sin(th0) * np.cos(th) - np.cos(th0) * np.sin(th) * np.cos(dl)
        ang = np.arctan2(np.hypot(east, north), np.sin(th0) * np.sin(th) * np.cos(dl) + np.cos(th0) * np.cos(th))
        wrap = lambda v: v - 360.0 * np.floor((v + 180.0) / 360.0)  # noqa: E731
        return dict(group_path_km=P, ground_range_km=RE * ang, az_dev_deg=wrap(np.degrees(np.arctan2(east, north) - az)),
                    apogee_km=apo, land_lat_deg=90.0 - np.degrees(th), land_lon_deg=wrap(np.degrees(y[2])))


def exact(case, seed):
    if case["entry"] in ("ionogram", "fans") or _n_rays(case) > 600:
        return None
    g, iono, fans = _spec(case, seed)
    got = _Exact(g, _density(case, g, iono), case["interp"]).trace(fans[0])
    return {**got, **{k: None for k in COUNTS}}
