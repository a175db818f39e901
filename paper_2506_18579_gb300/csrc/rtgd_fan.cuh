// rtgd_fan.cuh -- device side of a fan: canonical ray index to launch
// parameters, claim order, launch direction (shared by the mixed and the
// FP64 kernels).
#pragma once

#include "rtgd_device.cuh"
#include "rtgd_internal.h"

namespace rtgd {

// Canonical ray index -> (frequency, mode, elevation, azimuth) of the fan,
// order [freq][mode][el][az], with the per-fan table entries of each.
struct RayParams {
    double f_hz;
    float xfac, ab0;        // the mixed path's per-frequency factors
    double se, ce, sa, ca;  // sin, cos of elevation and azimuth
    double az;              // azimuth (rad)
    int mode;
};

// Fans hold fewer than 2^31 rays (checked on the host), so 32-bit index
// arithmetic suffices (64-bit divisions are long instruction sequences).
__device__ __forceinline__ RayParams ray_params(const FanDev &f, long long id64) {
    const unsigned id = (unsigned)id64;
    const unsigned a = id % (unsigned)f.n_az;
    const unsigned rest = id / (unsigned)f.n_az;
    const unsigned e = rest % (unsigned)f.n_el;
    const unsigned rest2 = rest / (unsigned)f.n_el;
    const unsigned m = rest2 % (unsigned)f.n_modes;
    const unsigned q = rest2 / (unsigned)f.n_modes;
    RayParams p;
    p.f_hz = f.freq[q].f_hz;
    p.xfac = f.freq[q].xfac;
    p.ab0 = f.freq[q].ab0;
    p.se = f.el[e].s;
    p.ce = f.el[e].c;
    p.sa = f.az[a].s;
    p.ca = f.az[a].c;
    p.az = f.az[a].rad;
    p.mode = (m == 0) ? f.mode0 : f.mode1;
    return p;
}

// Claim index -> canonical index.  ORDER_ELEVATION_FASTEST hands out
// neighbouring elevations of one azimuth together (similar paths, so the
// lanes of a warp gather from nearby cells).
__device__ __forceinline__ long long claim_to_ray(const FanDev &f, long long c64) {
    if (f.perm) return f.perm[f.perm_off + c64];
    if (f.order != RT_ORDER_ELEVATION_FASTEST) return c64;
    const unsigned c = (unsigned)c64;
    const unsigned e = c % (unsigned)f.n_el;
    const unsigned rest = c / (unsigned)f.n_el;
    const unsigned a = rest % (unsigned)f.n_az;
    const unsigned fm = rest / (unsigned)f.n_az;  // freq * n_modes + mode
    return ((long long)fm * f.n_el + e) * f.n_az + a;
}

// Launch direction (elevation above the horizontal, azimuth clockwise from
// north; the theta unit vector points south) and position of a ray, from the
// fan's sine and cosine tables.
__device__ __forceinline__ void launch_dir(const FanDev &f, const RayParams &p, double y[6]) {
    y[0] = f.tx_r;
    y[1] = f.tx_th;
    y[2] = f.tx_ph;
    y[3] = p.se;
    y[4] = -p.ce * p.ca;
    y[5] = p.ce * p.sa;
}

}  // namespace rtgd
