// rtgd_kernels.cu -- CUDA kernels of the RTM-GD tracer (sm_103a).
//
//   grid preparation  : ghost padding (FP64 + FP32 copies), the "quad" layout
//                       (4 consecutive altitude samples per float4) and the
//                       optional per-cell 64-sample table (Sec. II-C: the
//                       interpolation data are prepared once per grid cell).
//                       (The all-FP64 tracer is in rtgd_fp64.cu.)
//   trace_mixed_*     : mixed-precision tracer.  A group of 1, 2 or 4 lanes
//                       carries one ray; every loop iteration runs one whole
//                       RK attempt for all lanes of a warp (the stage index
//                       is warp-uniform), so the lanes stay converged.  The
//                       plain kernel gives each group one ray; the persistent
//                       kernel keeps a resident grid whose warps claim their
//                       next rays from an atomic counter once their current
//                       rays have ended.
//   eval_rhs          : diagnostic evaluation of dy/dP' at given states.
#include <cuda_runtime.h>
#include <math.h>

#include <algorithm>
#include <cmath>
#include <stdint.h>

#include "rtgd.h"
#include "rtgd_device.cuh"
#include "rtgd_fan.cuh"
#include "rtgd_fp64.cuh"
#include "rtgd_internal.h"

namespace rtgd {

// ===================================================================== grid
// Padded value at padded index (pi, pj, pk): interior nodes are copied; a
// ghost index maps to quadratic extrapolation u_{-1} = 3u_0 - 3u_1 + u_2
// (and its mirror at the far face), applied along every ghost axis (tensor
// product, so corners combine up to 27 nodes).
__device__ __forceinline__ int ghost_taps(int p, int n, int idx[3], double w[3]) {
    if (p == 0) {
        idx[0] = 0; idx[1] = 1; idx[2] = 2;
        w[0] = 3.0; w[1] = -3.0; w[2] = 1.0;
        return 3;
    }
    if (p == n + 1) {
        idx[0] = n - 1; idx[1] = n - 2; idx[2] = n - 3;
        w[0] = 3.0; w[1] = -3.0; w[2] = 1.0;
        return 3;
    }
    idx[0] = p - 1;
    w[0] = 1.0;
    return 1;
}

template <typename T>
__global__ void pad_kernel(const T *__restrict__ raw, double *__restrict__ pad64, float *__restrict__ pad32,
                           int n_lat, int n_lon, int n_alt) {
    const long long P_lon = n_lon + 2, P_alt = n_alt + 2;
    const long long total = (long long)(n_lat + 2) * P_lon * P_alt;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int pk = (int)(e % P_alt);
        const int pj = (int)((e / P_alt) % P_lon);
        const int pi = (int)(e / (P_alt * P_lon));
        int ia[3], ja[3], ka[3];
        double wa[3], wb[3], wc[3];
        const int na = ghost_taps(pi, n_lat, ia, wa);
        const int nb = ghost_taps(pj, n_lon, ja, wb);
        const int nc = ghost_taps(pk, n_alt, ka, wc);
        double v = 0.0;
        for (int a = 0; a < na; ++a)
            for (int b = 0; b < nb; ++b)
                for (int c = 0; c < nc; ++c)
                    v += wa[a] * wb[b] * wc[c] *
                         (double)raw[((long long)ia[a] * n_lon + ja[b]) * n_alt + ka[c]];
        pad64[e] = v;
        pad32[e] = (float)v;
    }
}

// quad[(pi, pj, k)] = padded samples k..k+3 (nodes k-1..k+2) of cell k.
__global__ void quad_kernel(const float *__restrict__ pad32, float4 *__restrict__ quad, int n_lat, int n_lon,
                            int n_alt) {
    const long long P_lon = n_lon + 2, P_alt = n_alt + 2, Q = n_alt - 1;
    const long long total = (long long)(n_lat + 2) * P_lon * Q;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const long long k = e % Q;
        const long long row = e / Q;  // pi * P_lon + pj
        const float *p = pad32 + row * P_alt + k;
        quad[e] = make_float4(p[0], p[1], p[2], p[3]);
    }
}

// table[cell * 16 + a * 4 + b] = the 4 altitude samples of row (a, b) of the
// 4x4x4 stencil of cell (i, j, k), each minus the cell's reference node
// (i, j, k) (padded (i+1, j+1, k+1)); cells are ordered [i][j][k].  The stage
// evaluation contracts samples relative to that node, so storing them that
// way saves the subtraction (the same float operation, done once per grid).
__global__ void table_kernel(const float4 *__restrict__ quad, float4 *__restrict__ table, int n_lat, int n_lon,
                             int n_alt) {
    const long long C_lon = n_lon - 1, C_alt = n_alt - 1, P_lon = n_lon + 2;
    const long long total = (long long)(n_lat - 1) * C_lon * C_alt * 16;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int ab = (int)(e & 15);
        const long long cell = e >> 4;
        const long long k = cell % C_alt;
        const long long j = (cell / C_alt) % C_lon;
        const long long i = cell / (C_alt * C_lon);
        const int a = ab >> 2, b = ab & 3;
        const float4 u = quad[((i + a) * P_lon + (j + b)) * C_alt + k];
        const float ref = quad[((i + 1) * P_lon + (j + 1)) * C_alt + k].y;
        table[e] = make_float4(u.x - ref, u.y - ref, u.z - ref, u.w - ref);
    }
}

static int blocks_for(long long n, int threads) {
    long long b = (n + threads - 1) / threads;
    if (b > 152 * 64) b = 152 * 64;
    if (b < 1) b = 1;
    return (int)b;
}

cudaError_t launch_grid_prep(const void *raw, int dtype, const GridSizes &sz, double *pad64, float *pad32,
                             float4 *quad, float4 *table, cudaStream_t st) {
    const long long n_pad = (long long)(sz.n_lat + 2) * (sz.n_lon + 2) * (sz.n_alt + 2);
    if (dtype == RT_F64)
        pad_kernel<double><<<blocks_for(n_pad, 256), 256, 0, st>>>((const double *)raw, pad64, pad32, sz.n_lat,
                                                                    sz.n_lon, sz.n_alt);
    else
        pad_kernel<float><<<blocks_for(n_pad, 256), 256, 0, st>>>((const float *)raw, pad64, pad32, sz.n_lat,
                                                                   sz.n_lon, sz.n_alt);
    const long long n_quad = (long long)(sz.n_lat + 2) * (sz.n_lon + 2) * (sz.n_alt - 1);
    quad_kernel<<<blocks_for(n_quad, 256), 256, 0, st>>>(pad32, quad, sz.n_lat, sz.n_lon, sz.n_alt);
    if (table) {
        const long long n_tab = (long long)(sz.n_lat - 1) * (sz.n_lon - 1) * (sz.n_alt - 1) * 16;
        table_kernel<<<blocks_for(n_tab, 256), 256, 0, st>>>(quad, table, sz.n_lat, sz.n_lon, sz.n_alt);
    }
    return cudaGetLastError();
}

// ================================================================ utilities
__device__ __forceinline__ double wrap180(double x) { return x - 360.0 * floor((x + 180.0) / 360.0); }

// Output quantities of a final state (Sec. II-C: group path, ground distance,
// azimuth deviation, reflection height): central angle and initial bearing
// on the sphere from the transmitter (tx_th, tx_ph) to (th, ph).  Out of line
// (it runs once per ray) with scalar arguments, so that neither the caller's
// state nor the kernel parameters need an address.
__device__ __noinline__ void finish_result(double tx_th, double tx_ph, double az_launch, double th, double ph,
                                           double P, double apo, int status, int n_steps, int n_att, int n_evals,
                                           double R_E, rt_ray_result *out) {
    double s0, c0, s1, c1, sd, cd;
    sincos(tx_th, &s0, &c0);
    sincos(th, &s1, &c1);
    sincos(ph - tx_ph, &sd, &cd);
    const double east = s1 * sd;                 // components of the final point in the
    const double north = s0 * c1 - c0 * s1 * cd;  // tangent plane at the transmitter
    const double dot = s0 * s1 * cd + c0 * c1;
    const double ang = atan2(sqrt(east * east + north * north), dot);
    rt_ray_result r;
    r.group_path_km = P;
    r.ground_range_km = R_E * ang;
    r.az_dev_deg = ang > 1e-15 ? wrap180(atan2(east, north) * kRad2Deg - az_launch * kRad2Deg) : 0.0;
    r.apogee_km = apo;
    r.land_lat_deg = 90.0 - th * kRad2Deg;
    r.land_lon_deg = wrap180(ph * kRad2Deg);
    r.status = status;
    r.n_steps = n_steps;
    r.n_attempts = n_att;
    r.n_evals = n_evals;
    *out = r;
}

// RKF45 error norm (<= 1 accepts) and step factor, as documented in rtgd.h.
__device__ __forceinline__ float rkf45_err(float r, float sth, float kmag, const float e[6], float rtol, float atol) {
    const float pos = fmax(fabs(e[0]), fmax(r * fabs(e[1]), r * sth * fabs(e[2])));
    const float kerr = fmax(fabs(e[3]), fmax(fabs(e[4]), fabs(e[5])));
    return fmax(fdiv(pos, atol + rtol * r), fdiv(kerr, rtol * fmax(kmag, 1e-3f)));
}

// =============================================================== mixed path
// The ray state (r, theta, phi, k) and the group path stay in double.  Each
// step attempt starts from a "base": the grid cell and in-cell coordinates of
// the state plus float copies of r, k and of the sines and cosines of theta
// and phi.  A stage works on float offsets delta from the base: its grid
// coordinates are base + delta * (d coord / d state) (the coordinates are
// linear in r, theta, phi), and sin/cos of theta + delta by angle addition,
// so everything after (weights, contraction, dipole, Appleton-Hartree, Eq. 1)
// runs in float without losing the base's resolution.  An accepted step adds
// the float increment to the double position (r, theta, phi) and the double
// group path -- the only FP64 arithmetic of a step; the wave vector, a
// quantity of order 1, accumulates as a compensated float pair (hi + lo).
// The base (cells, altitude, radius, sines and cosines) follows by the same
// increment in float and is recomputed from the double state every
// kResyncSteps accepted steps.  GB300 issues FP64 at 1/64 of the FP32 rate,
// so the step bookkeeping must stay out of double precision.
constexpr int kResyncSteps = 16;

struct Base32 {
    int ia, ib, ic;            // cell of the base (may lie outside the grid)
    float ta, tb, tc;          // in-cell coordinates
    float r, alt;              // radius and altitude (km)
    float sth, cth, sph, cph;  // sin/cos of colatitude and longitude
    float k[3];
};

__device__ __noinline__ double widen_rare(float x) { return (double)x; }
__device__ __noinline__ float narrow_rare(double x) { return (float)x; }

// (double)x and (float)x by integer operations: a conversion is an FP64-rate
// instruction (64 cycles of a warp on GB300), these are ~8 integer ones.
// Subnormals, infinities, NaN and doubles outside the normal float range take
// the conversion, out of line (see wrap360_rare).
__device__ __forceinline__ double widen(float x) {
    const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0) return widen_rare(x);
    return __hiloint2double((int)((b & 0x80000000u) | (m == 0 ? 0u : (m >> 3) + 0x38000000u)), (int)(b << 29));
}
__device__ __forceinline__ float narrow(double x) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x), m = b & 0x7fffffffffffffffull;
    const unsigned e = (unsigned)(m >> 52);
    if (e - 897u >= 253u) return narrow_rare(x);  // exponents 897..1149: normal floats, rounding cannot overflow
    const unsigned long long r = m - (896ull << 52) + 0x0fffffffull + ((m >> 29) & 1ull);  // to nearest, ties to even
    return __uint_as_float((unsigned)(r >> 29) | ((unsigned)(b >> 32) & 0x80000000u));
}

__device__ __noinline__ int floor_cell_rare(double x, float *t, int far) {
    const double f = floor(x);
    *t = (float)(x - f);
    return (int)fmin(fmax(f, -(double)far), (double)far);
}

// floor(x) as an integer and the fraction x - floor(x): one addition rounded
// down.  Beyond +-far (and for NaN) the cell is clamped to that (negative side
// for NaN), which lies outside of the grid.
__device__ __forceinline__ int floor_cell(double x, float &t, int far) {
    const double magic = 6755399441055744.0;  // 1.5 * 2^52
    const int hi = __double2hiint(x) & 0x7fffffff;
    if (hi >= 0x41d00000) return floor_cell_rare(x, &t, far);  // |x| >= 2^30
    const double big = __dadd_rd(x, magic);
    t = narrow(x - (big - magic));
    return min(max(__double2loint(big), -far), far);
}

// Base of a double state (double arithmetic; used at launch and to resync).
// Out of line with scalar arguments (it runs at launch and every kResyncSteps
// accepted steps), returning the base by value; the caller sets the wave
// vector.  The rays of a warp resync at different steps, so almost every
// attempt of a full warp waits for this once: 17 FP64 instructions (a further
// 8 in lane_fold), where floors, clamps, conversions and a division-free wrap
// in FP64 made it ~65.
__device__ __noinline__ Base32 base_of(double lat0, double lon0, double inv_dlat, double inv_dlon, double R_E,
                                       double alt0, double inv_dalt, int far, double r, double th,
                                       double ph) {
    Base32 b;
    const double lat = 90.0 - th * kRad2Deg;
    const double lonrel = wrap360(ph * kRad2Deg - lon0);
    const double alt = r - R_E;
    b.ia = floor_cell((lat - lat0) * inv_dlat, b.ta, far);
    b.ib = floor_cell(lonrel * inv_dlon, b.tb, far);
    b.ic = floor_cell((alt - alt0) * inv_dalt, b.tc, far);
    b.r = narrow(r);
    b.alt = narrow(alt);
    sincosf(narrow(th), &b.sth, &b.cth);
    sincosf(narrow(ph), &b.sph, &b.cph);
    return b;
}

__device__ __forceinline__ void base_from_state(const GridDev &g, const double y[6], Base32 &b) {
    b = base_of(g.lat0, g.lon0, g.inv_dlat, g.inv_dlon, g.R_E, g.alt0, g.inv_dalt, g.far_cells, y[0], y[1], y[2]);
#pragma unroll
    for (int i = 0; i < 3; ++i) b.k[i] = (float)y[3 + i];
}

// (A shift of more than 2^29 cells stays in t; the index stays within 1.5 * 2^30.)
__device__ __forceinline__ void shift_axis(int &i, float &t, float dt) {
    const float u = t + dt;
    const float fl = fminf(fmaxf(floorf(u), -0x1p29f), 0x1p29f);
    i = min(max(i, -(1 << 30)), 1 << 30) + (int)fl;
    t = u - fl;
}

// sin/cos of (x0 + d) from sin/cos of x0, for |d| well below 0.1 rad (series
// error < d^7/5040).
__device__ __forceinline__ void angle_add(float s0, float c0, float d, float &s, float &c) {
    const float d2 = d * d;
    const float sd = d * (1.0f - d2 * (1.0f / 6.0f) * (1.0f - d2 * 0.05f));
    const float cd = 1.0f - 0.5f * d2 * (1.0f - d2 * (1.0f / 12.0f));
    s = s0 * cd + c0 * sd;
    c = c0 * cd - s0 * sd;
}

// Moves the base by the accepted increment d in float; k_hi is the new wave
// vector (high parts).
__device__ __forceinline__ void advance_base(const GridDev &g, Base32 &b, const float d[6], const float k_hi[3]) {
    shift_axis(b.ia, b.ta, g.sa * d[1]);
    shift_axis(b.ib, b.tb, g.sb * d[2]);
    shift_axis(b.ic, b.tc, g.sc * d[0]);
    b.r += d[0];
    b.alt += d[0];
    float s, c;
    angle_add(b.sth, b.cth, d[1], s, c);
    b.sth = s;
    b.cth = c;
    angle_add(b.sph, b.cph, d[2], s, c);
    b.sph = s;
    b.cph = c;
    b.k[0] = k_hi[0];
    b.k[1] = k_hi[1];
    b.k[2] = k_hi[2];
}

// hi + lo += d with the rounding error of hi + d kept in lo (Knuth's TwoSum).
__device__ __forceinline__ void two_sum_add(float &hi, float &lo, float d) {
    const float s = hi + d;
    const float bp = s - hi;
    const float err = (hi - (s - bp)) + (d - bp);
    hi = s;
    lo += err;
}

// Stage cell along one axis from base cell i0 and offset coordinate t = t0 +
// delta * scale; false outside [0, n-1], and then cell 0 at t = 0, so that the
// caller can gather from an in-bounds cell without branching.  On the critical
// path of every stage, so floor(t) costs one addition: t + 1.5 * 2^23 rounded
// down holds it in the low mantissa bits.  That is exact for |t| < 2^22.  Beyond
// that, and for NaN, the integer lands at least 2^22 cells out, which the index
// test refuses where base cells lie within 2^21 of a grid of at most 2^20 nodes
// per axis; longer axes have g.far_stage.  Nine instructions; with a clamp and a
// round-to-nearest that was corrected afterwards it took sixteen.
__device__ __forceinline__ bool stage_cell(int i0, float t, int n, int &i, float &tt) {
    const float magic = 12582912.0f;
    const float big = __fadd_rd(t, magic);
    const int ii = (int)((unsigned)i0 + (unsigned)__float_as_int(big) - (unsigned)__float_as_int(magic));
    const float tr = t - (big - magic);
    const bool last = (ii == n - 1) & (tr == 0.0f);  // the last node: cell n-2 at t = 1
    // tr = t - floor(t) lies in [0, 1] by construction, so the cell index alone decides
    const bool ok = (unsigned)ii < (unsigned)(n - 1);
    i = last ? n - 2 : (ok ? ii : 0);
    tt = last ? 1.0f : (ok ? tr : 0.0f);
    return ok | last;
}

// Lat-weights of the rows a = q*4/G .. (q+1)*4/G - 1 handled by lane q of a
// group of G lanes (G = 1: all four).
template <int G, int IP>
__device__ __forceinline__ void own_lat_weights(float ta, int q, float wa[4], float da[4]) {
    if (G == 1) {
        axis_weights<IP>(ta, wa, da);
    } else if (G == 2) {
        const bool hi = q != 0;  // rows 2, 3: nodes j+1, j+2
        float wm1, w0, dm1, d0;
        half_weights<IP>(hi ? 1.0f - ta : ta, wm1, w0, dm1, d0);
        wa[0] = hi ? w0 : wm1;
        wa[1] = hi ? wm1 : w0;
        da[0] = hi ? -d0 : dm1;
        da[1] = hi ? -dm1 : d0;
    } else {
        const bool hi = q >= 2;
        float wm1, w0, dm1, d0;
        half_weights<IP>(hi ? 1.0f - ta : ta, wm1, w0, dm1, d0);
        const bool outer = q == 0 || q == 3;  // nodes j-1, j+2
        wa[0] = outer ? wm1 : w0;
        da[0] = (outer ? dm1 : d0) * (hi ? -1.0f : 1.0f);
    }
}

// Index of (i, j, k) in an array of rows of n_k entries, n_j rows per i: the
// row number in 32 bits (a grid with 2^32 (lat, lon) rows of four samples
// would not fit the device), then one wide multiply-add.
__device__ __forceinline__ unsigned long long row_index(int i, int n_j, int j, int n_k, int k) {
    const unsigned row = (unsigned)i * (unsigned)n_j + (unsigned)j;
    return (unsigned long long)row * (unsigned)n_k + (unsigned)k;
}

// dy/dP' (float) at base + delta.  STENCIL selects where the 64 samples come
// from and IP the interpolant (0 GD, 1 Catmull-Rom); with G > 1 the G lanes
// of a group (lane q, shuffle mask gmask) split the 16 sample rows and combine
// their partial sums with a butterfly, whose every addition is commutative,
// so all lanes hold bitwise equal results.  The body has no branch: the field
// terms (which do not need Ne) come first and can overlap the sample gathers,
// and a stage outside the grid gathers from cell 0 and discards the result.
template <int STENCIL, int G, int IP, bool FIRST>
__device__ __forceinline__ void rhs_mixed(const GridDev &g, const RayPhys<float> &rp, const Base32 &b,
                                          const float d[6], float dy[6], float *mu2, int q, unsigned gmask) {
    StageIn<float> s;
    const float xa = b.ta + g.sa * d[1], xb = b.tb + g.sb * d[2], xc = b.tc + g.sc * d[0];
    s.r = b.r + d[0];
    angle_add(b.sth, b.cth, d[1], s.sth, s.cth);
    angle_add(b.sph, b.cph, d[2], s.sph, s.cph);
    s.k[0] = b.k[0] + d[3];
    s.k[1] = b.k[1] + d[4];
    s.k[2] = b.k[2] + d[5];
    const FieldTerms F = field_terms(rp, s);
    int ia, ib, ic;
    float ta, tb, tc;
    const bool in_a = stage_cell(b.ia, xa, g.n_lat, ia, ta);
    const bool in_b = stage_cell(b.ib, xb, g.n_lon, ib, tb);
    const bool in_c = stage_cell(b.ic, xc, g.n_alt, ic, tc);
    const bool inside = in_a & in_b & in_c;  // each axis is in bounds by itself
    // beyond far_stage NaN, so that the adaptive step control retries with a
    // smaller step and a fixed step ends the ray as not finite
    const float far = fmaxf(fmaxf(fabsf(xa), fabsf(xb)), fabsf(xc)) <= g.far_stage ? 0.0f : NAN;
    float wa[4], da[4], wb[4], db[4], wc[4], dc[4], out[4], ref;
    constexpr int NA = 4 / G;
    const int a0 = q * NA;
    own_lat_weights<G, IP>(ta, q, wa, da);
    axis_weights<IP>(tb, wb, db);
    axis_weights<IP>(tc, wc, dc);
    if (STENCIL == RT_STENCIL_QUAD) {
        // quad (pi, pj, k): 4 samples of cell k in padded row (pi, pj); node i-1 -> padded i
        const long long sj = g.q_alt, si = (long long)(g.n_lon + 2) * g.q_alt;
        const float4 *qp = g.quad + row_index(ia, g.n_lon + 2, ib, g.q_alt, ic);
        ref = __ldg(qp + si + sj).y;  // node (ia, ib, ic)
#define RTGD_ROWQ(a, b, u0, u1, u2, u3)                    \
    {                                                      \
        const float4 v_ = __ldg(qp + (a) * si + (b) * sj); \
        u0 = v_.x;                                        \
        u1 = v_.y;                                        \
        u2 = v_.z;                                        \
        u3 = v_.w;                                        \
    }
        RTGD_CONTRACT((G > 1), RTGD_ROWQ, ref, a0, NA, wa, da, wb, db, wc, dc, out);
#undef RTGD_ROWQ
    } else if (STENCIL == RT_STENCIL_TABLE) {
        // one lane per ray: products in 64 bits.  Fewer instructions through
        // row_index, but the one-lane loop then schedules its 17 loads worse
        // (495,122 rays 71.6 against 65.6 ms); several lanes gain (C2 fan at four
        // lanes 11.75 against 11.9 ms)
        const long long cell = G == 1 ? ((long long)ia * (g.n_lon - 1) + ib) * (g.n_alt - 1) + ic
                                      : (long long)row_index(ia, g.n_lon - 1, ib, g.q_alt, ic);
        const float4 *qp = g.table + cell * 16;  // samples minus the node (ia, ib, ic)
        ref = __ldg(g.pad32 + (G == 1 ? (long long)(ia + 1) * g.p_lon * g.p_alt + (long long)(ib + 1) * g.p_alt + ic + 1
                                      : (long long)row_index(ia + 1, g.p_lon, ib + 1, g.p_alt, ic + 1)));
#define RTGD_ROWT(a, b, u0, u1, u2, u3)              \
    {                                                \
        const float4 v_ = __ldg(qp + (a) * 4 + (b)); \
        u0 = v_.x;                                  \
        u1 = v_.y;                                  \
        u2 = v_.z;                                  \
        u3 = v_.w;                                  \
    }
        RTGD_CONTRACT((G > 1), RTGD_ROWT, 0.0f, a0, NA, wa, da, wb, db, wc, dc, out);
#undef RTGD_ROWT
    } else {
        const long long sj = g.p_alt, si = (long long)g.p_lon * g.p_alt;
        const float *p = g.pad32 + row_index(ia, g.p_lon, ib, g.p_alt, ic);
        ref = __ldg(p + si + sj + 1);  // node (ia, ib, ic)
#define RTGD_ROWG(a, b, u0, u1, u2, u3)            \
    {                                              \
        const float *p_ = p + (a) * si + (b) * sj; \
        u0 = __ldg(p_);                            \
        u1 = __ldg(p_ + 1);                        \
        u2 = __ldg(p_ + 2);                        \
        u3 = __ldg(p_ + 3);                        \
    }
        RTGD_CONTRACT((G > 1), RTGD_ROWG, ref, a0, NA, wa, da, wb, db, wc, dc, out);
#undef RTGD_ROWG
    }
    if (G > 1) {
#pragma unroll
        for (int o = 1; o < G; o <<= 1) {
#pragma unroll
            for (int i = 0; i < 4; ++i) out[i] += __shfl_xor_sync(gmask, out[i], o);
        }
    }
    out[0] += ref;
    // Ne = 0 outside the grid box (selects, so that samples gathered there,
    // whatever they hold, never reach the result)
    s.X = inside ? fmaf(rp.xfac, out[0], far) : far;
    s.dX[0] = inside ? rp.xfac * out[3] * g.sc : 0.0f;
    s.dX[1] = inside ? rp.xfac * out[1] * g.sa : 0.0f;
    s.dX[2] = inside ? rp.xfac * out[2] * g.sb : 0.0f;
    ray_rhs<FIRST>(rp, s, F, dy, mu2);
}

// Butcher tables in "shifted accumulator" form.  After stage s produced k_s,
// acc[t] <- acc[t+1] + A[s][t] k_s (t = 0..4, acc[5] = 0), so acc[0] always
// holds sum_j a[s+1][j] k_j, the offset (over h) of the next stage; y4 and the
// error estimate accumulate B4[s] k_s and E[s] k_s.
struct Tableau {
    // row s: {A[s][0..3]} and {A[s][4], B4[s], E[s], 0}, two 16-byte loads per stage
    float4 lo[6];
    float4 hi[6];
    int ns;
};

__constant__ Tableau c_tab[2];  // [RT_RK4], [RT_RKF45]

// Quantised step factor in float (the mixed path's counterpart of
// step_factor64): 2^(k/4), k = floor(4 log2 of the limited 0.9 err^(-1/5)).
// One logarithm gives that exponent to ~1e-5; within 1e-3 of an integer (and
// for err = 0, infinite or NaN) the factor itself decides.
__device__ __forceinline__ float step_factor_f(float err) {
    const float l = -0.608012374f - 0.8f * __log2f(err);  // 4 log2(0.9 err^-0.2)
    const float fl = floorf(l), d = l - fl;
    int k = (int)fl;
    if (!(d > 1e-3f && d < 0.999f)) {
        const float fac = (err == 0.0f) ? 5.0f : fminf(5.0f, fmaxf(0.2f, 0.9f * __powf(err, -0.2f)));
        k = (int)floorf(4.0f * __log2f(fac));
    }
    k = k < -10 ? -10 : (k > 9 ? 9 : k);
    // 2^(k/4): the mantissa of 2^0, 2^(1/4), 2^(1/2) or 2^(3/4) and the exponent floor(k/4)
    const int m = (k & 2) ? ((k & 1) ? 0x3fd744fd : 0x3fb504f3) : ((k & 1) ? 0x3f9837f0 : 0x3f800000);
    return __int_as_float(m + ((k >> 2) << 23));
}

// Peak rise of the cubic Hermite fit over one step, relative to its start:
// p(s) = m0 s + B s^2 + A s^3 with p(1) = dr, p'(0) = m0 > 0 >= p'(1) = m1.
__device__ __noinline__ float hermite_rise_f(float dr, float m0, float m1) {  // once per ray: out of line
    const float A = m0 + m1 - 2.0f * dr, B = 3.0f * dr - 2.0f * m0 - m1;
    float lo = 0.0f, hi = 1.0f;
    for (int it = 0; it < 24; ++it) {
        const float mid = 0.5f * (lo + hi);
        if (m0 + 2.0f * B * mid + 3.0f * A * mid * mid > 0.0f) lo = mid;
        else hi = mid;
    }
    const float s = 0.5f * (lo + hi);
    return s * (m0 + s * (B + s * A));
}

// Float counterpart of face_axis64 on the base's (cell, fraction) grid
// coordinates: the distance to the next face is (integer - fraction) / rate.
// Without branches: the three axes' quotients overlap, and the rays of a warp
// head in different directions (with branches on the signs it took 670 cycles
// of a lone warp's 7,600 per attempt).
__device__ __forceinline__ float face_axis_f(int i, float t, int n, float v) {
    const bool up = v > 0.0f;
    const int F = up ? max(i + 1, 0) : min(t > 0.0f ? i : i - 1, n - 1);
    const bool ok = up ? F <= n - 1 : (v < 0.0f && F >= 0);
    const float d = fdiv((float)(F - i) - t, v);
    return ok ? d : INFINITY;
}

__device__ __forceinline__ float face_distance_f(const GridDev &g, const Base32 &b, const float k1[6]) {
    const float c = face_axis_f(b.ic, b.tc, g.n_alt, g.sc * k1[0]);
    const float l = fminf(face_axis_f(b.ia, b.ta, g.n_lat, g.sa * k1[1]), face_axis_f(b.ib, b.tb, g.n_lon, g.sb * k1[2]));
    // lateral faces count only inside the altitude span
    const bool in_alt = (unsigned)b.ic < (unsigned)(g.n_alt - 1) || (b.ic == g.n_alt - 1 && b.tc == 0.0f);
    return in_alt ? fminf(c, l) : c;
}

// Per-lane state of the mixed tracer.
struct Lane {
    double y[3];              // r (km), theta, phi (rad): the FP64 position
    double P;                 // group path (km)
    float inc_hi[4], inc_lo[4];  // increments of (r, theta, phi, P') not yet added to y and P,
                                 // as compensated float pairs (see lane_fold)
    float k_hi[3], k_lo[3];   // wave vector as a compensated float pair
    float r_prev;             // radius at the start of the last accepted step
    float h, hs;              // next step / step of the current attempt (km)
    float h_prev, dr_prev;    // last accepted step and its dr/dP' at the start
    float apo;                // reflection height so far (km)
    float acc[5][6];
    float y4[6], e[6];
    float k1[6];
    float xfac, ab0;
    Base32 b;
    int out_id, mode;
    int n_steps, n_att, n_ev, status, since_sync;
    bool active, launch, landing, exiting, have_prev, k1_valid, at_face;
};

// State of the landing / exit solve of one lane (Illinois regula falsi on the
// step size: bracket [la, lb] with signed distances lfa, lfb from the target
// radius).  Used only on a ray's last step: the persistent kernel keeps it in
// a per-thread shared-memory slot (its refill code leaves fewer registers for
// the ray state; measured 8 % faster on the 495k-ray batch), the plain
// kernels in registers.
struct LandState {
    double la, lfa, lb, lfb;
    int side, it;
};

__device__ __forceinline__ RayPhys<float> lane_phys(const GridDev &g, const Lane &L) {
    RayPhys<float> p;
    p.xfac = L.xfac;
    p.ab0 = L.ab0;
    p.R_E = g.R_Ef;
    p.m[0] = g.mf[0];
    p.m[1] = g.mf[1];
    p.m[2] = g.mf[2];
    p.iso = g.iso != 0;
    p.mode = L.mode;
    return p;
}

// Stage 0 of an attempt: acc/y4/e start from k1.
__device__ __forceinline__ void accumulate_first(Lane &L, const Tableau &T, const float k1[6]) {
    const float4 lo = T.lo[0], hi = T.hi[0];
    const float A[5] = {lo.x, lo.y, lo.z, lo.w, hi.x};
    const float b4 = hi.y, e = hi.z;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
#pragma unroll
        for (int t = 0; t < 5; ++t) L.acc[t][c] = A[t] * k1[c];
        L.y4[c] = b4 * k1[c];
        L.e[c] = e * k1[c];
    }
}

// Stage s >= 1: shift the accumulators and add stage s's output ks.
__device__ __forceinline__ void accumulate_next(Lane &L, const Tableau &T, int s, const float ks[6]) {
    const float4 lo = T.lo[s], hi = T.hi[s];
    const float A[5] = {lo.x, lo.y, lo.z, lo.w, hi.x};
    const float b4 = hi.y, e = hi.z;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
#pragma unroll
        for (int t = 0; t < 4; ++t) L.acc[t][c] = L.acc[t + 1][c] + A[t] * ks[c];
        L.acc[4][c] = A[4] * ks[c];
        L.y4[c] += b4 * ks[c];
        L.e[c] += e * ks[c];
    }
}

// Base of the transmitter position (the launch state of every ray of the
// fan; the wave vector part is set per ray).
__device__ __forceinline__ Base32 tx_base(const GridDev &g, const FanDev &f) {
    Base32 b = base_of(g.lat0, g.lon0, g.inv_dlat, g.inv_dlon, g.R_E, g.alt0, g.inv_dalt, g.far_cells, f.tx_r, f.tx_th, f.tx_ph);
    b.k[0] = b.k[1] = b.k[2] = 0.0f;
    return b;
}

// Starts ray `id`: per-ray constants from the fan's tables, FP64 launch
// state, and the float base: the transmitter's (btx, shared by the fan) with
// this ray's wave vector.
__device__ void lane_begin_ray(Lane &L, const GridDev &g, const FanDev &f, long long id, const Base32 &btx) {
    const RayParams p = ray_params(f, id);
    L.out_id = (int)id;
    L.xfac = p.xfac;
    L.ab0 = p.ab0;
    L.mode = p.mode;
    double y[6];
    launch_dir(f, p, y);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        L.y[i] = y[i];
        L.k_hi[i] = (float)y[3 + i];
        L.k_lo[i] = 0.0f;
    }
    L.P = 0.0;
#pragma unroll
    for (int i = 0; i < 4; ++i) L.inc_hi[i] = L.inc_lo[i] = 0.0f;
    L.h = f.h0_f;
    L.apo = (float)(f.tx_r - g.R_E);
    L.n_steps = L.n_att = L.n_ev = 0;
    L.since_sync = 0;
    L.status = RT_RAY_NOT_RUN;
    L.have_prev = L.k1_valid = L.landing = L.exiting = false;
    L.launch = true;
    L.b = btx;
#pragma unroll
    for (int i = 0; i < 3; ++i) L.b.k[i] = (float)y[3 + i];
}

// Adds the pending increments to the FP64 position and group path.  An
// accepted step adds its float increments of r, theta, phi and P' to
// compensated float pairs (TwoSum: hi + lo carries their sum to ~2^-48
// relative), and the pairs reach the double state only here: at the base
// resync every kResyncSteps steps, before a landing / exit solve and when the
// ray ends.  So the FP64 pipe (1/64 of the FP32 rate on GB300) sees four
// conversions and additions per component every kResyncSteps steps instead of
// two per component every step; the position agrees with step-by-step double
// accumulation to ~1e-12 km.
__device__ __forceinline__ void lane_fold(Lane &L) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        L.y[i] += widen(L.inc_hi[i]) + widen(L.inc_lo[i]);
        L.inc_hi[i] = L.inc_lo[i] = 0.0f;
    }
    L.P += widen(L.inc_hi[3]) + widen(L.inc_lo[3]);
    L.inc_hi[3] = L.inc_lo[3] = 0.0f;
}

// Double copy of the full state (position, wave vector hi + lo); the pending
// increments must have been folded in.
__device__ __forceinline__ void lane_state(const Lane &L, double y[6]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        y[i] = L.y[i];
        y[3 + i] = (double)L.k_hi[i] + (double)L.k_lo[i];
    }
}

// Writes a ray's raw final state into its record: colatitude and longitude
// (rad) stand in the ground-range and azimuth-deviation fields until
// finish_records_kernel turns them into the outputs.  The outputs' double
// trigonometry would otherwise run here, in a branch taken by the lanes of
// one ray while the rest of the warp waits on the 1/64-rate FP64 pipe.
__device__ __forceinline__ void lane_finish(Lane &L, const GridDev &g, const FanDev &f, rt_ray_result *out,
                                            bool writer = true) {
    L.active = false;
    if (!writer) return;
    lane_fold(L);
    rt_ray_result r;
    r.group_path_km = L.P;
    r.ground_range_km = L.y[1];
    r.az_dev_deg = L.y[2];
    r.apogee_km = (double)L.apo;
    r.land_lat_deg = 0.0;
    r.land_lon_deg = 0.0;
    r.status = L.status;
    r.n_steps = L.n_steps;
    r.n_attempts = L.n_att;
    r.n_evals = L.n_ev;
    out[L.out_id] = r;
}

// Final outputs of the records, one thread per record (a converged pass after
// the trace, mixed and FP64): record k of a fan holds the raw final state that
// lane_finish or write_raw wrote; k is its canonical index, which gives the
// launch azimuth.
__global__ void finish_records_kernel(double R_E, FanDev f, rt_ray_result *__restrict__ out, long long n) {
    const long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (k >= n) return;
    const rt_ray_result r = out[k];
    const double az = f.az[(unsigned)k % (unsigned)f.n_az].rad;
    finish_result(f.tx_th, f.tx_ph, az, r.ground_range_km, r.az_dev_deg, r.group_path_km, r.apogee_km, r.status,
                  r.n_steps, r.n_attempts, r.n_evals, R_E, out + k);
}

// The same for the records of several fans traced in one launch: record i
// belongs to fan k with first[k] <= i < first[k + 1].
__global__ void finish_fans_records_kernel(double R_E, const FanDev *__restrict__ fans,
                                           const long long *__restrict__ first, int n_fans,
                                           rt_ray_result *__restrict__ out) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= first[n_fans]) return;
    int lo = 0, hi = n_fans - 1;
    while (lo < hi) {  // largest k with first[k] <= i
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    const FanDev &f = fans[lo];
    const long long k = i - first[lo];
    const rt_ray_result r = out[i];
    const double az = f.az[(unsigned)k % (unsigned)f.n_az].rad;
    finish_result(f.tx_th, f.tx_ph, az, r.ground_range_km, r.az_dev_deg, r.group_path_km, r.apogee_km, r.status,
                  r.n_steps, r.n_attempts, r.n_evals, R_E, out + i);
}

// Once k1 is known: the accumulators start from it, an adaptive step ends just
// past the next cell face, and the group-path limit clips it.  The
// accumulation's 42 products stand in the face distance's block, beside its
// divisions.
__device__ __forceinline__ void lane_limit_step(Lane &L, const GridDev &g, const FanDev &f, const Tableau &T) {
    if (f.integrator == RT_RKF45) {
        const float hf = face_distance_f(g, L.b, L.k1);
        accumulate_first(L, T, L.k1);
        const bool cut = !L.landing && hf > 1e-3f * L.hs && hf < L.hs;
        L.hs = cut ? hf * (1.0f + 1e-4f) : L.hs;
        L.at_face = L.at_face || cut;
    } else {
        accumulate_first(L, T, L.k1);
    }
    if (f.has_max_path && !L.landing) {
        const double P = L.P + ((double)L.inc_hi[3] + (double)L.inc_lo[3]);
        if (P + (double)L.hs > f.max_path) L.hs = (float)(f.max_path - P);
    }
}

// Sets up the next step attempt from the current state; returns false when
// the ray stops (step budget).
__device__ __forceinline__ bool lane_next_attempt(Lane &L, const FanDev &f) {
    if (L.n_att >= f.max_steps) {
        L.status = RT_RAY_MAX_STEPS;
        return false;
    }
    if (!L.landing) {
        L.hs = L.h;
        L.at_face = false;
    }
    return true;
}

// The launch evaluation: mu^2 at the transmitter for the launch direction,
// then |k| = mu.  Returns true when the ray has finished (status set).
template <int STENCIL, int G, int IP, bool FIRST>
__device__ bool lane_launch(Lane &L, const GridDev &g, const FanDev &f, int q, unsigned gmask) {
    const RayPhys<float> rp = lane_phys(g, L);
    float d[6], ks[6], mu2;
#pragma unroll
    for (int c = 0; c < 6; ++c) d[c] = 0.0f;
    rhs_mixed<STENCIL, G, IP, FIRST>(g, rp, L.b, d, ks, &mu2, q, gmask);
    ++L.n_ev;
    L.launch = false;
    if (!(mu2 > 0.0f)) {
        L.status = RT_RAY_NONFINITE;
        return true;
    }
    // |k| = mu: rescale the launch direction (double), split into hi + lo
    const double mu = sqrt((double)mu2);
    double y[6];
    lane_state(L, y);
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const double k = y[3 + i] * mu;
        L.k_hi[i] = (float)k;
        L.k_lo[i] = (float)(k - (double)L.k_hi[i]);
        L.b.k[i] = L.k_hi[i];
    }
    return !lane_next_attempt(L, f);
}

// Stage 0 bookkeeping once k1 is known: apogee check, face-limited step,
// accumulators.
__device__ __forceinline__ void lane_stage0_done(Lane &L, const GridDev &g, const FanDev &f, const Tableau &T,
                                                 bool fresh) {
    if (fresh) {
        L.k1_valid = true;
        if (L.have_prev && L.dr_prev > 0.0f && L.k1[0] <= 0.0f) {
            const float rise = hermite_rise_f(L.b.r - L.r_prev, L.h_prev * L.dr_prev, L.h_prev * L.k1[0]);
            L.apo = fmaxf(L.apo, L.b.alt - (L.b.r - L.r_prev) + rise);
        }
        L.have_prev = false;
    }
    lane_limit_step(L, g, f, T);
}

// The stages of one step attempt.  Every lane of a warp runs its attempt in
// the same loop, so the stage index is warp-uniform: the lanes stay converged
// and the Butcher coefficients are broadcast reads.  Stage 0 is evaluated
// only when k1 at the current state is not yet known (after a rejected
// attempt or during the landing solve it is): such lanes sit out that one
// evaluation.  With one lane per ray (throughput-bound fans) one copy of the
// stage evaluation serves all stages, which keeps the loop inside the
// instruction cache; with 2 or 4 lanes per ray (latency-bound fans) stage 0
// is a separate copy, which schedules better.
template <int STENCIL, int G, int IP, bool FIRST>
__device__ __forceinline__ void lane_attempt(Lane &L, const GridDev &g, const FanDev &f, const Tableau &T, int q,
                                             unsigned gmask) {
    const RayPhys<float> rp = lane_phys(g, L);
    float d[6], ks[6];
    if (G == 1) {
#pragma unroll 1
        for (int s = 0; s < T.ns; ++s) {
            const bool fresh = s == 0 && !L.k1_valid;
            if (s > 0 || fresh) {
#pragma unroll
                for (int c = 0; c < 6; ++c) d[c] = s == 0 ? 0.0f : L.hs * L.acc[0][c];
                rhs_mixed<STENCIL, G, IP, FIRST>(g, rp, L.b, d, ks, nullptr, q, gmask);
                ++L.n_ev;
            }
            if (s == 0) {
                if (fresh) {
#pragma unroll
                    for (int c = 0; c < 6; ++c) L.k1[c] = ks[c];
                }
                lane_stage0_done(L, g, f, T, fresh);
            } else {
                accumulate_next(L, T, s, ks);
            }
        }
    } else {
        const bool fresh = !L.k1_valid;
        if (fresh) {
#pragma unroll
            for (int c = 0; c < 6; ++c) d[c] = 0.0f;
            rhs_mixed<STENCIL, G, IP, FIRST>(g, rp, L.b, d, L.k1, nullptr, q, gmask);
            ++L.n_ev;
        }
        lane_stage0_done(L, g, f, T, fresh);
#pragma unroll 1
        for (int s = 1; s < T.ns; ++s) {
#pragma unroll
            for (int c = 0; c < 6; ++c) d[c] = L.hs * L.acc[0][c];
            rhs_mixed<STENCIL, G, IP, FIRST>(g, rp, L.b, d, ks, nullptr, q, gmask);
            ++L.n_ev;
            accumulate_next(L, T, s, ks);
        }
    }
}

// Bracket of the landing / exit solve (Illinois regula falsi on the step size).
struct Bracket {
    double la, lfa, lb, lfb;
    int side;
};

// One regula falsi update with the new point (c, fc); returns the next step
// size.  Out of line: it runs only on the last step of a ray.
__device__ __noinline__ double bracket_update(Bracket &B, double c, double fc) {
    if (fc < 0.0) {
        B.lb = c;
        B.lfb = fc;
        if (B.side == -1) B.lfa *= 0.5;
        B.side = -1;
    } else {
        B.la = c;
        B.lfa = fc;
        if (B.side == 1) B.lfb *= 0.5;
        B.side = 1;
    }
    return B.lb - B.lfb * (B.lb - B.la) / (B.lfb - B.lfa);
}

__device__ __noinline__ double bracket_first(double lb, double lfa, double lfb) {
    return lb - lfb * lb / (lfb - lfa);  // la = 0
}

// Bookkeeping after an attempt: landing/exit solve, accept or reject, state
// update in double.  Returns true when the ray has finished (status set).
__device__ bool lane_end_attempt(Lane &L, const GridDev &g, const FanDev &f, LandState &ls) {
    const double RE = g.R_E;
    const float hf = L.hs;
    ++L.n_att;
    float dy4[6], ef[6];
    bool fin = true;
#pragma unroll
    for (int c = 0; c < 6; ++c) {
        dy4[c] = hf * L.y4[c];
        ef[c] = hf * L.e[c];
        fin = fin && isfinite(dy4[c]);
    }
    if (L.landing) {
        // Illinois regula falsi on the step size: f(h*) = +-(r(step(h*)) - target)
        const double sg = L.exiting ? -1.0 : 1.0;
        const double r_target = L.exiting ? RE + g.top : RE;
        const double fc = sg * ((L.y[0] - r_target) + (double)dy4[0]);
        ++ls.it;
        const double c = (double)L.hs;
        const bool done = fabs(fc) < f.land_tol || ls.it >= 60 || fabs(ls.lb - ls.la) < 1e-9 || !fin;
        if (!done) {
            Bracket B{ls.la, ls.lfa, ls.lb, ls.lfb, ls.side};
            L.hs = (float)bracket_update(B, c, fc);
            ls.la = B.la;
            ls.lfa = B.lfa;
            ls.lb = B.lb;
            ls.lfb = B.lfb;
            ls.side = B.side;
            return !lane_next_attempt(L, f);
        }
        if (!fin) {
            L.status = RT_RAY_NONFINITE;
            return true;
        }
        L.P += c;
        ++L.n_steps;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            L.y[i] += (double)dy4[i];
            two_sum_add(L.k_hi[i], L.k_lo[i], dy4[3 + i]);
        }
        if (L.exiting) L.apo = fmaxf(L.apo, (float)(L.y[0] - RE));
        L.status = L.exiting ? RT_RAY_ESCAPED : RT_RAY_LANDED;
        return true;
    }
    float fac = 1.0f;
    bool accept = true;
    if (f.integrator == RT_RKF45) {
        const float kmag = fsqrt(L.b.k[0] * L.b.k[0] + L.b.k[1] * L.b.k[1] + L.b.k[2] * L.b.k[2]);
        const float err = rkf45_err(L.b.r, L.b.sth, kmag, ef, f.rtol_f, f.atol_f);
        fac = step_factor_f(err);
        accept = err <= 1.0f;
    }
    const float alt_new = L.b.alt + dy4[0];
    const bool lands = alt_new < 0.0f;
    // one branch for everything but an accepted step, so that the usual path
    // below is one block
    if (!(accept && fin) || lands || alt_new > g.top_f) {
        if (!accept) {
            // the nominal step changes only by quantised factors of itself
            L.h = L.h * fac;
            if (L.h < f.hmin_f) {
                L.status = RT_RAY_STEP_UNDERFLOW;
                return true;
            }
            return !lane_next_attempt(L, f);
        }
        if (!fin) {
            L.status = RT_RAY_NONFINITE;
            return true;
        }
        // ground return or exit through the grid top inside this step
        lane_fold(L);
        const double r_new = L.y[0] + (double)dy4[0];
        L.landing = true;
        L.exiting = !lands;
        const double r_target = lands ? RE : RE + g.top;
        const double sg = lands ? 1.0 : -1.0;
        ls.la = 0.0;
        ls.lfa = sg * (L.y[0] - r_target);
        ls.lb = (double)L.hs;
        ls.lfb = sg * (r_new - r_target);
        ls.side = 0;
        ls.it = 0;
        L.hs = (float)bracket_first(ls.lb, ls.lfa, ls.lfb);
        return !lane_next_attempt(L, f);
    }
    if (f.integrator == RT_RKF45)
        L.h = fminf(fmaxf(L.h * (L.at_face ? fminf(1.0f, fac) : fac), f.hmin_f), f.hmax_f);
    L.r_prev = L.b.r;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        two_sum_add(L.inc_hi[i], L.inc_lo[i], dy4[i]);
        two_sum_add(L.k_hi[i], L.k_lo[i], dy4[3 + i]);
    }
    two_sum_add(L.inc_hi[3], L.inc_lo[3], L.hs);
    ++L.n_steps;
    L.apo = fmaxf(L.apo, alt_new);
    L.have_prev = true;
    L.dr_prev = L.k1[0];
    L.h_prev = L.hs;
    L.k1_valid = false;
    if (++L.since_sync >= kResyncSteps) {
        L.since_sync = 0;
        lane_fold(L);
        L.b = base_of(g.lat0, g.lon0, g.inv_dlat, g.inv_dlon, g.R_E, g.alt0, g.inv_dalt, g.far_cells, L.y[0], L.y[1], L.y[2]);
#pragma unroll
        for (int i = 0; i < 3; ++i) L.b.k[i] = L.k_hi[i] + L.k_lo[i];
    } else {
        advance_base(g, L.b, dy4, L.k_hi);
    }
    const bool in_lat = (unsigned)L.b.ia < (unsigned)(g.n_lat - 1) || (L.b.ia == g.n_lat - 1 && L.b.ta == 0.0f);
    const bool in_lon = (unsigned)L.b.ib < (unsigned)(g.n_lon - 1) || (L.b.ib == g.n_lon - 1 && L.b.tb == 0.0f);
    if (L.b.alt >= g.alt0_f && !(in_lat && in_lon)) {
        L.status = RT_RAY_LEFT_GRID;
        return true;
    }
    if (f.has_max_path) {
        lane_fold(L);
        if (L.P >= f.max_path - 1e-6) {
            L.status = RT_RAY_MAX_PATH;
            return true;
        }
    }
    return !lane_next_attempt(L, f);
}

// Loads the Butcher table of the fan's integrator into shared memory; the
// stage loop reads it at a warp-uniform stage index (broadcast reads).  With
// btx, also the transmitter's base of fan f (computed once per block: it is
// double arithmetic, and the persistent kernel would otherwise redo it for
// every lane it refills).
__device__ __forceinline__ void load_tableau(Tableau &T, int integrator, Base32 *btx = nullptr,
                                             const GridDev *g = nullptr, const FanDev *f = nullptr) {
    const Tableau &src = c_tab[integrator == RT_RKF45 ? 1 : 0];
    const float *s = (const float *)&src;
    float *d = (float *)&T;
    for (int i = threadIdx.x; i < (int)(sizeof(Tableau) / sizeof(float)); i += blockDim.x) d[i] = s[i];
    if (btx && threadIdx.x == 0) *btx = tx_base(*g, *f);
    __syncthreads();
}

// Shuffle mask of the G-lane group of this lane.
template <int G>
__device__ __forceinline__ unsigned group_mask(int lane) {
    return G == 1 ? (1u << lane) : (((1u << G) - 1u) << (lane & ~(G - 1)));
}

// One ray per thread group of G lanes; each group loops attempt by attempt
// until its ray ends.  Launch bounds: one lane per ray is throughput-bound
// (three blocks of 128 per SM, <= 168 registers); 2 or 4 lanes per ray serve
// fans whose time is the latency of their slowest ray, and there the
// compiler's own register choice (~200, two blocks per SM) schedules a lone
// warp's stage evaluation faster.
template <int STENCIL, int G, int IP>
__global__ void __launch_bounds__(128, G == 1 ? 3 : 2) trace_mixed_plain_kernel(GridDev g, FanDev f, rt_ray_result *__restrict__ out) {
    constexpr bool FIRST = G > 1;  // see appleton_hartree
    __shared__ Tableau T;
    __shared__ Base32 btx;
    load_tableau(T, f.integrator, &btx, &g, &f);
    const long long tid = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    const long long id = tid / G;
    if (id >= f.n_rays) return;  // whole groups leave together
    const int lane = threadIdx.x & 31, q = lane % G;
    const unsigned gmask = group_mask<G>(lane);
    const long long ray = claim_to_ray(f, id);
    if (ray < 0) return;  // a hole in an ordered plan's claim order: no ray for this group
    Lane L;
    L.active = true;
    lane_begin_ray(L, g, f, ray, btx);
    bool done = lane_launch<STENCIL, G, IP, FIRST>(L, g, f, q, gmask);
    // the landing state stays in registers here (a shared-memory slot per
    // thread would take L1 that the sample gathers use; measured 3 % slower on
    // the 495k-ray batch), unlike in the persistent kernel
    LandState land;
    // bounded: every attempt counts against max_steps, so max_steps + 1 attempts end every ray
    const long long max_att = (long long)f.max_steps + 2;
    for (long long it = 0; it < max_att && !done; ++it) {
        lane_attempt<STENCIL, G, IP, FIRST>(L, g, f, T, q, gmask);
        done = lane_end_attempt(L, g, f, land);
    }
    if (!done) L.status = RT_RAY_MAX_STEPS;
    lane_finish(L, g, f, out, q == 0);
}

// Persistent kernel: resident blocks whose warps claim rays from an atomic
// counter (one atomicAdd per warp), between attempts, where all lanes of the
// warp meet; a warp takes its next rays once all of its current ones ended.
template <int STENCIL, int G, int IP>
__global__ void __launch_bounds__(128, G == 1 ? 3 : 2) trace_mixed_persistent_kernel(GridDev g, FanDev f,
                                                                     rt_ray_result *__restrict__ out,
                                                                     unsigned long long *__restrict__ counter) {
    constexpr bool FIRST = G > 1 || STENCIL != RT_STENCIL_GATHER;  // see appleton_hartree
    __shared__ Tableau T;
    __shared__ Base32 btx;
    __shared__ LandState land[128];
    load_tableau(T, f.integrator, &btx, &g, &f);
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31, q = lane % G;
    const unsigned gmask = group_mask<G>(lane);
    Lane L;
    L.active = false;
    bool exhausted = false;  // warp-uniform
    long long iters = 0;
    const long long n = f.n_rays;
    // bound on the warp's loop iterations: every ray ends within max_steps + 1
    // attempts (+ its launch), and a warp runs at most all n rays
    const long long max_iter = ((long long)f.max_steps + 4) * (n + 32) + 64;
    for (;;) {
        // The warp refills once all its rays have ended, with the next 32 / G
        // consecutive claims: rays launched together from neighbouring
        // elevations cross the same cells at the same time, so their stencil
        // gathers coalesce in L1.  Refilling each lane as soon as its ray ends
        // keeps the lanes busier but puts rays of different ages side by side;
        // on the 495,122-ray batch that took 96 ms against 69 ms for warp-wide
        // refills (a refill at 8 / 16 / 24 idle lanes: 84 / 77 / 78 ms).
        const bool idle_warp = !__any_sync(FULL, L.active);
        if (idle_warp && !exhausted) {
            const int n_take = 32 / G;
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(counter, (unsigned long long)n_take);
            base = __shfl_sync(FULL, base, 0);
            if (base + (unsigned long long)n_take >= (unsigned long long)n) exhausted = true;
            const unsigned long long c = base + (unsigned long long)(lane / G);
            if (c < (unsigned long long)n) {
                L.active = true;
                lane_begin_ray(L, g, f, claim_to_ray(f, (long long)c), btx);
                if (lane_launch<STENCIL, G, IP, FIRST>(L, g, f, q, gmask)) lane_finish(L, g, f, out, q == 0);
            }
        }
        if (!__any_sync(FULL, L.active)) break;
        // the warp's rays to their end; the refill above stays out of this
        // hot loop (with it inside, the loop ran 1-2 % slower on the batch)
        bool over = false;
        do {
            if (++iters > max_iter) {  // defensive bound; never reached for valid inputs
                if (L.active) {
                    L.status = RT_RAY_MAX_STEPS;
                    lane_finish(L, g, f, out, q == 0);
                    L.active = false;
                }
                over = true;
                break;
            }
            if (L.active) {
                lane_attempt<STENCIL, G, IP, FIRST>(L, g, f, T, q, gmask);
                if (lane_end_attempt(L, g, f, land[threadIdx.x])) lane_finish(L, g, f, out, q == 0);
            }
        } while (__any_sync(FULL, L.active));
        if (over) break;
    }
}

// ================================================================ fused fans
// Several small fans on one grid in one launch (the request server's fused
// batches).  Ray i of the launch belongs to fan k with first[k] <= i <
// first[k + 1] (binary search over the n_fans + 1 offsets); its record goes
// to out + first[k] + its index within fan k.  The fans share one integrator
// (the block's Butcher table).  Four lanes per ray, as for any fan too small
// to fill the GPU: the per-ray code is that of the four-lane plain kernel,
// with the fan read from global memory.
template <int STENCIL, int IP>
__global__ void __launch_bounds__(128, 2) trace_mixed_fans_kernel(GridDev g, const FanDev *__restrict__ fans,
                                                                  const long long *__restrict__ first, int n_fans,
                                                                  int integrator, rt_ray_result *__restrict__ out) {
    constexpr int G = 4;
    constexpr bool FIRST = true;  // see appleton_hartree
    __shared__ Tableau T;
    load_tableau(T, integrator);
    const long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / G;
    if (i >= first[n_fans]) return;  // whole groups leave together
    int lo = 0, hi = n_fans - 1;
    while (lo < hi) {  // largest k with first[k] <= i
        const int mid = (lo + hi + 1) >> 1;
        if (first[mid] <= i) lo = mid;
        else hi = mid - 1;
    }
    const FanDev &f = fans[lo];
    const int lane = threadIdx.x & 31, q = lane % G;
    const unsigned gmask = group_mask<G>(lane);
    Lane L;
    L.active = true;
    lane_begin_ray(L, g, f, claim_to_ray(f, i - first[lo]), tx_base(g, f));
    bool done = lane_launch<STENCIL, G, IP, FIRST>(L, g, f, q, gmask);
    LandState land;
    const long long max_att = (long long)f.max_steps + 2;
    for (long long it = 0; it < max_att && !done; ++it) {
        lane_attempt<STENCIL, G, IP, FIRST>(L, g, f, T, q, gmask);
        done = lane_end_attempt(L, g, f, land);
    }
    if (!done) L.status = RT_RAY_MAX_STEPS;
    lane_finish(L, g, f, out + first[lo], q == 0);
}

// ================================================================ ionogram
// One warp per (frequency, mode) trace: lanes scan neighbouring elevation
// pairs; the pairs whose landed rays bracket the receiver distance d_rx emit
// an ionogram point, appended through one atomicAdd per warp (ballot +
// popc rank: warp-level compaction).  Branch numbers are assigned after the
// host sorts the points.
__global__ void ionogram_kernel(const rt_ray_result *__restrict__ res, const double *__restrict__ freq,
                                const double *__restrict__ el, int n_freq, int n_modes, int mode0, int n_el,
                                double d_rx, rt_ionogram_point *__restrict__ out, unsigned long long cap,
                                unsigned long long *__restrict__ count) {
    const unsigned FULL = 0xffffffffu;
    const int lane = threadIdx.x & 31;
    const long long trace = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / 32;
    if (trace >= (long long)n_freq * n_modes) return;  // whole warps leave together
    const int fi = (int)(trace / n_modes), mi = (int)(trace % n_modes);
    const rt_ray_result *row = res + trace * n_el;  // the fan has one azimuth
    for (int j0 = 0; j0 < n_el - 1; j0 += 32) {
        const int j = j0 + lane;
        bool hit = false;
        rt_ionogram_point p;
        if (j < n_el - 1) {
            const rt_ray_result a = row[j], b = row[j + 1];
            if (a.status == RT_RAY_LANDED && b.status == RT_RAY_LANDED) {
                const double fa = a.ground_range_km - d_rx, fb = b.ground_range_km - d_rx;
                if ((fa < 0.0 && fb >= 0.0) || (fa >= 0.0 && fb < 0.0)) {
                    const double t = fa / (fa - fb);
                    p.freq_mhz = freq[fi];
                    p.group_path_km = a.group_path_km + t * (b.group_path_km - a.group_path_km);
                    p.el_deg = el[j] + t * (el[j + 1] - el[j]);
                    p.ground_range_km = d_rx;
                    p.mode = (mi == 0) ? mode0 : -1;
                    p.branch = 0;
                    hit = true;
                }
            }
        }
        const unsigned m = __ballot_sync(FULL, hit);
        if (m) {
            unsigned long long base = 0;
            if (lane == 0) base = atomicAdd(count, (unsigned long long)__popc(m));
            base = __shfl_sync(FULL, base, 0);
            if (hit) {
                const unsigned long long idx = base + __popc(m & ((1u << lane) - 1u));
                if (idx < cap) out[idx] = p;
            }
        }
    }
}

cudaError_t launch_ionogram(const rt_ray_result *res, const double *freq, const double *el, int n_freq, int n_modes,
                            int mode0, int n_el, double d_rx, rt_ionogram_point *out, unsigned long long cap,
                            unsigned long long *count, cudaStream_t st) {
    const long long threads = (long long)n_freq * n_modes * 32;
    if (threads == 0) return cudaSuccess;
    ionogram_kernel<<<(unsigned)((threads + 127) / 128), 128, 0, st>>>(res, freq, el, n_freq, n_modes, mode0, n_el,
                                                                      d_rx, out, cap, count);
    return cudaGetLastError();
}

// ============================================================== diagnostics
// The mixed path's right-hand side (the FP64 path's: eval_rhs_fp64_kernel).
__global__ void eval_rhs_kernel(GridDev g, const double *__restrict__ ys, double *__restrict__ dys,
                                double *__restrict__ mu2s, double freq_mhz, int mode, int stencil, long long n) {
    const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
    if (i >= n) return;
    double y[6];
#pragma unroll
    for (int c = 0; c < 6; ++c) y[c] = ys[i * 6 + c];
    const RayPhys<float> rp = make_phys<float>(g, freq_mhz * 1e6, mode);
    Base32 b;
    base_from_state(g, y, b);
    float d[6] = {0, 0, 0, 0, 0, 0}, dyf[6], m2;
    if (g.interp == 1) {
        if (stencil == RT_STENCIL_TABLE) rhs_mixed<RT_STENCIL_TABLE, 1, 1, true>(g, rp, b, d, dyf, &m2, 0, 0u);
        else if (stencil == RT_STENCIL_GATHER) rhs_mixed<RT_STENCIL_GATHER, 1, 1, true>(g, rp, b, d, dyf, &m2, 0, 0u);
        else rhs_mixed<RT_STENCIL_QUAD, 1, 1, true>(g, rp, b, d, dyf, &m2, 0, 0u);
    } else {
        if (stencil == RT_STENCIL_TABLE) rhs_mixed<RT_STENCIL_TABLE, 1, 0, true>(g, rp, b, d, dyf, &m2, 0, 0u);
        else if (stencil == RT_STENCIL_GATHER) rhs_mixed<RT_STENCIL_GATHER, 1, 0, true>(g, rp, b, d, dyf, &m2, 0, 0u);
        else rhs_mixed<RT_STENCIL_QUAD, 1, 0, true>(g, rp, b, d, dyf, &m2, 0, 0u);
    }
#pragma unroll
    for (int c = 0; c < 6; ++c) dys[i * 6 + c] = dyf[c];
    mu2s[i] = m2;
}

// ================================================================ launchers
// Packs Butcher coefficients A[s][t], B4[s], E[s] (s = 0..5) into the
// two-float4-per-stage layout of Tableau.
static void pack_tableau(Tableau &T, const float A[6][5], const float B4[6], const float E[6], int ns) {
    for (int s = 0; s < 6; ++s) {
        T.lo[s] = make_float4(A[s][0], A[s][1], A[s][2], A[s][3]);
        T.hi[s] = make_float4(A[s][4], B4[s], E[s], 0.0f);
    }
    T.ns = ns;
}

static void fill_tableaus(Tableau tab[2]) {
    float A[6][5], B4[6], E[6];
    auto clear = [&]() {
        for (int s = 0; s < 6; ++s) {
            for (int u = 0; u < 5; ++u) A[s][u] = 0.0f;
            B4[s] = E[s] = 0.0f;
        }
    };
    // classic RK4: a21 = a32 = 1/2, a43 = 1; b = (1, 2, 2, 1)/6; A[s][t] = a[s+1+t][s]
    clear();
    double a4[4][4] = {{0}};
    a4[1][0] = 0.5;
    a4[2][1] = 0.5;
    a4[3][2] = 1.0;
    const double b4[4] = {1.0 / 6.0, 1.0 / 3.0, 1.0 / 3.0, 1.0 / 6.0};
    for (int s = 0; s < 4; ++s) {
        for (int u = 0; u < 5; ++u) A[s][u] = (s + 1 + u < 4) ? (float)a4[s + 1 + u][s] : 0.0f;
        B4[s] = (float)b4[s];
    }
    pack_tableau(tab[0], A, B4, E, 4);
    // Fehlberg 4(5)
    clear();
    double a[6][6] = {{0}};
    a[1][0] = 1.0 / 4.0;
    a[2][0] = 3.0 / 32.0;
    a[2][1] = 9.0 / 32.0;
    a[3][0] = 1932.0 / 2197.0;
    a[3][1] = -7200.0 / 2197.0;
    a[3][2] = 7296.0 / 2197.0;
    a[4][0] = 439.0 / 216.0;
    a[4][1] = -8.0;
    a[4][2] = 3680.0 / 513.0;
    a[4][3] = -845.0 / 4104.0;
    a[5][0] = -8.0 / 27.0;
    a[5][1] = 2.0;
    a[5][2] = -3544.0 / 2565.0;
    a[5][3] = 1859.0 / 4104.0;
    a[5][4] = -11.0 / 40.0;
    const double b4f[6] = {25.0 / 216.0, 0.0, 1408.0 / 2565.0, 2197.0 / 4104.0, -1.0 / 5.0, 0.0};
    const double b5f[6] = {16.0 / 135.0, 0.0, 6656.0 / 12825.0, 28561.0 / 56430.0, -9.0 / 50.0, 2.0 / 55.0};
    for (int s = 0; s < 6; ++s) {
        for (int u = 0; u < 5; ++u) A[s][u] = (s + 1 + u < 6) ? (float)a[s + 1 + u][s] : 0.0f;
        B4[s] = (float)b4f[s];
        E[s] = (float)(b5f[s] - b4f[s]);
    }
    pack_tableau(tab[1], A, B4, E, 6);
}

cudaError_t upload_tableaus() {
    Tableau tab[2];
    fill_tableaus(tab);
    return cudaMemcpyToSymbol(c_tab, tab, sizeof(tab));
}

template <int STENCIL, int G, int IP>
static cudaError_t launch_mixed_gi(const GridDev &g, const FanDev &f, rt_ray_result *out,
                                   unsigned long long *counter, const LaunchPlan &lp, cudaStream_t st) {
    if (lp.kernel == RT_KERNEL_PERSISTENT) {
        trace_mixed_persistent_kernel<STENCIL, G, IP><<<lp.blocks, lp.threads, 0, st>>>(g, f, out, counter);
    } else {
        // GATHER's samples come from the quad layout, which every grid holds: the
        // same values and records, 16 vector loads a stage instead of 64 (495,122
        // rays 77.4 -> 67.0 ms, C2 fan 21.5 -> 17.2 ms at one lane per ray, 12.6 ->
        // 11.3 at four).  The fused launches do the same.
        constexpr int S = STENCIL == RT_STENCIL_GATHER ? RT_STENCIL_QUAD : STENCIL;
        const long long blocks = (f.n_rays * G + lp.threads - 1) / lp.threads;
        if (lp.started) {
            cudaLaunchConfig_t lc = {};
            lc.gridDim = dim3((unsigned)blocks);
            lc.blockDim = dim3((unsigned)lp.threads);
            lc.dynamicSmemBytes = (size_t)lp.smem;
            lc.stream = st;
            cudaLaunchAttribute at[1];
            at[0].id = cudaLaunchAttributeLaunchCompletionEvent;
            at[0].val.launchCompletionEvent.event = lp.started;
            at[0].val.launchCompletionEvent.flags = 0;
            lc.attrs = at;
            lc.numAttrs = 1;
            return cudaLaunchKernelEx(&lc, trace_mixed_plain_kernel<S, G, IP>, g, f, out);
        }
        trace_mixed_plain_kernel<S, G, IP><<<(unsigned)blocks, lp.threads, (size_t)lp.smem, st>>>(g, f, out);
    }
    return cudaGetLastError();
}

template <int STENCIL, int G, int IP>
static cudaError_t exclusive_smem_gi(int *bytes) {
    int dev = 0, per_sm = 0, per_block = 0, reserved = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&per_block, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
    cudaFuncAttributes fa;
    if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, trace_mixed_plain_kernel<STENCIL, G, IP>);
    if (e != cudaSuccess) return e;
    // the block's static + dynamic shared memory plus the per-block
    // reservation take the SM's whole capacity
    const int dyn = std::min(per_block, per_sm - reserved) - (int)fa.sharedSizeBytes;
    if (dyn <= 0) return cudaErrorInvalidValue;
    e = cudaFuncSetAttribute(trace_mixed_plain_kernel<STENCIL, G, IP>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             dyn);
    if (e == cudaSuccess) *bytes = dyn;
    return e;
}

template <int STENCIL, int G>
static cudaError_t exclusive_smem_g(int interp, int *bytes) {
    return interp == 1 ? exclusive_smem_gi<STENCIL, G, 1>(bytes) : exclusive_smem_gi<STENCIL, G, 0>(bytes);
}

template <int STENCIL>
static cudaError_t exclusive_smem_s(int lanes, int interp, int *bytes) {
    switch (lanes) {
        case 2: return exclusive_smem_g<STENCIL, 2>(interp, bytes);
        case 4: return exclusive_smem_g<STENCIL, 4>(interp, bytes);
        default: return exclusive_smem_g<STENCIL, 1>(interp, bytes);
    }
}

cudaError_t plain_exclusive_smem(const LaunchPlan &lp, int interp, int *bytes) {
    switch (lp.stencil) {
        case RT_STENCIL_TABLE: return exclusive_smem_s<RT_STENCIL_TABLE>(lp.lanes, interp, bytes);
        default: return exclusive_smem_s<RT_STENCIL_QUAD>(lp.lanes, interp, bytes);
    }
}

template <int STENCIL, int G>
static cudaError_t launch_mixed_g(const GridDev &g, const FanDev &f, rt_ray_result *out,
                                  unsigned long long *counter, const LaunchPlan &lp, cudaStream_t st) {
    return g.interp == 1 ? launch_mixed_gi<STENCIL, G, 1>(g, f, out, counter, lp, st)
                         : launch_mixed_gi<STENCIL, G, 0>(g, f, out, counter, lp, st);
}

template <int STENCIL>
static cudaError_t launch_mixed(const GridDev &g, const FanDev &f, rt_ray_result *out,
                                unsigned long long *counter, const LaunchPlan &lp, cudaStream_t st) {
    switch (lp.lanes) {
        case 2: return launch_mixed_g<STENCIL, 2>(g, f, out, counter, lp, st);
        case 4: return launch_mixed_g<STENCIL, 4>(g, f, out, counter, lp, st);
        default: return launch_mixed_g<STENCIL, 1>(g, f, out, counter, lp, st);
    }
}

cudaError_t launch_trace_only(const GridDev &g, const FanDev &f, rt_ray_result *out, unsigned long long *counter,
                              const LaunchPlan &lp, cudaStream_t st) {
    if (f.n_rays == 0) return cudaSuccess;
    if (f.precision == RT_FP64) return launch_trace_fp64(g, f, lp.fp64_rays, out, st);
    switch (lp.stencil) {
        case RT_STENCIL_GATHER: return launch_mixed<RT_STENCIL_GATHER>(g, f, out, counter, lp, st);
        case RT_STENCIL_TABLE: return launch_mixed<RT_STENCIL_TABLE>(g, f, out, counter, lp, st);
        default: return launch_mixed<RT_STENCIL_QUAD>(g, f, out, counter, lp, st);
    }
}

cudaError_t launch_finish(const GridDev &g, const FanDev &f, rt_ray_result *out, long long n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int threads = 128;
    finish_records_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0, st>>>(g.R_E, f, out, n);
    return cudaGetLastError();
}

cudaError_t launch_trace(const GridDev &g, const FanDev &f, rt_ray_result *out, unsigned long long *counter,
                         const LaunchPlan &lp, cudaStream_t st) {
    const cudaError_t e = launch_trace_only(g, f, out, counter, lp, st);
    if (e != cudaSuccess) return e;
    return launch_finish(g, f, out, f.n_rays, st);
}

template <int STENCIL>
static cudaError_t launch_fans_s(const GridDev &g, const FanDev *fans, const long long *first, int n_fans,
                                 long long n_total, int integrator, rt_ray_result *out, int threads, cudaStream_t st) {
    const unsigned blocks = (unsigned)((n_total * 4 + threads - 1) / threads);  // four lanes per ray
    if (g.interp == 1)
        trace_mixed_fans_kernel<STENCIL, 1><<<blocks, threads, 0, st>>>(g, fans, first, n_fans, integrator, out);
    else
        trace_mixed_fans_kernel<STENCIL, 0><<<blocks, threads, 0, st>>>(g, fans, first, n_fans, integrator, out);
    return cudaGetLastError();
}

cudaError_t launch_trace_fans(const GridDev &g, const FanDev *fans, const long long *first, int n_fans,
                              long long n_total, int integrator, rt_ray_result *out, const LaunchPlan &lp,
                              cudaStream_t st) {
    if (n_total == 0) return cudaSuccess;
    cudaError_t e;
    switch (lp.stencil) {
        case RT_STENCIL_TABLE:
            e = launch_fans_s<RT_STENCIL_TABLE>(g, fans, first, n_fans, n_total, integrator, out, lp.threads, st);
            break;
        default:
            e = launch_fans_s<RT_STENCIL_QUAD>(g, fans, first, n_fans, n_total, integrator, out, lp.threads, st);
    }
    if (e != cudaSuccess) return e;
    const int threads = 128;
    finish_fans_records_kernel<<<(unsigned)((n_total + threads - 1) / threads), threads, 0, st>>>(g.R_E, fans, first,
                                                                                                 n_fans, out);
    return cudaGetLastError();
}

template <int STENCIL>
static cudaError_t occupancy_s(int lanes, int threads, int *blocks_per_sm) {
    switch (lanes) {
        case 2:
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                blocks_per_sm, trace_mixed_persistent_kernel<STENCIL, 2, 0>, threads, 0);
        case 4:
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                blocks_per_sm, trace_mixed_persistent_kernel<STENCIL, 4, 0>, threads, 0);
        default:
            return cudaOccupancyMaxActiveBlocksPerMultiprocessor(
                blocks_per_sm, trace_mixed_persistent_kernel<STENCIL, 1, 0>, threads, 0);
    }
}

cudaError_t persistent_occupancy(int stencil, int lanes, int threads, int *blocks_per_sm) {
    switch (stencil) {
        case RT_STENCIL_GATHER: return occupancy_s<RT_STENCIL_GATHER>(lanes, threads, blocks_per_sm);
        case RT_STENCIL_TABLE: return occupancy_s<RT_STENCIL_TABLE>(lanes, threads, blocks_per_sm);
        default: return occupancy_s<RT_STENCIL_QUAD>(lanes, threads, blocks_per_sm);
    }
}

cudaError_t launch_eval_rhs(const GridDev &g, const double *ys, double *dys, double *mu2s, double freq_mhz, int mode,
                            int stencil, long long n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int threads = 128;
    eval_rhs_kernel<<<(unsigned)((n + threads - 1) / threads), threads, 0, st>>>(g, ys, dys, mu2s, freq_mhz, mode,
                                                                               stencil, n);
    return cudaGetLastError();
}

}  // namespace rtgd
