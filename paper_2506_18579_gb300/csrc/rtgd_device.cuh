// rtgd_device.cuh -- device-side building blocks of the RTM-GD tracer.
//
// What the mixed path's stage evaluation needs (the FP64 path's, with its
// roundings spelt out, is in rtgd_fp64.cuh):
//   - p = 3 Galerkin-Difference weights and their derivatives (Appendix A),
//   - the 4x4x4 tensor contraction of Eq. 13 giving Ne and its gradient,
//   - the centred dipole field and its Jacobian in local spherical components,
//   - Appleton-Hartree (Eq. 3) with hand-derived partial derivatives,
//   - the Hamiltonian partials (Eq. 2) and the ray equations (Eq. 1a-1f).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "rtgd.h"

namespace rtgd {

constexpr double kPi = 3.14159265358979323846;
constexpr double kRad2Deg = 180.0 / kPi;
constexpr double kDeg2Rad = kPi / 180.0;
// f_N^2 = 80.6 Ne (Hz^2, Ne in m^-3), so X = f_N^2 / f^2 (Sec. II-A).
constexpr double kPlasmaHz2PerM3 = 80.6;
// f_H = e B / (2 pi m_e) in Hz per tesla, so Y = f_H / f (Sec. II-A).
constexpr double kGyroHzPerTesla = 2.7992489872e10;

// Device view of a grid.  Node (i, j, k), i in [0, n_lat), sits at padded
// index (i+1, j+1, k+1) of the ghost-padded arrays.
struct GridDev {
    int n_lat, n_lon, n_alt;
    int p_lon, p_alt;                // padded sizes n_lon + 2, n_alt + 2
    int q_alt;                       // n_alt - 1 cells per (lat, lon) row of the quad layout
    double lat0, lon0, alt0;
    double inv_dlat, inv_dlon, inv_dalt;
    double R_E, top;                 // earth radius; top = alt0 + (n_alt - 1) dalt
    double b0;                       // dipole strength (0: isotropic)
    double m[3];                     // unit vector to the geomagnetic north pole
    float sa, sb, sc;                // d(grid coord)/d(theta, phi, r): -rad2deg/dlat, rad2deg/dlon, 1/dalt
    float R_Ef, mf[3];               // float copies of R_E and m
    float top_f, alt0_f;             // top and alt0 as floats
    // Mixed path: base cells are kept within +-far_cells, and a stage offset of
    // more than far_stage cells makes its derivatives NaN.  2^21 and no limit; on
    // an axis of more than 2^20 nodes 2^30 (no axis has more: 4 nodes on each of
    // the others, 2^34 in all) and the offsets that stage_cell resolves.
    int far_cells;
    float far_stage;
    int iso;                         // no field (b0 == 0)
    int interp;                      // 0: Galerkin-Difference p=3, 1: Catmull-Rom (comparison)
    const double *pad64;             // (n_lat+2)(n_lon+2)(n_alt+2) doubles
    const float *pad32;              // same, rounded to float
    const float4 *quad;              // (n_lat+2)(n_lon+2)(n_alt-1): samples k-1..k+2 of cell k
    const float4 *table;             // (n_lat-1)(n_lon-1)(n_alt-1) cells x 16 float4 (64 samples)
};

// --------------------------------------------------------------------------
// GD p = 3 weights (Appendix A).  For a point at local coordinate t in [0, 1]
// of the cell [x_j, x_{j+1}], the weight of node j-1 is the printed piece
// psi_1 (in powers of t), of node j the piece psi_0, of node j+1 psi_{-1} and
// of node j+2 psi_{-2}.  The global basis function is even, so the last two
// are the first two mirrored: w_{j+1}(t) = w_j(1-t), w_{j+2}(t) = w_{j-1}(1-t).
// half_weights gives those of nodes j-1 and j and their derivatives at s = t;
// at s = 1 - t, derivatives negated, they are those of nodes j+2 and j+1.  IP = 1:
// Catmull-Rom (Eq. 7), w_{-1} = (-s^3 + 2s^2 - s)/2, w_0 = (3s^3 - 5s^2 + 2)/2.
template <int IP>
__device__ __forceinline__ void half_weights(float s, float &wm1, float &w0, float &dm1, float &d0) {
    if (IP == 1) {
        wm1 = s * (-0.5f + s * (1.0f - s * 0.5f));
        w0 = 1.0f + s * s * (-2.5f + s * 1.5f);
        dm1 = -0.5f + s * (2.0f - s * 1.5f);
        d0 = s * (-5.0f + s * 4.5f);
    } else {
        wm1 = s * (-0.5f + s * (float(11.0 / 12.0) +
                                s * (float(-1.0 / 6.0) + s * (float(-5.0 / 12.0) + s * float(1.0 / 6.0)))));
        w0 = 1.0f + s * s * (-2.25f + s * (0.5f + s * (1.25f - s * 0.5f)));
        dm1 = -0.5f + s * (float(11.0 / 6.0) + s * (-0.5f + s * (float(-5.0 / 3.0) + s * float(5.0 / 6.0))));
        d0 = s * (-4.5f + s * (1.5f + s * (5.0f - s * 2.5f)));
    }
}

// All four weights of one axis, interpolant fixed at compile time: nodes j-1,
// j from half_weights(t), nodes j+2, j+1 from its mirror half_weights(1 - t).
template <int IP>
__device__ __forceinline__ void axis_weights(float t, float w[4], float d[4]) {
    float wp2, wp1, dp2, dp1;
    half_weights<IP>(t, w[0], w[1], d[0], d[1]);
    half_weights<IP>(1.0f - t, wp2, wp1, dp2, dp1);
    w[2] = wp1;
    w[3] = wp2;
    d[2] = -dp1;
    d[3] = -dp2;
}

// Eq. 13 contraction of one row of 4 altitude samples.  PACK:
// packed FMAs on the sample pairs (u0, u1) and (u2, u3) against the weight
// pairs, then one addition per sum -- four instructions fewer per two sums
// and a shorter chain; the sum is formed in another order (pairs first).
template <bool PACK>
__device__ __forceinline__ void row4(float u0, float u1, float u2, float u3, const float wc[4], const float dc[4],
                                     float &v, float &dv) {
    v = u0 * wc[0] + u1 * wc[1] + u2 * wc[2] + u3 * wc[3];
    dv = u0 * dc[0] + u1 * dc[1] + u2 * dc[2] + u3 * dc[3];
}

template <>
__device__ __forceinline__ void row4<true>(float u0, float u1, float u2, float u3, const float wc[4],
                                           const float dc[4], float &v, float &dv) {
    const float2 a = make_float2(u0, u1), b = make_float2(u2, u3);
    const float2 p = __ffma2_rn(b, make_float2(wc[2], wc[3]), __fmul2_rn(a, make_float2(wc[0], wc[1])));
    const float2 q = __ffma2_rn(b, make_float2(dc[2], dc[3]), __fmul2_rn(a, make_float2(dc[0], dc[1])));
    v = p.x + p.y;
    dv = q.x + q.y;
}

// Accumulates the (a, b) row into the lon/lat partial sums.
__device__ __forceinline__ void acc_row(float v, float dv, float wb, float db, float &s, float &sb, float &sc) {
    s += v * wb;
    sb += v * db;
    sc += dv * wb;
}

// Partial sums {Ne - REF, dNe/dxa, dNe/dxb, dNe/dxc} (per-cell units) over
// the rows a = A0 .. A0+NA-1 (all b) of the 16 rows of 4 altitude samples;
// wa/da hold the NA lat-weights of those rows.  ROW(a, b, u0..u3) loads row
// (a, b).  The samples are contracted relative to REF (Ne = REF + sum (u -
// REF) w, the weights summing to 1 and their derivatives to 0), so that in
// float the sums do not cancel against the magnitude of Ne; the caller adds
// REF back (after combining partial sums, when the rows are split).  PACK
// selects the packed altitude rows (row4).
#define RTGD_CONTRACT(PACK, ROW, REF, A0, NA, wa, da, wb, db, wc, dc, out)        \
    do {                                                                          \
        float n_ = 0.0f, na_ = 0.0f, nb_ = 0.0f, nc_ = 0.0f;                      \
        _Pragma("unroll") for (int a_ = 0; a_ < (NA); ++a_) {                     \
            float s_ = 0.0f, sb_ = 0.0f, sc_ = 0.0f;                              \
            _Pragma("unroll") for (int b_ = 0; b_ < 4; ++b_) {                    \
                float u0_, u1_, u2_, u3_, v_, dv_;                                \
                ROW((A0) + a_, b_, u0_, u1_, u2_, u3_);                           \
                u0_ -= (REF);                                                     \
                u1_ -= (REF);                                                     \
                u2_ -= (REF);                                                     \
                u3_ -= (REF);                                                     \
                row4<(PACK)>(u0_, u1_, u2_, u3_, wc, dc, v_, dv_);                \
                acc_row(v_, dv_, wb[b_], db[b_], s_, sb_, sc_);                   \
            }                                                                     \
            n_ += s_ * wa[a_];                                                    \
            na_ += s_ * da[a_];                                                   \
            nb_ += sb_ * wa[a_];                                                  \
            nc_ += sc_ * wa[a_];                                                  \
        }                                                                         \
        out[0] = n_;                                                              \
        out[1] = na_;                                                             \
        out[2] = nb_;                                                             \
        out[3] = nc_;                                                             \
    } while (0)

// 1/x: the fast reciprocal (MUFU.RCP, within 2 ulp), which is ample for the
// mixed path's tolerance.
__device__ __forceinline__ float recip(float x) { return __fdividef(1.0f, x); }

// sqrt: x * rsqrt(x) (MUFU.RSQ, a few ulp, no special-case branch), 0 for x <= 0.
__device__ __forceinline__ float fsqrt(float x) { return x > 0.0f ? x * rsqrtf(x) : 0.0f; }

// a / b: the fast division (MUFU.RCP based, 2 ulp, no special-case branch) for
// the step-control arithmetic.
__device__ __forceinline__ float fdiv(float a, float b) { return __fdividef(a, b); }

// --------------------------------------------------------------------------
// Physics at one stage: everything after the interpolation.
template <typename R>
struct StageIn {
    R r, sth, cth, sph, cph;  // position (km, sin/cos of colatitude and longitude)
    R k[3];                   // wave vector (r, theta, phi components), units of omega/c
    R X;                      // f_N^2 / f^2
    R dX[3];                  // dX/dr, dX/dtheta, dX/dphi
};

// Per-ray physics constants in the precision of the stage arithmetic.
template <typename R>
struct RayPhys {
    R xfac;   // 80.6 / f^2: X = xfac * Ne
    R ab0;    // (kGyroHzPerTesla / f) * B0: |Y| at the magnetic equator on the ground
    R R_E;
    R m[3];   // unit vector to the geomagnetic north pole
    bool iso; // no field
    int mode; // +1 ordinary, -1 extraordinary
};

template <typename R>
__device__ __forceinline__ RayPhys<R> make_phys(const GridDev &g, double f_hz, int mode) {
    RayPhys<R> p;
    p.xfac = R(kPlasmaHz2PerM3 / (f_hz * f_hz));
    p.ab0 = R(kGyroHzPerTesla / f_hz * g.b0);
    p.R_E = R(g.R_E);
    p.m[0] = R(g.m[0]);
    p.m[1] = R(g.m[1]);
    p.m[2] = R(g.m[2]);
    p.iso = g.iso != 0;
    p.mode = mode;
    return p;
}

// Appleton-Hartree mu^2(X, L = Y_L^2, T = Y_T^2) (Eq. 3) and its partials.
// Ordinary wave (upper sign): the printed denominator 2u - T + S (u = 1 - X,
// S = sqrt(T^2 + 4 L u^2)) is rewritten with S - T = 4 L u^2 / (S + T), which
// gives mu^2 = 1 - X / (1 + g), g = 2 L u / (S + T): the same function, free
// of the 0/0 at X = 1.  Extraordinary wave: the printed form.
// FIRST: which product of S's sum is fused, T^2 or (4 L u) u.  Spelt out because
// the compiler's choice has gone either way with the code around it, and the
// records must not: each kernel states the form its records have.
template <bool FIRST>
__device__ __forceinline__ void appleton_hartree(float X, float L, float T, int mode, float &mu2, float &FX, float &FL,
                                                 float &FT) {
    const float u = 1.0f - X;
    const float S = fsqrt(FIRST ? __fmaf_rn(T, T, 4.0f * L * u * u) : __fmaf_rn(4.0f * L * u, u, T * T));
    if (mode > 0) {
        // one reciprocal gives 1/S, 1/W and 1/(1 + g) = W/V with V = W + 2 L u
        const float W = S + T;
        const float V = W + 2.0f * L * u;
        const float SW = S * W;
        const float m = recip(SW * V);
        const float iS = W * V * m;
        const float iW = S * V * m;
        const float g = 2.0f * L * u * iW;
        const float opg = 1.0f + g;
        const float iopg = SW * W * m;
        const float gX = 2.0f * L * (4.0f * L * u * u * iS - W) * iW * iW;
        const float gL = 2.0f * u * iW - 4.0f * L * u * u * u * iS * iW * iW;
        const float gT = -g * iS;
        mu2 = 1.0f - X * iopg;
        const float i2 = iopg * iopg;
        FX = (X * gX - opg) * i2;
        FL = X * gL * i2;
        FT = X * gT * i2;
    } else {
        const float D = 2.0f * u - T - S;
        const float m = recip(S * D);  // 1/S and 1/D from one reciprocal
        const float iS = D * m;
        const float iD = S * m;
        const float N = 2.0f * X * u;
        const float SX = -4.0f * L * u * iS;
        const float SL = 2.0f * u * u * iS;
        const float ST = T * iS;
        const float iD2 = iD * iD;
        mu2 = 1.0f - N * iD;
        FX = (N * (-2.0f - SX) - (2.0f - 4.0f * X) * D) * iD2;
        FL = N * (-SL) * iD2;
        FT = N * (-1.0f - ST) * iD2;
    }
}

// Field terms of one stage that do not depend on the electron density: the
// centred dipole Y = A (-2 m_r, m_th, m_ph) with A = ab0 (R_E / r)^3, |Y|^2,
// k . Y, and the partials of |Y|^2 and of k . Y along (r, theta, phi).  From
// dm_r/dth = m_th, dm_th/dth = -m_r, dm_ph/dth = 0, dm_r/dph = sin m_ph,
// dm_th/dph = cos m_ph, dm_ph/dph = -(sin m_r + cos m_th):
//   dY/dr = -3 Y / r,  dY/dth = A (-2 m_th, -m_r, 0),
//   dY/dph = A (-2 sin m_ph, cos m_ph, -(sin m_r + cos m_th)),
// so d|Y|^2/dx = 2 Y . dY/dx = (-6 |Y|^2 / r, 6 A^2 m_r m_th, 6 A^2 m_r sin m_ph).
struct FieldTerms {
    float Y[3];     // Y (units of the wave frequency)
    float YY, kY;   // |Y|^2, k . Y
    float gYY[3];   // d|Y|^2 / d(r, theta, phi)
    float gkY[3];   // d(k . Y) / d(r, theta, phi) at fixed k
    float ir;       // 1 / r
};

__device__ __forceinline__ FieldTerms field_terms(const RayPhys<float> &rp, const StageIn<float> &s) {
    FieldTerms F;
    const float kr = s.k[0], kt = s.k[1], kp = s.k[2];
    const float mx = rp.m[0], my = rp.m[1], mz = rp.m[2];
    const float mr = mx * s.sth * s.cph + my * s.sth * s.sph + mz * s.cth;
    const float mt = mx * s.cth * s.cph + my * s.cth * s.sph - mz * s.sth;
    const float mp = -mx * s.sph + my * s.cph;
    F.ir = recip(s.r);
    const float q = rp.R_E * F.ir;
    const float A = rp.ab0 * q * q * q;
    F.Y[0] = -2.0f * A * mr;
    F.Y[1] = A * mt;
    F.Y[2] = A * mp;
    const float A2 = A * A;
    F.YY = A2 * (1.0f + 3.0f * mr * mr);  // m is a unit vector
    F.kY = kr * F.Y[0] + kt * F.Y[1] + kp * F.Y[2];
    const float smp = s.sth * mp;
    const float A6mr = 6.0f * A2 * mr;
    F.gYY[0] = -6.0f * F.YY * F.ir;
    F.gYY[1] = A6mr * mt;
    F.gYY[2] = A6mr * smp;
    F.gkY[0] = -3.0f * F.kY * F.ir;
    F.gkY[1] = A * (-2.0f * kr * mt - kt * mr);
    F.gkY[2] = A * (-2.0f * kr * smp + kt * s.cth * mp - kp * (s.sth * mr + s.cth * mt));
    return F;
}

// Hamiltonian H = (|k|^2 - mu^2)/2 (Eq. 2, k in units of omega/c) and the ray
// equations (Eq. 1a-1f, with k_phi sin(theta) dphi/dP' in the k_r equation as
// the canonical momentum p_phi = r sin(theta) k_phi requires).  With G =
// omega dH/domega at fixed k:
//   dr/dP' = -H_kr/G, dtheta/dP' = -H_kth/(r G), dphi/dP' = -H_kph/(r sin G),
//   dk_r/dP'   = H_r/G + k_th dtheta + k_ph sin dphi,
//   dk_th/dP'  = (H_th/G - k_th dr + k_ph r cos dphi) / r,
//   dk_ph/dP'  = (H_ph/G - k_ph sin dr - k_ph r cos dtheta) / (r sin).
// F holds the field terms of the same stage; mu2_out receives mu^2.
template <bool FIRST>
__device__ __forceinline__ void ray_rhs(const RayPhys<float> &rp, const StageIn<float> &s, const FieldTerms &F,
                                        float dy[6], float *mu2_out) {
    const float kr = s.k[0], kt = s.k[1], kp = s.k[2];
    const float kk = kr * kr + kt * kt + kp * kp;
    float Hr, Ht, Hp, Hk0, Hk1, Hk2, G, mu2;
    if (rp.iso) {
        // no field: mu^2 = 1 - X, so H_x = grad(X)/2, H_k = k, G = -|k|^2 - X
        mu2 = 1.0f - s.X;
        Hr = 0.5f * s.dX[0];
        Ht = 0.5f * s.dX[1];
        Hp = 0.5f * s.dX[2];
        Hk0 = kr;
        Hk1 = kt;
        Hk2 = kp;
        G = -kk - s.X;
    } else {
        const float ikk = recip(kk);
        const float L = F.kY * F.kY * ikk;
        float T = F.YY - L;
        if (T < 0.0f) T = 0.0f;
        float Fm, FX, FL, FT;
        appleton_hartree<FIRST>(s.X, L, T, rp.mode, Fm, FX, FL, FT);
        mu2 = Fm;
        // mu^2 = F(X, L, T) with T = Y^2 - L: d/dY^2 = F_T, d/dL|_{Y^2} = F_L - F_T;
        // dL/dx at fixed k = c2 d(k . Y)/dx with c2 = 2 kY / |k|^2
        const float FYL = FL - FT;
        const float c2 = 2.0f * F.kY * ikk;
        const float cL = FYL * c2;
        Hr = -0.5f * (FX * s.dX[0] + FT * F.gYY[0] + cL * F.gkY[0]);
        Ht = -0.5f * (FX * s.dX[1] + FT * F.gYY[1] + cL * F.gkY[1]);
        Hp = -0.5f * (FX * s.dX[2] + FT * F.gYY[2] + cL * F.gkY[2]);
        // dL/dk_i = (2 kY / |k|^2) (Y_i - (kY / |k|^2) k_i)
        const float kYn = F.kY * ikk;
        const float hf = 0.5f * cL;
        Hk0 = kr - hf * (F.Y[0] - kYn * kr);
        Hk1 = kt - hf * (F.Y[1] - kYn * kt);
        Hk2 = kp - hf * (F.Y[2] - kYn * kp);
        // omega dH/domega: X, L and T all scale as omega^-2, |k|^2 as omega^-2
        G = -kk + s.X * FX + L * FL + T * FT;
    }
    const float iG = recip(G);
    const float ir = F.ir;
    const float irs = ir * recip(s.sth);
    const float dr = -Hk0 * iG;
    const float dt = -Hk1 * iG * ir;
    const float dp = -Hk2 * iG * irs;
    dy[0] = dr;
    dy[1] = dt;
    dy[2] = dp;
    dy[3] = Hr * iG + kt * dt + kp * s.sth * dp;
    dy[4] = (Ht * iG - kt * dr + kp * s.r * s.cth * dp) * ir;
    dy[5] = (Hp * iG - kp * s.sth * dr - kp * s.r * s.cth * dt) * irs;
    if (mu2_out) *mu2_out = mu2;
}

}  // namespace rtgd
