// rtgd_fp64.cuh -- the all-double stage evaluation (one thread per state) and
// the grid-coordinate helpers of the FP64 path.
#pragma once

#include "rtgd_device.cuh"

namespace rtgd {

// Rare cases are out of line here and below: inlined, the compiler predicates
// them, and a predicated-off FP64 instruction still occupies the warp for its
// 64 cycles.
static __device__ __noinline__ double wrap360_rare(double x) { return x - 360.0 * floor(x / 360.0); }

// x - 360 floor(x / 360): the longitude offset wrapped to [0, 360).  The two
// ranges a ray's longitude lies in are told apart by the high word (a double
// division costs a warp ~10 FP64 instructions, an integer compare none):
// for 0 <= x < 360 the quotient stays below 1 after rounding, so the floor is
// 0; for -360 < x < 0 it is -1.
__device__ __forceinline__ double wrap360(double x) {
    const unsigned hi = (unsigned)__double2hiint(x);
    if (hi < 0x40768000u) return x;  // [0, 360)
    if (hi - 0x80100000u < 0xC0768000u - 0x80100000u) return x + 360.0;  // (-360, 0), normal numbers
    return wrap360_rare(x);
}

// max(|a|, sb |b|, sc |c|) with infinities or NaN among them: fmax, which
// ignores a NaN.  A negative scale (sin(theta) beyond a pole) takes its term out
// of the maximum, as in the step control's bit compare of finite values.
__host__ __device__ __noinline__ inline double max3_rare(double a, double sb, double b, double sc, double c) {
    return fmax(fabs(a), fmax(sb * fabs(b), sc * fabs(c)));
}

// Grid coordinate of a position along one axis (0 latitude, 1 longitude, 2
// altitude): (90 - deg(theta) - lat0) / dlat, (deg(phi) - lon0 wrapped) / dlon,
// (r - R_E - alt0) / dalt.  One form for the three axes, chosen by selects, so
// that lanes with different axes share the FP64 instructions; the fused
// multiply-add is spelt out so that every caller rounds alike.
__device__ __forceinline__ double grid_coord64(const GridDev &g, int axis, double y0, double y1, double y2) {
    const double p = axis == 0 ? -y1 : axis == 1 ? y2 : y0;
    const double c = axis == 0 ? 90.0 : axis == 1 ? -g.lon0 : -g.R_E;
    double x = fma(p, axis == 2 ? 1.0 : kRad2Deg, c);
    if (axis == 1) x = wrap360(x);
    return (x - (axis == 0 ? g.lat0 : axis == 1 ? 0.0 : g.alt0)) *
           (axis == 0 ? g.inv_dlat : axis == 1 ? g.inv_dlon : g.inv_dalt);
}

// Cell index and local coordinate of grid coordinate x; false outside
// [0, n-1] (and for NaN), then cell 0 at t = 0.  The integer part comes from
// the bits: floor, the two range compares and the two conversions are FP64
// instructions (64 cycles of a warp each), the shifts are not.  t = x - floor(x)
// is the one FP64 operation left.
__device__ __forceinline__ bool cell64(double x, int n, int &i, double &t) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(x);
    const unsigned hi = (unsigned)(b >> 32);
    const bool range = hi < 0x41D00000u || b == 0x8000000000000000ull;  // [0, 2^30) or -0
    const int e = range ? (int)((hi >> 20) & 0x7ffu) - 1023 : -1;       // exponent, < 30
    const int sh = 52 - (e < 0 ? 0 : e);
    const unsigned long long frac = (1ull << sh) - 1;
    const unsigned long long m = (b & 0xfffffffffffffull) | 0x10000000000000ull;
    const int fi = e < 0 ? 0 : (int)(m >> sh);
    const double fl = e < 0 ? 0.0 : __longlong_as_double((long long)(b & ~frac));
    const bool whole = e < 0 ? (b << 1) == 0 : (b & frac) == 0;
    const bool last = fi == n - 1 && whole;  // the last node: cell n-2 at t = 1
    const bool ok = range && (fi < n - 1 || last);
    const double tr = x - fl;
    i = ok ? (last ? n - 2 : fi) : 0;
    t = ok ? (last ? 1.0 : tr) : 0.0;
    return ok;
}

// Field terms, Appleton-Hartree and ray equations of one stage in double
// (field_terms and ray_rhs with the roundings spelt out: which of two
// products a compiler fuses depends on the surrounding code, and the records
// must not).  Sequential form: one thread evaluates everything.
__device__ __forceinline__ void tail64(const RayPhys<double> &rp, const StageIn<double> &s, double dy[6],
                                       double *mu2) {
    const double kr = s.k[0], kt = s.k[1], kp = s.k[2], X = s.X;
    const double kk = fma(kp, kp, fma(kr, kr, __dmul_rn(kt, kt)));
    const double ir = __drcp_rn(s.r);
    double H[3], K[3], G;
    if (rp.iso) {
        // no field: mu^2 = 1 - X, so H_x = grad(X)/2, H_k = k, G = -|k|^2 - X
        if (mu2) *mu2 = __dadd_rn(1.0, -X);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            H[j] = __dmul_rn(0.5, s.dX[j]);
            K[j] = s.k[j];
        }
        G = __dadd_rn(-kk, -X);
    } else {
        const double mx = rp.m[0], my = rp.m[1], mz = rp.m[2];
        const double mr = fma(mz, s.cth, fma(__dmul_rn(my, s.sth), s.sph, __dmul_rn(__dmul_rn(mx, s.sth), s.cph)));
        const double mt = fma(-mz, s.sth, fma(__dmul_rn(my, s.cth), s.sph, __dmul_rn(__dmul_rn(mx, s.cth), s.cph)));
        const double mp = fma(my, s.cph, -__dmul_rn(mx, s.sph));
        const double q = __dmul_rn(rp.R_E, ir);
        const double A = __dmul_rn(__dmul_rn(__dmul_rn(rp.ab0, q), q), q);
        const double A2 = __dmul_rn(A, A);
        const double Y[3] = {__dmul_rn(__dmul_rn(-2.0, A), mr), __dmul_rn(A, mt), __dmul_rn(A, mp)};
        const double YY = __dmul_rn(A2, fma(__dmul_rn(3.0, mr), mr, 1.0));
        const double kY = fma(kp, Y[2], fma(kr, Y[0], __dmul_rn(kt, Y[1])));
        const double smp = __dmul_rn(s.sth, mp), A6mr = __dmul_rn(__dmul_rn(6.0, A2), mr);
        const double gYY[3] = {__dmul_rn(__dmul_rn(-6.0, YY), ir), __dmul_rn(A6mr, mt), __dmul_rn(A6mr, smp)};
        const double m2kr = __dmul_rn(-2.0, kr);
        const double gkY[3] = {__dmul_rn(__dmul_rn(-3.0, kY), ir),
                               __dmul_rn(A, fma(m2kr, mt, -__dmul_rn(kt, mr))),
                               __dmul_rn(A, fma(-kp, fma(s.sth, mr, __dmul_rn(s.cth, mt)),
                                                fma(m2kr, smp, __dmul_rn(__dmul_rn(kt, s.cth), mp))))};
        const double ikk = __drcp_rn(kk);
        const double L = __dmul_rn(__dmul_rn(kY, kY), ikk);
        double T = __dadd_rn(YY, -L);
        if (T < 0.0) T = 0.0;
        const double u = __dadd_rn(1.0, -X);
        const double L4u = __dmul_rn(__dmul_rn(4.0, L), u), L4uu = __dmul_rn(L4u, u);
        const double S = sqrt(fma(T, T, L4uu));
        double FX, FL, FT;
        if (rp.mode > 0) {
            const double L2 = __dmul_rn(2.0, L), L2u = __dmul_rn(L2, u);
            const double W = __dadd_rn(S, T), V = __dadd_rn(W, L2u), SW = __dmul_rn(S, W);
            const double m = __drcp_rn(__dmul_rn(SW, V));
            const double iS = __dmul_rn(__dmul_rn(W, V), m), iW = __dmul_rn(__dmul_rn(S, V), m);
            const double iopg = __dmul_rn(__dmul_rn(SW, W), m);
            const double gg = __dmul_rn(L2u, iW), opg = __dadd_rn(1.0, gg);
            const double gX = __dmul_rn(__dmul_rn(__dmul_rn(L2, fma(L4uu, iS, -W)), iW), iW);
            const double gL = fma(__dmul_rn(2.0, u), iW,
                                  -__dmul_rn(__dmul_rn(__dmul_rn(__dmul_rn(L4uu, u), iS), iW), iW));
            const double gT = __dmul_rn(-gg, iS);
            const double i2 = __dmul_rn(iopg, iopg);
            if (mu2) *mu2 = __dadd_rn(1.0, -__dmul_rn(X, iopg));
            FX = __dmul_rn(fma(X, gX, -opg), i2);
            FL = __dmul_rn(__dmul_rn(X, gL), i2);
            FT = __dmul_rn(__dmul_rn(X, gT), i2);
        } else {
            const double D = __dadd_rn(fma(2.0, u, -T), -S);
            const double m = __drcp_rn(__dmul_rn(S, D));
            const double iS = __dmul_rn(D, m), iD = __dmul_rn(S, m), iD2 = __dmul_rn(iD, iD);
            const double N = __dmul_rn(__dmul_rn(2.0, X), u);
            const double SL = __dmul_rn(__dmul_rn(__dmul_rn(2.0, u), u), iS);
            if (mu2) *mu2 = __dadd_rn(1.0, -__dmul_rn(N, iD));
            FX = __dmul_rn(fma(N, fma(L4u, iS, -2.0), -__dmul_rn(fma(-4.0, X, 2.0), D)), iD2);
            FL = __dmul_rn(__dmul_rn(N, -SL), iD2);
            FT = __dmul_rn(__dmul_rn(N, fma(-T, iS, -1.0)), iD2);
        }
        const double cL = __dmul_rn(__dadd_rn(FL, -FT), __dmul_rn(__dmul_rn(2.0, kY), ikk));
        const double kYn = __dmul_rn(kY, ikk), hf = __dmul_rn(0.5, cL);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            H[j] = __dmul_rn(-0.5, fma(cL, gkY[j], fma(FX, s.dX[j], __dmul_rn(FT, gYY[j]))));
            K[j] = fma(-hf, fma(-kYn, s.k[j], Y[j]), s.k[j]);
        }
        G = fma(T, FT, fma(L, FL, fma(X, FX, -kk)));
    }
    const double iG = __drcp_rn(G), irs = __dmul_rn(ir, __drcp_rn(s.sth));
    const double dr = __dmul_rn(-K[0], iG), dt = __dmul_rn(__dmul_rn(-K[1], iG), ir);
    const double dp = __dmul_rn(__dmul_rn(-K[2], iG), irs);
    const double kps = __dmul_rn(kp, s.sth), kprc = __dmul_rn(__dmul_rn(kp, s.r), s.cth);
    dy[0] = dr;
    dy[1] = dt;
    dy[2] = dp;
    dy[3] = fma(kps, dp, fma(H[0], iG, __dmul_rn(kt, dt)));
    dy[4] = __dmul_rn(fma(kprc, dp, fma(H[1], iG, -__dmul_rn(kt, dr))), ir);
    dy[5] = __dmul_rn(fma(-kprc, dt, fma(H[2], iG, -__dmul_rn(kps, dr))), irs);
}

// Polynomials of the one-dimensional weights (Appendix A; Eq. 7 for
// Catmull-Rom) as Horner coefficients, highest power first: kinds 0 and 1
// are the weights of nodes j-1 and j, kinds 2 and 3 their derivatives.
//   kind 0: t p4(t), kind 1: 1 + t^2 p3(t), kind 2: p4(t), kind 3: t p3(t)
// with p4 of all five coefficients and p3 of the first four.
static __constant__ double c_poly[2][4][5] = {
    {{1.0 / 6.0, -5.0 / 12.0, -1.0 / 6.0, 11.0 / 12.0, -0.5},
     {-0.5, 1.25, 0.5, -2.25, 0.0},
     {5.0 / 6.0, -5.0 / 3.0, -0.5, 11.0 / 6.0, -0.5},
     {-2.5, 5.0, 1.5, -4.5, 0.0}},
    {{0.0, 0.0, -0.5, 1.0, -0.5},
     {0.0, 0.0, 1.5, -2.5, 0.0},
     {0.0, 0.0, -1.5, 2.0, -0.5},
     {0.0, 0.0, 4.5, -5.0, 0.0}}};

// One altitude row's sum, and the same against the derivative weights.
__device__ __forceinline__ double row64(double u0, double u1, double u2, double u3, const double *w) {
    return fma(u3, w[3], fma(u2, w[2], fma(u0, w[0], __dmul_rn(u1, w[1]))));
}

// Weights of one axis at local coordinate t, all four polynomials in one
// thread: the operations of density64, in its order.
__device__ __forceinline__ void weights64(const double (*c)[5], double t, double w[4], double d[4]) {
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        const double s = side ? 1.0 - t : t;
        double p[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            p[k] = fma(s, fma(s, fma(s, c[k][0], c[k][1]), c[k][2]), c[k][3]);
            if (k == 0 || k == 2) p[k] = fma(s, p[k], c[k][4]);
        }
        const double outer = __dmul_rn(p[0], s), inner = __dadd_rn(1.0, __dmul_rn(__dmul_rn(s, s), p[1]));
        const double dinner = __dmul_rn(s, p[3]);
        w[side ? 3 : 0] = outer;
        w[side ? 2 : 1] = inner;
        d[side ? 3 : 0] = side ? -p[2] : p[2];
        d[side ? 2 : 1] = side ? -dinner : dinner;
    }
}

// dy/dP' at state y, all in double, by one thread: Ne and its gradient from
// the FP64 padded grid (Eq. 13), then the dipole, Appleton-Hartree and Eq. 1.
// The same operations in the same order as the lane groups' evaluation.
// sth_out receives sin(theta).
__device__ __forceinline__ void rhs64(const GridDev &g, const RayPhys<double> &rp, const double y[6], double dy[6],
                                      double *mu2, double *sth_out = nullptr) {
    StageIn<double> s;
    s.r = y[0];
    sincos(y[1], &s.sth, &s.cth);
    sincos(y[2], &s.sph, &s.cph);
    s.k[0] = y[3];
    s.k[1] = y[4];
    s.k[2] = y[5];
    if (sth_out) *sth_out = s.sth;
    int ia, ib, ic;
    double ta, tb, tc;
    s.X = 0.0;
    s.dX[0] = s.dX[1] = s.dX[2] = 0.0;
    const bool in_a = cell64(grid_coord64(g, 0, y[0], y[1], y[2]), g.n_lat, ia, ta);
    const bool in_b = cell64(grid_coord64(g, 1, y[0], y[1], y[2]), g.n_lon, ib, tb);
    const bool in_c = cell64(grid_coord64(g, 2, y[0], y[1], y[2]), g.n_alt, ic, tc);
    if (in_a && in_b && in_c) {
        const double (*c)[5] = c_poly[g.interp == 1 ? 1 : 0];
        double wa[4], da[4], wb[4], db[4], wc[4], dc[4], out[4] = {0.0, 0.0, 0.0, 0.0};
        weights64(c, ta, wa, da);
        weights64(c, tb, wb, db);
        weights64(c, tc, wc, dc);
        const long long sj = g.p_alt, si = (long long)g.p_lon * g.p_alt;
        // padded index of node (ia-1, ib-1, ic-1) is (ia, ib, ic)
        const double *base = g.pad64 + (long long)ia * si + (long long)ib * sj + ic;
#pragma unroll
        for (int a = 0; a < 4; ++a) {
            double sv = 0.0, sd = 0.0, sc = 0.0;
#pragma unroll
            for (int b = 0; b < 4; ++b) {
                const double *p = base + a * si + b * sj;
                const double u0 = __ldg(p), u1 = __ldg(p + 1), u2 = __ldg(p + 2), u3 = __ldg(p + 3);
                const double v = row64(u0, u1, u2, u3, wc), dv = row64(u0, u1, u2, u3, dc);
                sv = fma(v, wb[b], sv);
                sd = fma(v, db[b], sd);
                sc = fma(dv, wb[b], sc);
            }
            out[0] = fma(sv, wa[a], out[0]);
            out[1] = fma(sv, da[a], out[1]);
            out[2] = fma(sd, wa[a], out[2]);
            out[3] = fma(sc, wa[a], out[3]);
        }
        s.X = rp.xfac * out[0];
        s.dX[0] = rp.xfac * out[3] * g.inv_dalt;
        s.dX[1] = -rp.xfac * out[1] * g.inv_dlat * kRad2Deg;
        s.dX[2] = rp.xfac * out[2] * g.inv_dlon * kRad2Deg;
    }
    tail64(rp, s, dy, mu2);
}

}  // namespace rtgd
