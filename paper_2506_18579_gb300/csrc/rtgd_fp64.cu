// rtgd_fp64.cu -- the all-FP64 tracer.
//
// What bounds it: GB300 issues FP64 at 1/64 of the FP32 rate.  Measured: one
// FP64 instruction occupies a warp for 64 cycles whether 1 or 32 of its lanes
// are active and however many independent ones follow, and four or more warps
// of an SM share a rate of one per 19 cycles.  So lanes are free and warp
// instructions are not: with one ray per lane an evaluation took ~770 FP64
// warp instructions (23.8 us) however few rays the warp still held.
//
// Layout: a block's first warp holds up to eight rays.  While n of them are
// in flight, each is carried by a group of G = 32 / 2^ceil(log2 n) lanes,
// which share the evaluation's independent parts (the polynomials of the
// weights, the 16 sample rows, the state components, the coordinates, the
// divisions, the r/theta/phi components of the field and the ray equations):
// ~250 FP64 instructions at G = 4, ~175 at G = 32.  As rays end the warp
// regroups, so that its last ray runs on all 32 lanes.  The block's second
// warp takes the part of an evaluation that need not wait for the rest (Duo):
// the electron density, ~90 of the 250 instructions at G = 4, ~25 of the 175 at
// G = 32 and there the field's gradients (~15) too.  A ray's arithmetic is the
// same operations in the same order for every G (only the warp and lane that
// perform them change), so its record depends neither on G nor on its warp
// mates.  Ray states live in shared memory (slots), so that regrouping moves
// no data.  The host starts a warp with as many rays as fill the GPU
// (fp64_rays_per_warp); a fan that fills it many times over starts with 32 rays
// a warp, one per lane, and goes over to groups once 16 are left, eight of those
// at a time: 20.2 FP64 warp instructions per evaluation and ray over a 63,432-ray
// scan, step control and launch included, where eight rays a warp take 38.9 on
// the 24,840-ray fan.  Measured with one thread per ray / lane groups / and
// the second warp: 16 rays RK4 without a field 133 / 32 / 24.9 ms, one RKF45
// ray 42.5 / 16.1 / 11.9 ms (one evaluation 21.2 / 8.0 / 5.9 us), 522 rays - /
// 19.3 / 16.6 ms, 3,232 rays - / 49.0 / 38.4 ms, the 24,840-ray fan 418 / 172 /
// 147 ms; 495,122 rays 2,026 ms, 2,551 from eight rays a warp and 1,535 from 32.
#include <cuda_runtime.h>
#include <math.h>

#include "rtgd_fan.cuh"
#include "rtgd_fp64.cuh"

namespace rtgd {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Shared memory of a block, in doubles.  Slot (one per ray): state, k1,
// sin(theta) at the state, then the scalars below.
enum {
    kY = 0, kK1 = 6, kSth = 12, kP, kH, kHs, kApo, kRPrev, kDrPrev, kHPrev, kLa, kLfa, kLb, kLfb, kXfac, kAb0,
    kInts,             // 4 doubles: 8 ints (kId ...)
    kSlot = kInts + 5
};
enum { kId = 0, kMode, kSteps, kAtt, kEv, kFlags, kSide, kIt };
enum { kK1Valid = 1, kHavePrev = 2, kLands = 4, kExits = 8 };
// Scratch (one per group): derivatives k2..k6, stage state / new state, error
// estimate, in-cell coordinates t and 1 - t and cells of the three axes, the 24 weights,
// the altitude, longitude and latitude sums.
enum { cK = 0, cT = 30, cE = 36, cFrac = 42, cCell = 48 /* 3 ints */, cW = 50, cV = 74, cS = 106, cO = 118, cGroup = 123 };
// One lane per ray: the derivatives, the stage state and the error estimate only.
enum { cLane = 43 };
static_assert(kSlot % 2 == 1 && cGroup % 2 == 1 && cLane % 2 == 1 && cLane >= cFrac, "odd strides spread the groups over the banks");
constexpr int kGroups = 8;    // groups of a warp at most (G = 4)
constexpr int kBlocksPerSm = 6;
constexpr int kWideRays = 32;  // rays that a warp of the wide kernel starts with
// One lane per ray until this few are left.  Twice eight of 16 cost the pipe
// about what 16 lanes of their own do, and take a cluster of long rays to its end
// sooner.  Measured at 8 / 16 / 20 / 24: 24,840 rays 148 / 152 / 160 / 162 ms,
// 100,434 rays 564 / 483 / 490 / 493 ms, 248,442 rays 775 / 788 / 797 / 824 ms.
constexpr int kWideLeft = 16;
constexpr int kPoly = 4 * 5, kPow2 = 20;  // tables at the start of the shared memory

__device__ __noinline__ double div_rare(double x, double c) { return x / c; }

// x / c for a constant c with rc = 1/c correctly rounded: one Newton
// correction of x rc gives the correctly rounded quotient (Markstein's
// theorem), 3 FP64 instructions instead of ~10.  Non-finite and tiny x take
// the division.
__device__ __forceinline__ double div_const(double x, double c, double rc) {
    const double q = x * rc;
    const double r = fma(-c, q, x);
    const double d = fma(r, rc, q);
    const unsigned hi = (unsigned)__double2hiint(x) & 0x7fffffffu;
    if ((hi >> 20) - 128u >= 1800u && hi != 0) return div_rare(x, c);
    return d;
}

__device__ __forceinline__ bool finite64(double x) {
    return ((unsigned)__double2hiint(x) & 0x7ff00000u) != 0x7ff00000u;
}

// max of two numbers at least one of which is >= +0 (not NaN): the order of
// such doubles is the order of their bits as signed integers.
__device__ __forceinline__ double max_bits(double a, double b) {
    return __double_as_longlong(a) > __double_as_longlong(b) ? a : b;
}

// Stage s (1..5) of Fehlberg 4(5): y + h * (its combination of k1..ks), one
// component.  The fused multiply-adds are spelt out, here and below, because
// the branches otherwise decide which products the compiler fuses.
__device__ __forceinline__ double rkf45_stage(int s, double y, double h, const double *k1, const double *k, int c) {
    const double k1c = k1[c];
    if (s == 1) return fma(h, k1c * 0.25, y);
    const double k2c = k[c];
    if (s == 2) return fma(h, fma(3.0 / 32.0, k1c, __dmul_rn(9.0 / 32.0, k2c)), y);
    const double k3c = k[6 + c];
    if (s == 3)
        return fma(h, fma(7296.0 / 2197.0, k3c, fma(1932.0 / 2197.0, k1c, -__dmul_rn(7200.0 / 2197.0, k2c))), y);
    const double k4c = k[12 + c];
    if (s == 4)
        return fma(h, fma(-845.0 / 4104.0, k4c,
                          fma(3680.0 / 513.0, k3c, fma(439.0 / 216.0, k1c, -__dmul_rn(8.0, k2c)))), y);
    const double k5c = k[18 + c];
    return fma(h, fma(-11.0 / 40.0, k5c,
                      fma(1859.0 / 4104.0, k4c,
                          fma(-3544.0 / 2565.0, k3c, fma(-8.0 / 27.0, k1c, __dmul_rn(2.0, k2c))))), y);
}

// Fourth-order solution and local error estimate (5th - 4th order) of one
// component, the latter as h sum((b5_i - b4_i) k_i) so that it keeps full
// relative precision (y5 - y4 would cancel against r ~ 6371 km).
__device__ __forceinline__ void rkf45_end(double y, double h, const double *k1, const double *k, int c, double &yn,
                                          double &e) {
    const double k1c = k1[c], k3c = k[6 + c], k4c = k[12 + c], k5c = k[18 + c], k6c = k[24 + c];
    yn = __dadd_rn(y, __dmul_rn(h, __dadd_rn(fma(2197.0 / 4104.0, k4c,
                                                 fma(25.0 / 216.0, k1c, __dmul_rn(1408.0 / 2565.0, k3c))),
                                             -div_const(k5c, 5.0, 1.0 / 5.0))));
    e = h * fma(2.0 / 55.0, k6c,
                fma(1.0 / 5.0 - 9.0 / 50.0, k5c,
                    fma(28561.0 / 56430.0 - 2197.0 / 4104.0, k4c,
                        fma(16.0 / 135.0 - 25.0 / 216.0, k1c, __dmul_rn(6656.0 / 12825.0 - 1408.0 / 2565.0, k3c)))));
}

// Step-size factor: 0.9 err^(-1/5) limited to [0.2, 5], rounded down to a
// power of 2^(1/4), so step sizes change through discrete decisions only and
// round-off in err cannot feed back into the step sequence.  The exponent
// floor(4 log2 of it) is taken from a float logarithm wherever that is not
// within 1e-3 of an integer (its error is below 1e-5); only the rest pays for
// the double pow and logarithm (~150 FP64 instructions).
__device__ __forceinline__ double step_factor64(double err, const double *pow2q) {
    if (err == 0.0) return pow2q[19];  // 5 rounds down to 2^(9/4)
    const float e = (float)err;
    if (e > 1e-30f && e < 1e30f) {
        const float l = -0.608012374f - 0.8f * __log2f(e);  // 4 log2(0.9 err^-0.2)
        const float fl = floorf(l), d = l - fl;
        if (d > 1e-3f && d < 0.999f) {
            const int k = (int)fl;
            return pow2q[(k < -10 ? -10 : (k > 9 ? 9 : k)) + 10];
        }
    }
    const double fac = fmin(5.0, fmax(0.2, 0.9 * pow(err, -0.2)));
    return exp2(floor(4.0 * log2(fac)) * 0.25);
}

// Peak of the cubic Hermite fit of r(s), s in [0,1], through (r0, h d0) and
// (r1, h d1) with d0 > 0 >= d1 (zero of p'(s) by bisection).
__device__ __noinline__ double hermite_peak(double r0, double r1, double d0, double d1, double h) {
    const double m0 = h * d0, m1 = h * d1;
    const double A = 2.0 * (r0 - r1) + m0 + m1;
    const double B = 3.0 * (r1 - r0) - 2.0 * m0 - m1;
    double lo = 0.0, hi = 1.0;
    for (int it = 0; it < 60; ++it) {
        const double mid = 0.5 * (lo + hi);
        const double dp = m0 + 2.0 * B * mid + 3.0 * A * mid * mid;
        if (dp > 0.0) lo = mid;
        else hi = mid;
    }
    const double s = 0.5 * (lo + hi);
    return r0 + m0 * s + B * s * s + A * s * s * s;
}

// Group path to the face of one axis that the ray reaches next at coordinate
// x with rate v (coordinate per km), HUGE_VAL if there is none.  Faces are
// where the C1 interpolant's second derivatives jump (the right-hand side is
// only C0 there), the grid's outer faces included.  Adaptive steps end just
// past such a face instead of straddling it.
__device__ __forceinline__ double face_axis64(double x, double v, int n) {
    const bool up = v > 0.0, down = v < 0.0;
    double F = up ? floor(x) + 1.0 : ceil(x) - 1.0;
    if (up && F < 0.0) F = 0.0;
    if (!up && F > (double)(n - 1)) F = (double)(n - 1);
    const bool ok = (up && F <= (double)(n - 1)) || (down && F >= 0.0);
    const double d = (F - x) / v;
    return ok ? d : HUGE_VAL;
}

// Two warps on one ray.  A lone warp issues one FP64 instruction per 64 cycles,
// four warps of an SM about 3.4, so a block has a second warp that takes
// independent parts of every evaluation: X and its derivatives for all of the
// first warp's groups, and once a single ray is left (32 lanes) the gradients
// of its field.  Producer / consumer pairs of named barriers: one warp signals
// (arrives), the other waits.
struct Duo {
    enum { kStart = 1, kDensity = 2, kField = 3, kGradients = 4 };  // barrier numbers (0 is __syncthreads)
    enum { dXfac = 0, dM = 1, dA = 4, dA2, dYY, dKY, dIr, dIkk, dSth, dCth, dGYY, dGKY = dGYY + 3, dKV = dGKY + 3,
           dKYn = dKV + 3, dC2, dSize };
    double *D;          // shared: what the warps hand over
    // shared: lanes per ray G (+ kState: at the rays' states instead of their
    // stage states), 0 to stop; for the single ray of G = 32 instead kSingle times
    // 1 + the offset of its (stage) state in the block's shared memory
    int *request;
    int *slot_of;       // shared: the slot of each group's ray
    const double *sm;   // the block's shared memory
    enum { kState = 64, kSingle = 256 };

    static __device__ __forceinline__ void signal(int barrier) {
        __syncwarp();
        __threadfence_block();
        asm volatile("bar.arrive %0, 64;" ::"r"(barrier) : "memory");
    }
    static __device__ __forceinline__ void wait(int barrier) {
        __syncwarp();
        asm volatile("bar.sync %0, 64;" ::"r"(barrier) : "memory");
    }
    __device__ __forceinline__ void start(int what, int lane) {
        if (lane == 0) *(volatile int *)request = what;
        signal(kStart);
    }
};

// Component j of the gradients of |Y|^2 and of k . Y (at fixed k):
// gYY: (-6 YY) ir, ((6 A2) mr) mt, ((6 A2) mr) smp;
// gkY: (-3 kY) ir, A ((-2 kr) mt - kt mr), A ((-2 kr) smp + (kt cth) mp - kp (sth mr + cth mt)).
__device__ __forceinline__ void field_gradients(int j, double kr, double kt, double kp, double mr, double mt, double mj,
                                                double A, double A2, double YY, double kY, double ir, double sth,
                                                double cth, double &gYY, double &gkY) {
    const double smp = __dmul_rn(sth, mj);  // j = 2
    gYY = __dmul_rn(__dmul_rn(__dmul_rn(j == 0 ? -6.0 : 6.0, j == 0 ? YY : A2), j == 0 ? ir : mr),
                    j == 0 ? 1.0 : j == 1 ? mt : smp);
    const double m2kr = __dmul_rn(-2.0, kr), ktc = __dmul_rn(kt, cth);
    const double inner = fma(sth, mr, __dmul_rn(cth, mt));
    double e = __dmul_rn(j == 0 ? -3.0 : j == 1 ? -kt : ktc, j == 0 ? kY : j == 1 ? mr : mj);
    e = fma(j == 0 ? 1.0 : m2kr, j == 0 ? -0.0 : j == 1 ? mt : smp, e);
    e = fma(j < 2 ? 1.0 : -kp, j < 2 ? -0.0 : inner, e);
    gkY = __dmul_rn(j == 0 ? ir : A, e);
}

// tail64 by a quad of lanes: lane j = 0, 1, 2 carries the r, theta, phi
// component (lane 3 repeats lane 2), and the independent quotients and the
// partials FX, FL, FT of Appleton-Hartree stand side by side in lanes 0-2.
// The same operations in the same order as tail64 (a lane that has nothing to
// do in a shared instruction multiplies by 1 or adds -0, which changes
// nothing): ~110 FP64 instructions instead of ~175, without a field ~30
// instead of ~45.  d and dk receive dy[j] and dy[3 + j].  X and its derivatives
// come from the second warp in C[cO ..] (see density64); GRAD: so do the
// gradients of the field.
template <bool GRAD>
__device__ __forceinline__ void tail64_quad(const RayPhys<double> &rp, const StageIn<double> &s, const double *C, int j,
                                            int q, Duo &duo, double &d, double &dk) {
    auto from = [](double v, int lane) { return __shfl_sync(kFull, v, lane, 4); };
    const double kr = s.k[0], kt = s.k[1], kp = s.k[2];
    const double kj = j == 0 ? kr : j == 1 ? kt : kp;
    const double kk = fma(kp, kp, fma(kr, kr, __dmul_rn(kt, kt)));
    const double rc = __drcp_rn(j == 0 ? s.r : j == 1 ? s.sth : kk);
    const double ir = from(rc, 0), ist = from(rc, 1);
    double H, K, G, kv = 0.0;
    if (rp.iso) {
        Duo::wait(Duo::kDensity);
        const double X = C[cO], dXj = C[cO + (j == 0 ? 3 : j)];
        H = __dmul_rn(0.5, dXj);
        K = kj;
        G = __dadd_rn(-kk, -X);
    } else {
        const double ikk = from(rc, 2);
        // m_j: (my S) sph + (mx S) cph + mz C, and my cph - mx sph
        const double sj = j == 0 ? s.sth : j == 1 ? s.cth : 1.0;
        const double px = __dmul_rn(rp.m[0], sj), py = __dmul_rn(rp.m[1], sj);
        const double mj = fma(j == 0 ? rp.m[2] : j == 1 ? -rp.m[2] : 1.0, j == 0 ? s.cth : j == 1 ? s.sth : -0.0,
                              fma(py, j < 2 ? s.sph : s.cph, __dmul_rn(px, j < 2 ? s.cph : -s.sph)));
        const double rr = __dmul_rn(rp.R_E, ir);
        const double A = __dmul_rn(__dmul_rn(__dmul_rn(rp.ab0, rr), rr), rr);
        const double A2 = __dmul_rn(A, A);
        const double Yj = __dmul_rn(__dmul_rn(j == 0 ? -2.0 : 1.0, A), mj);
        const double mr = from(mj, 0), mt = from(mj, 1);
        const double kY = fma(kp, from(Yj, 2), fma(kr, from(Yj, 0), __dmul_rn(kt, from(Yj, 1))));
        const double YY = __dmul_rn(A2, fma(__dmul_rn(3.0, mr), mr, 1.0));
        double gYY, gkY;
        if (GRAD) {
            if (q < 3) duo.D[Duo::dM + q] = mj;
            if (q == 0) {
                duo.D[Duo::dA] = A;
                duo.D[Duo::dA2] = A2;
                duo.D[Duo::dYY] = YY;
                duo.D[Duo::dKY] = kY;
                duo.D[Duo::dIr] = ir;
                duo.D[Duo::dIkk] = ikk;
                duo.D[Duo::dSth] = s.sth;
                duo.D[Duo::dCth] = s.cth;
            }
            Duo::signal(Duo::kField);
        } else {
            field_gradients(j, kr, kt, kp, mr, mt, mj, A, A2, YY, kY, ir, s.sth, s.cth, gYY, gkY);
        }
        const double L = __dmul_rn(__dmul_rn(kY, kY), ikk);
        double T = __dadd_rn(YY, -L);
        if (T < 0.0) T = 0.0;
        Duo::wait(Duo::kDensity);
        const double X = C[cO], dXj = C[cO + (j == 0 ? 3 : j)];
        const double u = __dadd_rn(1.0, -X);
        const double L4u = __dmul_rn(__dmul_rn(4.0, L), u), L4uu = __dmul_rn(L4u, u);
        const double S = sqrt(fma(T, T, L4uu));
        // FX, FL, FT in lanes 0, 1, 2.  Groups of one warp may carry rays of both
        // modes: the branches hold no shuffle (a warp-wide shuffle in a divergent
        // branch would wait for lanes that never come).
        const bool ord = rp.mode > 0;
        const double u2 = __dmul_rn(2.0, u);
        double W = 0.0, V = 0.0, D = 0.0, den;
        if (ord) {
            W = __dadd_rn(S, T);
            V = __dadd_rn(W, __dmul_rn(__dmul_rn(2.0, L), u));
            den = __dmul_rn(__dmul_rn(S, W), V);
        } else {
            D = __dadd_rn(fma(2.0, u, -T), -S);
            den = __dmul_rn(S, D);
        }
        const double m = __drcp_rn(den);
        // ordinary: iS = (W V) m, iW = (S V) m, 1/(1 + g) = ((S W) W) m; extraordinary: iS = D m, iD = S m
        double iv = ord ? (j == 0 ? W : S) : (j == 0 ? D : S);
        if (ord) {
            if (j == 2) iv = __dmul_rn(S, W);
            iv = __dmul_rn(iv, j < 2 ? V : W);
        }
        iv = __dmul_rn(iv, m);
        const double iS = from(iv, 0), i1 = from(iv, 1), iopg = from(iv, 2);
        double F;
        if (ord) {
            const double L2 = __dmul_rn(2.0, L), gg = __dmul_rn(__dmul_rn(L2, u), i1), opg = __dadd_rn(1.0, gg);
            // gX = ((L2 (L4uu iS - W)) iW) iW, gL = u2 iW - (((L4uu u) iS) iW) iW, gT = -gg iS
            double t = fma(j < 2 ? L4uu : -gg, j == 1 ? u : iS, j == 0 ? -W : -0.0);
            t = __dmul_rn(t, j == 0 ? L2 : j == 1 ? iS : 1.0);
            t = __dmul_rn(t, j < 2 ? i1 : 1.0);
            t = __dmul_rn(t, j < 2 ? i1 : 1.0);
            t = fma(j == 1 ? u2 : 1.0, j == 1 ? i1 : t, j == 1 ? -t : -0.0);
            F = __dmul_rn(fma(X, t, j == 0 ? -opg : -0.0), __dmul_rn(iopg, iopg));
        } else {
            const double N = __dmul_rn(__dmul_rn(2.0, X), u), cD = __dmul_rn(fma(-4.0, X, 2.0), D);
            const double t = fma(j == 0 ? L4u : j == 1 ? -__dmul_rn(u2, u) : -T, iS, j == 0 ? -2.0 : j == 1 ? -0.0 : -1.0);
            F = __dmul_rn(fma(N, t, j == 0 ? -cD : -0.0), __dmul_rn(i1, i1));
        }
        const double FX = from(F, 0), FL = from(F, 1), FT = from(F, 2);
        double kYn, c2;
        if (GRAD) {
            Duo::wait(Duo::kGradients);
            gYY = duo.D[Duo::dGYY + j];
            gkY = duo.D[Duo::dGKY + j];
            kv = duo.D[Duo::dKV + j];
            kYn = duo.D[Duo::dKYn];
            c2 = duo.D[Duo::dC2];
        } else {
            kYn = __dmul_rn(kY, ikk);
            c2 = __dmul_rn(__dmul_rn(2.0, kY), ikk);
        }
        const double cL = __dmul_rn(__dadd_rn(FL, -FT), c2);
        const double hf = __dmul_rn(0.5, cL);
        H = __dmul_rn(-0.5, fma(cL, gkY, fma(FX, dXj, __dmul_rn(FT, gYY))));
        K = fma(-hf, fma(-kYn, kj, Yj), kj);
        G = fma(T, FT, fma(L, FL, fma(X, FX, -kk)));
    }
    const double iG = __drcp_rn(G), irs = __dmul_rn(ir, ist);
    const double sc = j == 0 ? 1.0 : j == 1 ? ir : irs;
    d = __dmul_rn(__dmul_rn(-K, iG), sc);
    const double dr = from(d, 0), dt = from(d, 1), dp = from(d, 2);
    // kp sth in lane 0, (kp r) cth in lanes 1, 2
    if (!GRAD || rp.iso) kv = __dmul_rn(__dmul_rn(kp, j == 0 ? s.sth : s.r), j == 0 ? 1.0 : s.cth);
    const double kps = from(kv, 0);
    double t = __dmul_rn(j == 0 ? kt : j == 1 ? -kt : -kps, j == 0 ? dt : dr);
    t = fma(j < 2 ? kv : -kv, j < 2 ? dp : dt, fma(H, iG, t));
    dk = __dmul_rn(t, sc);
}

// X and its derivatives along r, theta, phi at the stage state ys by the G
// lanes of a group (lane q): into C[cO .. cO + 3] as X, dX/dtheta, dX/dphi,
// dX/dr, zeros outside the grid.  coef: the weight polynomials of the grid's
// interpolant.  Called by whole warps only (it holds barriers); the caller
// synchronises the warp before reading the result.
template <int G>
__device__ __forceinline__ void density64(const GridDev &g, double xfac, const double *ys, double *C,
                                          const double *coef, int q) {
    static_assert(G >= 4, "an axis per lane");
    // cells: an axis per lane
    int *cell = (int *)(C + cCell);
    if (q < 3) {
        int i;
        double t;
        const bool ok = cell64(grid_coord64(g, q, ys[0], ys[1], ys[2]), q == 0 ? g.n_lat : q == 1 ? g.n_lon : g.n_alt, i, t);
        C[cFrac + q] = t;
        C[cFrac + 3 + q] = 1.0 - t;
        cell[q] = ok ? i : -1;
    }
    __syncwarp();
    const int ca = cell[0], cb = cell[1], cc = cell[2];
    const bool inside = (ca | cb | cc) >= 0;
    if (!__any_sync(kFull, inside)) {
        if (q < 4) C[cO + q] = 0.0;
        return;
    }
    // this lane's sample rows, loaded ahead of the weights that they wait for
    constexpr int kRows = G == 32 ? 1 : 16 / G;
    const long long sj = g.p_alt, si = (long long)g.p_lon * g.p_alt;
    const double *base = g.pad64 + (long long)(inside ? ca : 0) * si + (long long)(inside ? cb : 0) * sj + (inside ? cc : 0);
    double u[kRows][4];
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
        const int row = G == 32 ? (q & 15) : q + r * G;
        const double *p = base + (row >> 2) * si + (row & 3) * sj;
#pragma unroll
        for (int c = 0; c < 4; ++c) u[r][c] = __ldg(p + c);
    }
    // the 24 weights: weight p = 8 axis + 4 derivative + node, one polynomial each
    for (int p = q; p < 24; p += G) {
        const int node = p & 3, der = (p >> 2) & 1;
        const bool right = node >= 2;
        const bool outer = node == 0 || node == 3;  // nodes j-1, j+2
        const double *cf = coef + (der * 2 + (outer ? 0 : 1)) * 5;
        const double t = C[cFrac + (right ? 3 : 0) + (p >> 3)];
        double w = fma(t, cf[0], cf[1]);
        w = fma(t, w, cf[2]);
        w = fma(t, w, cf[3]);
        // kinds 0, 2: one more Horner step; kind 1: t^2; kind 3: times t (adding -0 changes nothing)
        const double w4 = fma(t, (der | (int)outer) ? w : t, outer ? cf[4] : -0.0);
        const double w5 = __dmul_rn(w4, outer ? t : w);
        w = der ? w4 : __dadd_rn(outer ? -0.0 : 1.0, w5);
        C[cW + p] = (der && right) ? -w : w;
    }
    __syncwarp();
    // altitude rows (Eq. 13): row 4 a + b; with 32 lanes the upper half forms the derivative sums
    if (G == 32) {
        const double *w = C + cW + 16 + ((q >> 4) << 2);
        C[cV + q] = row64(u[0][0], u[0][1], u[0][2], u[0][3], w);
    } else {
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
            C[cV + q + r * G] = row64(u[r][0], u[r][1], u[r][2], u[r][3], C + cW + 16);
            C[cV + 16 + q + r * G] = row64(u[r][0], u[r][1], u[r][2], u[r][3], C + cW + 20);
        }
    }
    __syncwarp();
    // longitude: for each a the sums of v wb, v db, dv wb
    for (int id = q; id < 12; id += G) {
        const int a = id / 3, j = id - 3 * a;
        const double *v = C + cV + (j == 2 ? 16 : 0) + 4 * a;
        const double *w = C + cW + 8 + (j == 1 ? 4 : 0);
        double sum = 0.0;
#pragma unroll
        for (int b = 0; b < 4; ++b) sum = fma(v[b], w[b], sum);
        C[cS + id] = sum;
    }
    __syncwarp();
    // latitude, then to X and its derivatives
    for (int o = q; o < 4; o += G) {
        const double *v = C + cS + (o == 3 ? 2 : o == 2 ? 1 : 0);
        const double *w = C + cW + (o == 1 ? 4 : 0);
        double sum = 0.0;
#pragma unroll
        for (int a = 0; a < 4; ++a) sum = fma(v[3 * a], w[a], sum);
        const double c1 = o == 0 ? 1.0 : o == 1 ? g.inv_dlat : o == 2 ? g.inv_dlon : g.inv_dalt;
        const double c2 = o == 1 || o == 2 ? kRad2Deg : 1.0;
        C[cO + o] = inside ? (o == 1 ? -xfac : xfac) * sum * c1 * c2 : 0.0;
    }
}

// The warp's rays' sines and cosines: theta on the even lanes, phi on the odd ones.
__device__ __forceinline__ void angles64(StageIn<double> &s, const double *ys, int q) {
    s.r = ys[0];
    s.k[0] = ys[3];
    s.k[1] = ys[4];
    s.k[2] = ys[5];
    double sn, cs;
    sincos(ys[1 + (q & 1)], &sn, &cs);
    const double so = __shfl_xor_sync(kFull, sn, 1), co = __shfl_xor_sync(kFull, cs, 1);
    s.sth = (q & 1) ? so : sn;
    s.cth = (q & 1) ? co : cs;
    s.sph = (q & 1) ? sn : so;
    s.cph = (q & 1) ? cs : co;
}

// dy/dP' at the stage state ys (6 doubles of shared memory: the ray's state if
// at_state, else C + cT) by the G lanes of a group (lane q, scratch C), into out
// if write is set; returns sin(theta).  Called by the whole first warp only.
// The block's second warp helps (Duo): it forms X and its derivatives while
// this one forms the sines, the field and Appleton-Hartree's arguments, and
// with 32 lanes the field's gradients while this one goes through
// Appleton-Hartree.
// G = 1: the lane evaluates alone, the second warp does nothing.
template <int G>
__device__ __forceinline__ double stage64(const GridDev &g, const RayPhys<double> &rp, const double *ys, bool at_state,
                                          const double *C, int q, double *out, bool write, Duo &duo) {
    if constexpr (G == 1) {
        double y[6], dy[6], sth;
#pragma unroll
        for (int i = 0; i < 6; ++i) y[i] = ys[i];
        rhs64(g, rp, y, dy, nullptr, &sth);
        if (write) {
#pragma unroll
            for (int i = 0; i < 6; ++i) out[i] = dy[i];
        }
        return sth;
    }
    StageIn<double> s;
    const int j = (q & 3) == 3 ? 2 : (q & 3);  // the component this lane carries
    double d, dk;
    duo.start(G == 32 ? Duo::kSingle * (1 + (int)(ys - duo.sm)) : G + (at_state ? Duo::kState : 0), threadIdx.x);
    angles64(s, ys, q);
    tail64_quad<G == 32>(rp, s, C, j, q, duo, d, dk);
    if (write && q < 3) {
        out[q] = d;
        out[3 + q] = dk;
    }
    return s.sth;
}

// X and its derivatives for every group of the first warp.
template <int G>
__device__ __forceinline__ void densities64(const GridDev &g, const double *slots, double *scratch, const double *coef,
                                            int lane, bool at_state, const Duo &duo) {
    const int grp = lane / G;
    const double *S = slots + duo.slot_of[grp] * kSlot;
    double *C = scratch + grp * cGroup;
    density64<G>(g, S[kXfac], at_state ? S + kY : C + cT, C, coef, lane % G);
}

// The second warp of a block: serves the first one's requests until it is
// told to stop.  The requests' sequence is fixed (start, density, and for a
// single ray in a field the gradients), so every barrier's two sides always meet.
__device__ __forceinline__ void helper64(const GridDev &g, const double *slots, double *scratch, const double *coef,
                                         int lane, Duo &duo) {
    const int j = (lane & 3) == 3 ? 2 : (lane & 3);
    for (;;) {
        Duo::wait(Duo::kStart);
        const int what = *(volatile int *)duo.request;
        if (what == 0) return;
        if (what < Duo::kSingle) {  // the densities of several rays
            const bool at_state = (what & Duo::kState) != 0;
            const int G = what & (Duo::kState - 1);
            if (G == 4) densities64<4>(g, slots, scratch, coef, lane, at_state, duo);
            else if (G == 8) densities64<8>(g, slots, scratch, coef, lane, at_state, duo);
            else densities64<16>(g, slots, scratch, coef, lane, at_state, duo);
            Duo::signal(Duo::kDensity);
            continue;
        }
        const double *ys = duo.sm + (what / Duo::kSingle - 1);
        density64<32>(g, duo.D[Duo::dXfac], ys, scratch, coef, lane);
        Duo::signal(Duo::kDensity);
        if (g.iso != 0) continue;
        Duo::wait(Duo::kField);
        const double *D = duo.D;
        const double kr = ys[3], kt = ys[4], kp = ys[5];
        const double mr = D[Duo::dM], mt = D[Duo::dM + 1], mj = D[Duo::dM + j], A = D[Duo::dA], kY = D[Duo::dKY];
        const double ir = D[Duo::dIr], sth = D[Duo::dSth], cth = D[Duo::dCth], ikk = D[Duo::dIkk];
        double gYY, gkY;
        field_gradients(j, kr, kt, kp, mr, mt, mj, A, D[Duo::dA2], D[Duo::dYY], kY, ir, sth, cth, gYY, gkY);
        if (lane < 3) {
            duo.D[Duo::dGYY + lane] = gYY;
            duo.D[Duo::dGKY + lane] = gkY;
            duo.D[Duo::dKV + lane] = __dmul_rn(__dmul_rn(kp, j == 0 ? sth : ys[0]), j == 0 ? 1.0 : cth);
        }
        const double kYn = __dmul_rn(kY, ikk), c2 = __dmul_rn(__dmul_rn(2.0, kY), ikk);
        if (lane == 0) {
            duo.D[Duo::dKYn] = kYn;
            duo.D[Duo::dC2] = c2;
        }
        Duo::signal(Duo::kGradients);
    }
}

// Raw final state of a ray into its record (the angles stand in the
// ground-range and azimuth fields; finish_records_kernel turns them into the
// outputs).
__device__ __forceinline__ void write_raw(rt_ray_result *out, int id, double P, double th, double ph, double apo,
                                          int status, int steps, int att, int ev) {
    rt_ray_result r;
    r.group_path_km = P;
    r.ground_range_km = th;
    r.az_dev_deg = ph;
    r.apogee_km = apo;
    r.land_lat_deg = 0.0;
    r.land_lon_deg = 0.0;
    r.status = status;
    r.n_steps = steps;
    r.n_attempts = att;
    r.n_evals = ev;
    out[id] = r;
}

// Runs the warp's rays, G lanes each, until at most half of the groups are
// still in use (G = 1: until kWideLeft rays are left); then packs the remaining rays' slots to the front of map.
// One iteration is one step attempt (or one trial of the landing / exit
// solve) of every ray.  Groups without a ray follow group 0's ray and write
// nothing, so that the warp's barriers stay uniform.  The loop ends: every
// iteration adds an attempt to each ray, and a ray takes at most max_steps of
// them plus 60 trials.
template <int G>
__device__ __forceinline__ void run_rays(const GridDev &g, const FanDev &f, double *slots, double *scratch,
                                         const double *pow2q, int *map, int &n_act,
                                         rt_ray_result *__restrict__ out, Duo &duo) {
    const int lane = threadIdx.x, grp = lane / G, q = lane % G;  // the block's first warp
    const bool has = grp < n_act;
    const int slot = map[has ? grp : 0];
    double *S = slots + slot * kSlot;
    int *SI = (int *)(S + kInts);
    double *C = scratch + grp * (G == 1 ? cLane : cGroup);
    const bool adaptive = f.integrator == RT_RKF45;
    const int ns = adaptive ? 6 : 4;
    const double RE = g.R_E;
    RayPhys<double> rp;
    rp.xfac = S[kXfac];
    rp.ab0 = S[kAb0];
    rp.R_E = RE;
    rp.m[0] = g.m[0];
    rp.m[1] = g.m[1];
    rp.m[2] = g.m[2];
    rp.iso = g.iso != 0;
    rp.mode = SI[kMode];
    double P = S[kP], h = S[kH], hs = S[kHs], apo = S[kApo], r_prev = S[kRPrev], dr_prev = S[kDrPrev], h_prev = S[kHPrev];
    double la = S[kLa], lfa = S[kLfa], lb = S[kLb], lfb = S[kLfb];
    int steps = SI[kSteps], att = SI[kAtt], ev = SI[kEv], flags = SI[kFlags], side = SI[kSide], it = SI[kIt];
    const int id = SI[kId];
    bool live = has;
    const bool writer = q == 0;
    if (G > 1 && writer) duo.slot_of[grp] = slot;
    if (G == 32 && writer) duo.D[Duo::dXfac] = rp.xfac;
    __syncwarp();
    for (;;) {
        const unsigned am = __ballot_sync(kFull, live && writer);
        const int n = __popc(am);
        if (n == 0 || (G == 1 ? n <= kWideLeft : G < 32 && 2 * n * G <= 32)) {
            if (live && writer) {
                S[kP] = P; S[kH] = h; S[kHs] = hs; S[kApo] = apo; S[kRPrev] = r_prev; S[kDrPrev] = dr_prev;
                S[kHPrev] = h_prev; S[kLa] = la; S[kLfa] = lfa; S[kLb] = lb; S[kLfb] = lfb;
                SI[kSteps] = steps; SI[kAtt] = att; SI[kEv] = ev; SI[kFlags] = flags; SI[kSide] = side; SI[kIt] = it;
                map[__popc(am & ((1u << lane) - 1u))] = slot;
            }
            n_act = n;
            __syncwarp();
            return;
        }
        if (!live) {  // a group without a ray repeats plain steps from a fixed state
            flags = kK1Valid;
            h = f.h0;
        }
        const bool solving = (flags & (kLands | kExits)) != 0;
        if (live && !solving && att >= f.max_steps) {
            if (writer) write_raw(out, id, P, S[kY + 1], S[kY + 2], apo, RT_RAY_MAX_STEPS, steps, att, ev);
            live = false;
        }
        // k1 where it is not known (a new state)
        const bool need = live && !(flags & kK1Valid);
        if (__any_sync(kFull, need)) {
            const double sth = stage64<G>(g, rp, S + kY, true, C, q, S + kK1, need, duo);
            if (need) {
                ++ev;
                flags |= kK1Valid;
                if (writer) S[kSth] = sth;
            }
            __syncwarp();
        }
        bool at_face = false;
        if (!solving) hs = h;
        if (adaptive) {
            // distance to the next cell face, predicted linearly from k1; lateral
            // faces count only inside the altitude span
            const double y0 = S[kY], y1 = S[kY + 1], y2 = S[kY + 2];
            auto face = [&](int ax, double &x) {
                x = grid_coord64(g, ax, y0, y1, y2);
                const double v = (ax == 0 ? -S[kK1 + 1] : ax == 1 ? S[kK1 + 2] : S[kK1]) * (ax == 2 ? 1.0 : kRad2Deg) *
                                 (ax == 0 ? g.inv_dlat : ax == 1 ? g.inv_dlon : g.inv_dalt);
                return face_axis64(x, v, ax == 0 ? g.n_lat : ax == 1 ? g.n_lon : g.n_alt);
            };
            double x, best;
            if constexpr (G == 1) {
                const double d0 = face(0, x), d1 = face(1, x), d2 = face(2, x);
                const bool in_alt = x >= 0.0 && x <= (double)(g.n_alt - 1);
                best = in_alt ? fmin(fmin(d0, d1), d2) : d2;
            } else {
                const int ax = (q & 3) == 3 ? 2 : (q & 3);  // an axis per lane
                best = face(ax, x);
                const double xc = __shfl_sync(kFull, x, 2, 4);
                const bool in_alt = xc >= 0.0 && xc <= (double)(g.n_alt - 1);
                if (ax < 2 && !in_alt) best = HUGE_VAL;
                best = fmin(best, __shfl_xor_sync(kFull, best, 1));
                best = fmin(best, __shfl_xor_sync(kFull, best, 2));
            }
            if (!solving && best > 1e-3 * hs && best < hs) {
                hs = best * (1.0 + 1e-4);
                at_face = true;
            }
        }
        const double k10 = S[kK1];
        if (!solving) {
            if (f.max_path > 0.0 && P + hs > f.max_path) hs = f.max_path - P;
            if ((flags & kHavePrev) && dr_prev > 0.0 && k10 <= 0.0)
                apo = fmax(apo, hermite_peak(r_prev, S[kY], dr_prev, k10, h_prev) - RE);
            flags &= ~kHavePrev;
        }
        // the attempt: stages 1 .. ns-1, then the new state (and error estimate)
#pragma unroll 1
        for (int s = 1; s < ns; ++s) {
#pragma unroll 1
            for (int c = q; c < 6; c += G) {
                const double y = S[kY + c];
                C[cT + c] = adaptive ? rkf45_stage(s, y, hs, S + kK1, C + cK, c)
                                     : fma(s == 3 ? hs : 0.5 * hs, s == 1 ? S[kK1 + c] : C[cK + 6 * (s - 2) + c], y);
            }
            __syncwarp();
            stage64<G>(g, rp, C + cT, false, C, q, C + cK + 6 * (s - 1), true, duo);
            __syncwarp();
        }
        if (adaptive) {
#pragma unroll 1
            for (int c = q; c < 6; c += G) rkf45_end(S[kY + c], hs, S + kK1, C + cK, c, C[cT + c], C[cE + c]);
        } else {
            const double h6 = div_const(hs, 6.0, 1.0 / 6.0);
#pragma unroll 1
            for (int c = q; c < 6; c += G)
                C[cT + c] = __dadd_rn(S[kY + c], __dmul_rn(h6, __dadd_rn(fma(2.0, C[cK + 6 + c], fma(2.0, C[cK + c], S[kK1 + c])),
                                                                         C[cK + 12 + c])));
        }
        __syncwarp();
        double yn[6];
#pragma unroll
        for (int i = 0; i < 6; ++i) yn[i] = C[cT + i];
        ++att;
        ev += adaptive ? 5 : 3;
        // error norm (<= 1 accepts), as documented in rtgd.h: the two quotients on the even and odd lanes
        double fac = 1.0;
        bool accept = true;
        if (adaptive) {
            const double r = S[kY], sth = S[kSth], ky = S[kY + 3], kt = S[kY + 4], kp = S[kY + 5];
            const double e0 = C[cE], e1 = C[cE + 1], e2 = C[cE + 2], e3 = C[cE + 3], e4 = C[cE + 4], e5 = C[cE + 5];
            const double kmag = sqrt(fma(kp, kp, fma(ky, ky, __dmul_rn(kt, kt))));
            double pos, kerr;
            if (finite64(e0) && finite64(e1) && finite64(e2) && finite64(e3) && finite64(e4) && finite64(e5)) {
                pos = max_bits(fabs(e0), max_bits(r * fabs(e1), r * sth * fabs(e2)));
                kerr = max_bits(fabs(e3), max_bits(fabs(e4), fabs(e5)));
            } else {
                pos = max3_rare(e0, r, e1, r * sth, e2);
                kerr = max3_rare(e3, 1.0, e4, 1.0, e5);
            }
            const double dp = fma(f.rtol, r, f.atol), dk = f.rtol * fmax(kmag, 1e-3);
            double err;
            if constexpr (G == 1) {
                err = fmax(pos / dp, kerr / dk);
            } else {
                const double v = ((q & 1) ? kerr : pos) / ((q & 1) ? dk : dp);
                err = fmax(v, __shfl_xor_sync(kFull, v, 1));
            }
            fac = step_factor64(err, pow2q);
            accept = err <= 1.0;
        }
        // new state inside the grid's lat/lon span?  (an axis per lane)
        int cell_i;
        double cell_t;
        const bool in_ax = cell64(grid_coord64(g, q & 1, yn[0], yn[1], yn[2]), (q & 1) ? g.n_lon : g.n_lat, cell_i, cell_t);
        bool lateral;
        if constexpr (G == 1)
            lateral = cell64(grid_coord64(g, 1, yn[0], yn[1], yn[2]), g.n_lon, cell_i, cell_t) && in_ax;
        else
            lateral = __shfl_xor_sync(kFull, (int)in_ax, 1) && in_ax;
        const double y0 = S[kY];
        if (solving) {
            // ground return or exit through the grid top: r(step(h*)) = R_E (or
            // R_E + top) for h* in (0, step], Illinois regula falsi; sg makes the
            // bracket function positive at the step start
            const bool lands = (flags & kLands) != 0;
            const double rt = lands ? RE : RE + g.top, sg = lands ? 1.0 : -1.0;
            const double fc = sg * (yn[0] - rt);
            ++it;
            if (fabs(fc) < 1e-9 || it >= 60) {
                P += hs;
                ++steps;
                if (!lands) apo = fmax(apo, yn[0] - RE);
                if (live && writer)
                    write_raw(out, id, P, yn[1], yn[2], apo, lands ? RT_RAY_LANDED : RT_RAY_ESCAPED, steps, att, ev);
                live = false;
            } else {
                if (fc < 0.0) {
                    lb = hs;
                    lfb = fc;
                    if (side == -1) lfa *= 0.5;
                    side = -1;
                } else {
                    la = hs;
                    lfa = fc;
                    if (side == 1) lfb *= 0.5;
                    side = 1;
                }
                hs = lb - lfb * (lb - la) / (lfb - lfa);
            }
        } else if (!accept) {
            // the nominal step changes only by quantised factors of itself
            h = h * fac;
            if (h < f.hmin) {
                if (live && writer)
                    write_raw(out, id, P, S[kY + 1], S[kY + 2], apo, RT_RAY_STEP_UNDERFLOW, steps, att, ev);
                live = false;
            }
        } else if (!(finite64(yn[0]) && finite64(yn[1]) && finite64(yn[2]) && finite64(yn[3]) && finite64(yn[4]) &&
                     finite64(yn[5]))) {
            if (live && writer) write_raw(out, id, P, S[kY + 1], S[kY + 2], apo, RT_RAY_NONFINITE, steps, att, ev);
            live = false;
        } else {
            const bool lands = yn[0] < RE;
            const bool exits = !lands && yn[0] - RE > g.top;
            if (lands || exits) {
                const double rt = lands ? RE : RE + g.top, sg = lands ? 1.0 : -1.0;
                flags |= lands ? kLands : kExits;
                la = 0.0;
                lfa = sg * (y0 - rt);
                lb = hs;
                lfb = sg * (yn[0] - rt);
                side = 0;
                it = 0;
                hs = lb - lfb * (lb - la) / (lfb - lfa);
            } else {
                P += hs;
                ++steps;
                apo = fmax(apo, yn[0] - RE);
                flags = (flags | kHavePrev) & ~kK1Valid;
                r_prev = y0;
                dr_prev = k10;
                h_prev = hs;
                int status = RT_RAY_NOT_RUN;
                if (yn[0] - RE >= g.alt0 && !lateral) status = RT_RAY_LEFT_GRID;
                else if (f.max_path > 0.0 && P >= f.max_path - 1e-12) status = RT_RAY_MAX_PATH;
                if (status != RT_RAY_NOT_RUN) {
                    if (live && writer) write_raw(out, id, P, yn[1], yn[2], apo, status, steps, att, ev);
                    live = false;
                }
                if (adaptive) h = fmin(fmax(h * (at_face ? fmin(1.0, fac) : fac), f.hmin), f.hmax);
            }
        }
        // (a reader of the old state above has passed the barrier before the new one is written)
        const bool moved = !(flags & kK1Valid);
        __syncwarp();
        if (live && writer && moved) {
#pragma unroll
            for (int i = 0; i < 6; ++i) S[kY + i] = yn[i];
        }
        __syncwarp();
    }
}

// Bytes of shared memory of a block that starts with R rays.
__host__ __device__ constexpr int fp64_scratch(int R) {
    return R <= kGroups ? R * cGroup : R * cLane > kGroups * cGroup ? R * cLane : kGroups * cGroup;
}
constexpr size_t fp64_smem_bytes(int R) {
    return sizeof(double) * (size_t)(kPoly + kPow2 + Duo::dSize + R * kSlot + fp64_scratch(R)) +
           (R + 1 + kGroups) * sizeof(int);
}
static_assert(fp64_smem_bytes(kGroups) <= 48 * 1024 && fp64_smem_bytes(kWideRays) <= 48 * 1024,
              "fits the default shared-memory limit");

// A warp with R rays (a power of two, at most kGroups; WIDE: kWideRays) at the
// start and its helper per block.  kBlocksPerSm = 6 blocks per SM (168 registers): the FP64
// pipe is full with four warps, and more blocks only slow a fan's longest rays
// (24,840 rays 149 ms, 162 with the eight of 128 registers).
template <bool WIDE>
__global__ void __launch_bounds__(64, kBlocksPerSm) trace_fp64_kernel(const __grid_constant__ GridDev g,
                                                        const __grid_constant__ FanDev f, int R,
                                                        rt_ray_result *__restrict__ out) {
    extern __shared__ double sm[];
    double *coef = sm, *pow2q = coef + kPoly, *hand = pow2q + kPow2, *slots = hand + Duo::dSize,
           *scratch = slots + R * kSlot;
    int *map = (int *)(scratch + fp64_scratch(R));
    Duo duo{hand, map + R, map + R + 1, sm};
    const int lane = threadIdx.x & 31;
    if (threadIdx.x >= 32) {
        helper64(g, slots, scratch, coef, lane, duo);
        return;
    }
    if (lane < kPoly) coef[lane] = (&c_poly[g.interp == 1 ? 1 : 0][0][0])[lane];
    if (lane < kPow2) pow2q[lane] = exp2((double)(lane - 10) * 0.25);
    // launch: |k| = mu at the transmitter (one ray per lane; spare lanes do nothing)
    const long long claim = (long long)blockIdx.x * R + lane;
    bool live = lane < R && claim < f.n_rays;
    if (live) {
        const long long ray = claim_to_ray(f, claim);
        const RayParams p = ray_params(f, ray);
        const RayPhys<double> rp = make_phys<double>(g, p.f_hz, p.mode);
        double y[6], dummy[6], mu2 = 0.0;
        launch_dir(f, p, y);
        rhs64(g, rp, y, dummy, &mu2);
        if (!(mu2 > 0.0)) {
            write_raw(out, (int)ray, 0.0, y[1], y[2], f.tx_r - g.R_E, RT_RAY_NONFINITE, 0, 0, 1);
            live = false;
        } else {
            const double mu = sqrt(mu2);
            y[3] *= mu;
            y[4] *= mu;
            y[5] *= mu;
            double *S = slots + lane * kSlot;
            int *SI = (int *)(S + kInts);
            for (int i = 0; i < 6; ++i) {
                S[kY + i] = y[i];
                S[kK1 + i] = 0.0;
            }
            S[kSth] = S[kP] = S[kRPrev] = S[kDrPrev] = S[kHPrev] = S[kLa] = S[kLfa] = S[kLb] = S[kLfb] = 0.0;
            S[kH] = S[kHs] = f.h0;
            S[kApo] = y[0] - g.R_E;
            S[kXfac] = rp.xfac;
            S[kAb0] = rp.ab0;
            SI[kId] = (int)ray;
            SI[kMode] = p.mode;
            SI[kSteps] = SI[kAtt] = SI[kFlags] = SI[kSide] = SI[kIt] = 0;
            SI[kEv] = 1;
        }
    }
    const unsigned am = __ballot_sync(kFull, live);
    if (live) map[__popc(am & ((1u << lane) - 1u))] = lane;
    __syncwarp();
    int n_act = __popc(am);
    while (n_act > 0) {
        if (WIDE && n_act > kWideLeft) {
            run_rays<1>(g, f, slots, scratch, pow2q, map, n_act, out, duo);
            continue;
        }
        const int wait = WIDE && n_act > kGroups ? n_act - kGroups : 0;  // rays at the front of map whose turn comes later
        int n = n_act - wait;
        if (n > 4) run_rays<4>(g, f, slots, scratch, pow2q, map + wait, n, out, duo);
        else if (n > 2) run_rays<8>(g, f, slots, scratch, pow2q, map + wait, n, out, duo);
        else if (n > 1) run_rays<16>(g, f, slots, scratch, pow2q, map + wait, n, out, duo);
        else run_rays<32>(g, f, slots, scratch, pow2q, map + wait, n, out, duo);
        n_act = wait + n;
    }
    duo.start(0, lane);  // the helper ends
}

// dy/dP' at the states of a block (diagnostic): G lanes each, as run_rays
// evaluates k1; count of them, in the slots.
template <int G>
__device__ __forceinline__ void eval_states(const GridDev &g, int mode, double *slots, double *scratch, int count,
                                            double *__restrict__ dys, Duo &duo) {
    const int lane = threadIdx.x, grp = lane / G, q = lane % G;
    const bool has = grp < count;
    double *S = slots + (has ? grp : 0) * kSlot;
    double *C = scratch + grp * (G == 1 ? cLane : cGroup);
    RayPhys<double> rp;
    rp.xfac = S[kXfac];
    rp.ab0 = S[kAb0];
    rp.R_E = g.R_E;
    rp.m[0] = g.m[0];
    rp.m[1] = g.m[1];
    rp.m[2] = g.m[2];
    rp.iso = g.iso != 0;
    rp.mode = mode;
    if (G > 1 && q == 0) duo.slot_of[grp] = has ? grp : 0;
    if (G == 32 && q == 0) duo.D[Duo::dXfac] = rp.xfac;
    __syncwarp();
    stage64<G>(g, rp, S + kY, true, C, q, S + kK1, has, duo);
    __syncwarp();
    for (int c = q; has && c < 6; c += G) dys[grp * 6 + c] = S[kK1 + c];
}

// R states per block, as many as a warp of a trace of n rays starts with: so the
// states are evaluated by the same code as that trace's, 1, 4, 8, 16 or 32 lanes
// each.  mu^2 is the launch's evaluation.
__global__ void __launch_bounds__(64, kBlocksPerSm) eval_rhs_fp64_kernel(const __grid_constant__ GridDev g,
                                                                      const double *__restrict__ ys,
                                                                      double *__restrict__ dys,
                                                                      double *__restrict__ mu2s, double f_hz, int mode,
                                                                      int R, long long n) {
    extern __shared__ double sm[];
    double *coef = sm, *hand = coef + kPoly + kPow2, *slots = hand + Duo::dSize, *scratch = slots + R * kSlot;
    int *map = (int *)(scratch + fp64_scratch(R));
    Duo duo{hand, map + R, map + R + 1, sm};
    const int lane = threadIdx.x & 31;
    if (threadIdx.x >= 32) {
        helper64(g, slots, scratch, coef, lane, duo);
        return;
    }
    if (lane < kPoly) coef[lane] = (&c_poly[g.interp == 1 ? 1 : 0][0][0])[lane];
    const long long first = (long long)blockIdx.x * R;
    const int count = (int)(n - first < R ? n - first : R);
    if (lane < count) {
        const RayPhys<double> rp = make_phys<double>(g, f_hz, mode);
        double *S = slots + lane * kSlot;
        double y[6], dy[6], mu2;
        for (int c = 0; c < 6; ++c) S[kY + c] = y[c] = ys[(first + lane) * 6 + c];
        S[kXfac] = rp.xfac;
        S[kAb0] = rp.ab0;
        rhs64(g, rp, y, dy, &mu2);
        mu2s[first + lane] = mu2;
    }
    __syncwarp();
    dys += first * 6;
    if (R > kGroups) eval_states<1>(g, mode, slots, scratch, count, dys, duo);
    else if (R > 4) eval_states<4>(g, mode, slots, scratch, count, dys, duo);
    else if (R > 2) eval_states<8>(g, mode, slots, scratch, count, dys, duo);
    else if (R > 1) eval_states<16>(g, mode, slots, scratch, count, dys, duo);
    else eval_states<32>(g, mode, slots, scratch, count, dys, duo);
    duo.start(0, lane);  // the helper ends
}

}  // namespace

// Rays a warp starts with, by the rays per SM: one while a block more fits the
// pipe beside the others (a first warp issues one FP64 instruction per 64 cycles,
// the pipe takes one per 19: about 3.4 blocks an SM), and twice as many rays at
// each doubling.  The first line lies a little above that: where two of the
// longest rays are neighbours, two rays a warp lose more than they gain
// elsewhere.  152 SMs, RKF45, a registration sector in ten ionospheres, two rays a
// warp against one: 414 rays 1.03 to 1.11 of the time, 468 rays 0.92 to 1.01, 522
// rays 0.92 to 1.02 (1.20 in an eleventh), 640 rays 0.77 to 0.84; four against two:
// 800 rays 1.08, 1,000 rays 0.99, 1,220 rays 0.95.  Other fans, 1 / 2 / 4 / 8 rays
// per warp: 2,000 rays 90 / 68.5 / 63.7 / 66.8 ms, 3,000 rays 101 / 75.4 / 70.8 /
// 71.2 ms, 4,968 rays 134 / 91 / 71.5 / 65.8 ms, 24,840 rays 571 / 335 / 210 /
// 149 ms.
//
// From two full waves of 32-ray warps (58,368 rays on 152 SMs) a fan is bound by
// the pipe's throughput rather than by its longest rays, and one lane per ray
// costs the least of it.  One thread per ray to the end / 8 rays / 32 rays per
// warp: 49,464 short uneven rays (20-28 MHz) 206 / 205 / 140 ms, 61,830 of them
// 211 / 252 / 174 ms, 98,928 of them 321 / 392 / 254 ms, 98,928 rays of 8-16 MHz
// 543 / 444 / 325 ms; an elevation scan at 0.1 degrees, whose long rays are
// neighbours: 51,098 rays 631 / 310 / 412 ms, 63,432 994 / 393 / 417 ms, 72,242
// 1,156 / 457 / 503 ms, 100,434 1,034 / 531 / 483 ms, 248,442 1,577 / 1,289 /
// 788 ms, 495,122 2,026 / 2,551 / 1,535 ms.
int fp64_rays_per_warp(long long n_rays, int sms) {
    const double per_sm = (double)n_rays / sms;
    if (per_sm >= 2 * kWideRays * kBlocksPerSm) return kWideRays;
    return per_sm <= 3.655 ? 1 : per_sm <= 7.266 ? 2 : per_sm <= 14.845 ? 4 : kGroups;
}

cudaError_t launch_trace_fp64(const GridDev &g, const FanDev &f, int rays_per_warp, rt_ray_result *out,
                              cudaStream_t st) {
    const int R = rays_per_warp;
    const long long blocks = (f.n_rays + R - 1) / R;
    if (R > kGroups) trace_fp64_kernel<true><<<(unsigned)blocks, 64, fp64_smem_bytes(R), st>>>(g, f, R, out);
    else trace_fp64_kernel<false><<<(unsigned)blocks, 64, fp64_smem_bytes(R), st>>>(g, f, R, out);
    return cudaGetLastError();
}

cudaError_t launch_eval_rhs_fp64(const GridDev &g, const double *ys, double *dys, double *mu2s, double freq_mhz,
                                 int mode, int sms, long long n, cudaStream_t st) {
    if (n == 0) return cudaSuccess;
    const int R = fp64_rays_per_warp(n, sms);
    eval_rhs_fp64_kernel<<<(unsigned)((n + R - 1) / R), 64, fp64_smem_bytes(R), st>>>(g, ys, dys, mu2s, freq_mhz * 1e6,
                                                                                     mode, R, n);
    return cudaGetLastError();
}

}  // namespace rtgd
