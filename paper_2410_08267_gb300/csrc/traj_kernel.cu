// Persistent trajectory kernel for relic overdensity profiles (sm_103a).
//
// One thread integrates TPT trajectories (one per (radius, |P0|, mu) triple,
// Sec. II.C) backward from z0 = 0 to z_end with classical RK4 in u = ln a
// (Eq. eoms), the force being the closed-form gradient of the compensated,
// growing NFW halo (App. A).  The state (x, y, vx, vy) stays in registers for
// the whole integration; the per-step coefficients (background, growth,
// coupling at the three RK stage times, built in FP64 on the host) come to each
// warp through a window of its own in shared memory.  At the end the Liouville
// map f0 = f_init(P_i) (Sec. II.C) and the weight of the trajectory in
// Eq. localdensity are applied, once per relic mass read from the trajectory
// (Sec. III), and each tile's sum is formed by a warp-shuffle + shared-memory tree.
// Tile sums land in a per-request array; the CTA that completes the last tile of a
// radius adds them in an order that the trajectories alone fix (so every result is
// bitwise independent of the kernel, of scheduling and of what else shares the
// launch) and writes n/nbar.  plan_shape chooses the kernel of a launch.
//
// Work distribution: CTAs of a persistent grid pull tile indices from one
// atomic counter; a tile is `tile` consecutive trajectories of one radius of
// one request, so uneven batches of requests share one launch.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <type_traits>

#include "nuprof_internal.h"

namespace nuprof {

static std::atomic<long long> g_launches{0};
void count_launch() { g_launches.fetch_add(1, std::memory_order_relaxed); }
long long launches() { return g_launches.load(std::memory_order_relaxed); }

// ---------------------------------------------------------------------------
// Force evaluation: m = Mhat(r, z) / r^3, so that gradPhi / F = m * (x, y).
//   Mhat = I(r/(r_s (1+z))) / I(c) - (r/R)^3   for r < r200 (1+z)
//        = 1 - (r/R)^3                         for r < R
//        = 0                                   otherwise          (App. A)
// which gives m = sel / r^3 - 1/R^3 with sel = I/I(c) inside the NFW edge and
// 1 in the shell, and m = 0 beyond R.
// ---------------------------------------------------------------------------

__device__ __forceinline__ float rsqrt_approx(float v)
{
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float lg2_approx(float v)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

__device__ __forceinline__ float rcp_approx(float v)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(v));
    return r;
}

// I(y) = ln(1+y) - y/(1+y) (Eq. nfw) in FP32.  For small y the two terms
// cancel, so inside the NFW part I = y^2 g(y) with g = I/y^2 approximated by a
// rational function N(y)/D(y) (nfw_rational_fit.py).  Two fits exist, and a
// request uses one of them for all of its evaluations:
//   wide:   degrees 4 and 5 on 0 <= y <= 16 (6e-8 relative, 3e-7 after float32
//           rounding; every coefficient positive), for halos with c > 8;
//   narrow: degrees 4 and 4 on 0 <= y <= 8 (6e-8, 3e-7), one fused
//           multiply-add cheaper, for halos with c <= 8, whose NFW part never
//           reaches y = 8.
// Above y = 16 (halos with c > 16) the two terms differ by more than a factor
// 1.5 and are subtracted directly, with the hardware base-2 logarithm and
// reciprocal (rcp(-u) = -1/u exactly).
__device__ __forceinline__ float nfw_N16(float y)
{
    float p = 3.952767202e-06f;
    p = fmaf(p, y, 2.387282439e-03f);
    p = fmaf(p, y, 6.631398201e-02f);
    p = fmaf(p, y, 3.795046508e-01f);
    p = fmaf(p, y, 5.000000596e-01f);
    return p;
}

__device__ __forceinline__ float nfw_D16(float y)
{
    float p = 5.989100318e-04f;
    p = fmaf(p, y, 3.099172190e-02f);
    p = fmaf(p, y, 3.629413843e-01f);
    p = fmaf(p, y, 1.422382593e+00f);
    p = fmaf(p, y, 2.092346668e+00f);
    p = fmaf(p, y, 1.0f);
    return p;
}

__device__ __forceinline__ float nfw_N8(float y)
{
    float p = -4.539978363e-06f;
    p = fmaf(p, y, 4.568357544e-04f);
    p = fmaf(p, y, 4.554858804e-02f);
    p = fmaf(p, y, 3.421576917e-01f);
    p = fmaf(p, y, 5.000000000e-01f);
    return p;
}

__device__ __forceinline__ float nfw_D8(float y)
{
    float p = 1.647129469e-02f;
    p = fmaf(p, y, 2.829689085e-01f);
    p = fmaf(p, y, 1.281258702e+00f);
    p = fmaf(p, y, 2.017652512e+00f);
    p = fmaf(p, y, 1.0f);
    return p;
}

// Largest concentration served by the narrow fit.
constexpr float kNarrowMaxC = 8.0f;

// y = r^2 rs is passed together with u = 1 + y formed as one fused
// multiply-add from r^2 and rs (every FP32 product that feeds a sum is written
// as an explicit fused multiply-add, here and in the packed path, so that no
// compiler contraction decides the rounding).
__device__ __forceinline__ float nfw_I_log(float y, float u)
{
    return fmaf(lg2_approx(u), 0.693147180559945309f, y * rcp_approx(-u));
}

// Same in FP64, accurate to a few ulp for every y.  With t = y/(1+y),
// I = -ln(1-t) - t = t^2 sum_{k>=0} t^k/(k+2), a series of positive terms; for
// t < 1/2 (y < 1) it is summed by Horner through k = 50 (truncation below
// 1e-16 relative), above that the two terms no longer cancel badly.
//
// An FP64 operation holds a scheduler's FP64 unit for 64 cycles here, where an FP32
// or integer one takes one or two: the FP64 force is bound by the number of its
// FP64 operations, one warp on a scheduler is enough to keep the unit busy, and
// work moved off it is free.  So:
// * Horner's recurrence p <- t p + 1/(k+2) forgets its start by a factor t a step.
//   It starts in FP32, whose relative error 2^-22 is multiplied by t^J in the J
//   FP64 steps that remain; J is the smallest multiple of 4 that makes that
//   2^-93, 2^-40 of an ulp of the sum.  So the sum has the bits of the whole
//   recurrence but where a rounding lies within 2^-40 ulp of a tie (none of 9e9
//   arguments differed).  Each lane starts at its own J while the warp runs the steps
//   of the largest, so the sum depends on t alone, not on what shares the warp.
// * Non-negative numbers are ordered as their bits, so tests are integer ones.
// * t is the quotient from Newton's iteration and Markstein's final correction (IBM
//   J. Res. Dev. 34, 1990), with an FP32 reciprocal as seed: the bits of the
//   division on all of 1.3e10 arguments from 2^-60 to 2^1000.
constexpr float kSeriesBits = 71.0f;       // 93 - 22
constexpr int kSeriesTail = 20;            // FP32 terms: 2^-23 at the largest t that uses them
constexpr int kSeriesMaxJ = 48;            // above: the whole recurrence

__device__ const float4 c_series[(kSeriesMaxJ + kSeriesTail) / 4] = {   // 1/(k+2)
#define NU_INV4(k) {1.0f / ((k) + 2), 1.0f / ((k) + 3), 1.0f / ((k) + 4), 1.0f / ((k) + 5)}
#define NU_INV16(k) NU_INV4(k), NU_INV4((k) + 4), NU_INV4((k) + 8), NU_INV4((k) + 12)
    NU_INV16(0), NU_INV16(16), NU_INV16(32), NU_INV16(48), NU_INV4(64)
#undef NU_INV16
#undef NU_INV4
};

// a < b for doubles that are not negative (false for a NaN a but where its sign is set,
// as the hardware's NaN may be: what follows from it is NaN either way)
__device__ __forceinline__ bool less_nonneg(double a, double b)
{
    return __double_as_longlong(a) < __double_as_longlong(b);
}

// float of a positive double, truncated (values below the float range: about 1e-38),
// and double of a positive float; integer operations only.
__device__ __forceinline__ float trunc_f32(double v)
{
    const int hi = max(__double2hiint(v), 0x38100000);
    return __uint_as_float(((unsigned)(hi - 0x38000000) << 3) | ((unsigned)__double2loint(v) >> 29));
}
__device__ __forceinline__ double widen_f32(float v)
{
    const unsigned b = __float_as_uint(v);
    return __hiloint2double((int)((b >> 3) + 0x38000000u), (int)(b << 29));
}

// y / u for y >= 0 and u = 1 + y as rounded (6 FP64 operations).
__device__ __forceinline__ double quotient(double y, double u)
{
    const double r0 = widen_f32(rcp_approx(trunc_f32(u)));   // 1/u to 2^-22
    const double e = fma(-u, r0, 1.0);
    const double r = fma(r0, fma(e, e, e), r0);               // to an ulp
    const double q = y * r;
    const double t = fma(fma(-q, u, y), r, q);                // the remainder is exact
    // from u = 2^54 on the quotient rounds to 1; the seed ends with the float range
    return less_nonneg(0x1p60, u) ? 1.0 : t;
}

template <int K>
__device__ __forceinline__ double series4(double p, double t)   // terms K + 3 .. K
{
    p = fma(p, t, 1.0 / (K + 5));
    p = fma(p, t, 1.0 / (K + 4));
    p = fma(p, t, 1.0 / (K + 3));
    return fma(p, t, 1.0 / (K + 2));
}

// The same where J > K, and the start value elsewhere.  The choice is made on the
// last step's operands: on its result it would lengthen the chain (FP64 cases 2 to 3 %).
template <int K>
__device__ __forceinline__ double series4_from(double p, double t, int J, double start)
{
    p = fma(p, t, 1.0 / (K + 5));
    p = fma(p, t, 1.0 / (K + 4));
    p = fma(p, t, 1.0 / (K + 3));
    return fma(p, J > K ? t : 0.0, J > K ? 1.0 / (K + 2) : start);
}

// FP64 steps that t < 1/2 needs: a multiple of 4 from 8 to kSeriesMaxJ, or more, up to
// 68 (the whole recurrence).  For any other t a number in that range.
__device__ __forceinline__ int series_steps(double t)
{
    const float above = __uint_as_float(__float_as_uint(trunc_f32(t)) + 1u);
    const int need = (int)fminf(kSeriesBits * rcp_approx(-lg2_approx(above)), 64.0f) + 1;
    return max(8, (need + 3) & ~3);
}

// Horner's value before the last J (48 where J is more) steps.  J_max: the warp's most,
// whose branch is uniform (one for each lane's J costs 3 %).
__device__ __forceinline__ double series_start(double t, int J, int J_max)
{
    const float tf = trunc_f32(t);
    const float4* c = c_series + min(J, kSeriesMaxJ) / 4;
    float s = 0.0f;
#pragma unroll
    for (int i = kSeriesTail / 4 - 1; i >= 0; --i) {
        const float4 q = __ldg(c + i);
        s = fmaf(fmaf(fmaf(fmaf(s, tf, q.w), tf, q.z), tf, q.y), tf, q.x);
    }
    double p = widen_f32(s);
    if (J_max > kSeriesMaxJ) {
        const double whole = fma(fma(1.0 / 52.0, t, 1.0 / 51.0), t, 1.0 / 50.0);
        if (J > kSeriesMaxJ) p = whole;
    }
    return p;
}

// sums_{k=0}^{50} t^k/(k+2) of N values 0 < t < 1/2, their chains side by side.  J: the
// steps that they need (series_steps); J_max: the most of the warp's, or more.
template <int N>
__device__ __forceinline__ void nfw_series_n(const double (&t)[N], const int (&J)[N], int J_max,
                                             double (&p)[N])
{
    double start[N];
#pragma unroll
    for (int i = 0; i < N; ++i) {
        p[i] = start[i] = series_start(t[i], J[i], J_max);
    }
#define NU_TERMS(K)                                                                      \
    case (K) + 4:                                                                        \
        _Pragma("unroll") for (int i = 0; i < N; ++i)                                    \
            p[i] = series4_from<K>(p[i], t[i], J[i], start[i]);
    switch (min(J_max, kSeriesMaxJ)) {
        NU_TERMS(44) NU_TERMS(40) NU_TERMS(36) NU_TERMS(32) NU_TERMS(28) NU_TERMS(24)
        NU_TERMS(20) NU_TERMS(16) NU_TERMS(12) NU_TERMS(8)
    default:;                                        // every case goes on with the next
    }
#undef NU_TERMS
#pragma unroll
    for (int i = 0; i < N; ++i) p[i] = series4<0>(series4<4>(p[i], t[i]), t[i]);
}
__device__ __forceinline__ double nfw_series(double t, int J, int J_max)
{
    double p[1];
    nfw_series_n<1>({t}, {J}, J_max, p);
    return p[0];
}
__device__ __forceinline__ void nfw_series2(double ta, double tb, int Ja, int Jb, int J_max, double& pa,
                                            double& pb)
{
    double p[2];
    nfw_series_n<2>({ta, tb}, {Ja, Jb}, J_max, p);
    pa = p[0];
    pb = p[1];
}

// Steps between two tests of the early exit in the counting launch (a power of two).
constexpr int kExitEvery = 4;

// Added to r^2 in FP32 so that a trajectory through r = 0 exactly gets a
// finite reciprocal square root.
constexpr float kR2Guard = 1e-20f;

// A trajectory is finished when its velocity can no longer change: it lies
// beyond R, where the gradient is exactly zero (mass compensation, App. A),
// and the straight line it follows from there along the integration direction
// (-v: the backward step moves it along -v) does not come back within R
// before z_end.  That holds when it recedes (x . v <= 0); when the line's
// closest approach to the centre, b^2 = r^2 - (x . v)^2 / v^2, stays beyond R
// (App. B's first criterion, for rays that miss the halo); or when the
// trajectory is too slow to cover the distance r - R before z_end (App. B's
// second criterion, v I_io < r - R), with irem the remaining force-free
// distance per unit speed of the discrete map.  All three are exact here
// because nothing acts outside R.  The factor kMiss keeps the tests safe
// against the rounding of the stepped positions (relative deviations below
// 1e-4 from the straight line).
template <typename T>
__device__ __forceinline__ bool escapes(T r2, T dot, T v2, T R2, T R, T irem)
{
    const T kMiss = T(1.001);
    if (!(r2 >= R2)) return false;
    if (dot <= T(0) || (r2 - kMiss * R2) * v2 >= dot * dot) return true;
    const T reach = R + sqrt(v2) * irem;          // farthest start that still reaches R
    return r2 >= kMiss * (reach * reach);
}

// c: the NFW edge r = r200 (1+z) in y = r S; narrow: c <= 8, the request uses
// the narrow rational fit.
struct HaloF32 { float invIc, invR3, R2, R, c; bool narrow; };
struct HaloF64 { double invIc, invR3, R2, R; };

// Branch tallies of force evaluations, kept only by the counting variant of the
// kernel (used once, untimed, to turn the data-dependent work into an exact
// algorithmic flop count): beyond R, shell, NFW part on the first branch of
// I(y) (FP32: the rational function; FP64: the series), NFW part on the
// logarithm branch, and the trajectory-steps of
// unfinished trajectories.  Steps that a finished trajectory runs only because
// its warp is still busy are not counted (they are not needed work); the sixth
// count is every lane-step the warps ran, needed or not (padding lanes too).
struct NoTally {
    __device__ __forceinline__ void add(int) {}
    __device__ __forceinline__ void set_live(bool) {}
    __device__ __forceinline__ void ran(unsigned) {}
};
struct Tally {
    unsigned n[6] = {0u, 0u, 0u, 0u, 0u, 0u};   // 4 branches, live steps, lane-steps run
    bool live = true;                           // only unfinished trajectories count
    __device__ __forceinline__ void add(int k) { n[k] += live ? 1u : 0u; }
    __device__ __forceinline__ void set_live(bool v)
    {
        live = v;
        n[4] += v ? 1u : 0u;
    }
    __device__ __forceinline__ void ran(unsigned k) { n[5] += k; }
};

// The compensated halo's gradient vanishes beyond R, and the NFW term only
// enters inside r200 (1+z): both tests are branches, so a warp whose lanes
// are all beyond R (or all in the shell) skips that work.  The result is the
// same value the full expression gives (0, resp. sel = 1).
//
// FP32 arithmetic of one evaluation, fixed per branch so that every code path
// (scalar, packed, any warp composition) gives a lane the same bits.  With
// rs = S/r and the table's T = S/I(c) (so y = r S = r^2 rs):
//   beyond R:              m = 0
//   NFW, y < Yq:           m = (N(y) (rs T)) rcp(D(y)) - 1/R^3
//                          (I rinv^3 / I(c) = y^2 g rinv^3 / I(c) = g S^2 rinv / I(c))
//   NFW, Yq <= y < c:      m = (I(y)/I(c)) rinv^3 - 1/R^3
//   shell:                 m = rinv^2 rinv - 1/R^3 (one rounding)
// Yq, the stage's bound of the rational branch (the FP32 table's C_Q slots),
// is min(c, 16, (1 - 1e-3) R S): y < Yq implies r < R with a margin far above
// the rounding of y, so that one compare classifies a lane.  The NFW part is
// y < c (the edge r = r200 (1+z) is y = c exactly), tested on y itself; the
// FP64 path tests r^2 against the table's squared edge.  The two tests differ
// only in the rounding at the edge, where the mass is continuous.
// The r -> 0 guard is folded into r^2 itself: r^2 = x^2 + (y^2 + 1e-20) with
// two fused multiply-adds, which changes the bits of r^2 only below ~2e-13 kpc^2.
__device__ __forceinline__ float guarded_r2(float x, float y)
{
    return fmaf(x, x, fmaf(y, y, kR2Guard));
}

template <class Ctr = NoTally>
__device__ __forceinline__ float accel_m(float x, float y, float S, float Yq, float T,
                                         const HaloF32& hc, Ctr& ctr)
{
    const float r2 = guarded_r2(x, y);
    float m = 0.0f;
    if (r2 < hc.R2) {
        const float rinv = rsqrt_approx(r2);
        const float rs = rinv * S;
        const float ys = r2 * rs;
        if (ys < Yq) {
            ctr.add(2);
            const float n = hc.narrow ? nfw_N8(ys) : nfw_N16(ys);
            const float d = hc.narrow ? nfw_D8(ys) : nfw_D16(ys);
            m = fmaf(n * (rs * T), rcp_approx(d), -hc.invR3);
        } else {
            const float rinv2 = rinv * rinv;
            if (ys < hc.c) {
                ctr.add(3);
                const float sel = nfw_I_log(ys, fmaf(r2, rs, 1.0f)) * hc.invIc;
                m = fmaf(sel, rinv2 * rinv, -hc.invR3);
            } else {
                ctr.add(1);
                m = fmaf(rinv2, rinv, -hc.invR3);
            }
        }
    } else {
        ctr.add(0);
    }
    return m;
}

// FP64.  WARP: every lane of the warp is here (the integration loops), and the
// series' steps are run for the lane that needs most.
template <class Ctr = NoTally, bool WARP = true>
__device__ __forceinline__ double accel_m(double x, double y, double S, double Q, double,
                                          const HaloF64& hc, Ctr& ctr)
{
    const double r2 = fma(x, x, y * y);
    const bool in = less_nonneg(r2, hc.R2), nfw = in && less_nonneg(r2, Q);
    double m = 0.0, rinv = 0.0, ys = 0.0, t = 0.0, sel = 1.0;
    if (in) rinv = rsqrt(less_nonneg(r2, 1e-200) ? 1e-200 : r2);
    bool series = false;
    if (nfw) {
        ys = (r2 * rinv) * S;
        t = quotient(ys, 1.0 + ys);
        series = less_nonneg(t, 0.5);
    }
    const int J = series_steps(t);
    int J_max = series ? J : 0;
    if (WARP) J_max = __reduce_max_sync(0xffffffffu, J_max);
    if (in) {
        if (nfw) {
            ctr.add(ys < 1.0 ? 2 : 3);
            const double I = series ? (t * t) * nfw_series(t, J, J_max) : log1p(ys) - t;
            sel = I * hc.invIc;
        } else {
            ctr.add(1);
        }
        m = fma(sel, rinv * rinv * rinv, -hc.invR3);
    } else {
        ctr.add(0);
    }
    return m;
}

template <typename T> struct PrecTraits;
template <> struct PrecTraits<float> {
    using Halo = HaloF32;
    static __device__ __forceinline__ Halo halo(const DevProblem& P)
    {
        const float c = (float)P.c_nfw;
        return {(float)P.invIc, (float)P.invR3, (float)P.R2, (float)sqrt(P.R2), c, c <= kNarrowMaxC};
    }
};
template <> struct PrecTraits<double> {
    using Halo = HaloF64;
    static __device__ __forceinline__ Halo halo(const DevProblem& P)
    {
        return {P.invIc, P.invR3, P.R2, sqrt(P.R2)};
    }
};

// Initial distribution f(q) (Sec. II.C, Sec. IV.B), evaluated in FP64 in both
// precision modes (it runs once per trajectory and mass, in the epilogue).
// The tabulated kind is linear in ln q between log-spaced nodes (stored in
// FP64), the first value below the first node and 0 above the last.
__device__ __forceinline__ double relic_f_table(const DevProblem& P, double q)
{
    const double* t = reinterpret_cast<const double*>(P.ftab);
    const int n = P.n_ftab;
    if (!(q > P.ftab_q0)) return t[0];
    if (q > P.ftab_q1) return 0.0;
    const double u = log(q / P.ftab_q0) * P.ftab_scale;
    if (u >= (double)(n - 1)) return t[n - 1];
    const int k = (int)u;
    const double w = u - (double)k;
    return t[k] + w * (t[k + 1] - t[k]);
}

__device__ __forceinline__ double relic_f_dev(const DevProblem& P, double q)
{
    if (P.f_kind == NU_F_TABLE) return relic_f_table(P, q);
    if (P.f_kind == NU_F_FREEZEIN) {
        const double qq = fmax(q, 1e-300);
        return exp(-qq) / sqrt(qq);
    }
    return 1.0 / (1.0 + exp(q - P.f_p0));
}

__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

__device__ __forceinline__ float fmaT(float a, float b, float c) { return fmaf(a, b, c); }
__device__ __forceinline__ double fmaT(double a, double b, double c) { return fma(a, b, c); }

// One classical RK4 step of size -h for one trajectory (Eq. eoms in ln a).
// c points at the step's C_COUNT coefficients (see CoefSlot).  Every product-sum
// is an explicit fused multiply-add, so the packed two-trajectory variant
// below performs exactly the same roundings.
template <typename T, class Ctr>
__device__ __forceinline__ void rk4_step(T& x, T& y, T& vx, T& vy, const T* c,
                                         const typename PrecTraits<T>::Halo& hc, Ctr& ctr)
{
    const T m1 = accel_m(x, y, c[C_S0], c[C_Q0], c[C_T0], hc, ctr);
    const T p1 = c[C_B1] * m1;
    const T X2 = fmaT(c[C_MA1], vx, x), Y2 = fmaT(c[C_MA1], vy, y);
    const T VX2 = fmaT(p1, x, vx), VY2 = fmaT(p1, y, vy);

    const T m2 = accel_m(X2, Y2, c[C_S1], c[C_Q1], c[C_T1], hc, ctr);
    const T p2 = c[C_B2] * m2;
    const T X3 = fmaT(c[C_MA2], VX2, x), Y3 = fmaT(c[C_MA2], VY2, y);
    const T VX3 = fmaT(p2, X2, vx), VY3 = fmaT(p2, Y2, vy);

    const T m3 = accel_m(X3, Y3, c[C_S1], c[C_Q1], c[C_T1], hc, ctr);
    const T p3 = c[C_B3] * m3;
    const T X4 = fmaT(c[C_MA3], VX3, x), Y4 = fmaT(c[C_MA3], VY3, y);
    const T VX4 = fmaT(p3, X3, vx), VY4 = fmaT(p3, Y3, vy);

    const T m4 = accel_m(X4, Y4, c[C_S2], c[C_Q2], c[C_T2], hc, ctr);
    const T p4 = c[C_B4] * m4;

    // x' = x - (h/6) (A_a v + 2 A_m V2 + 2 A_m V3 + A_b V4)
    const T nx = fmaT(c[C_W2], VX4, fmaT(c[C_W1], VX2 + VX3, fmaT(c[C_W0], vx, x)));
    const T ny = fmaT(c[C_W2], VY4, fmaT(c[C_W1], VY2 + VY3, fmaT(c[C_W0], vy, y)));
    // v' = v + (h/6) (BF_a m1 x + 2 BF_m m2 X2 + 2 BF_m m3 X3 + BF_b m4 X4)
    const T p2x2 = p2 * T(2);   // exact doubling
    const T third = T(1) / T(3);
    const T tx = fmaT(p3, X3, fmaT(p2x2, X2, p1 * x));
    const T ty = fmaT(p3, Y3, fmaT(p2x2, Y2, p1 * y));
    const T nvx = fmaT(p4, X4, fmaT(tx, third, vx));
    const T nvy = fmaT(p4, Y4, fmaT(ty, third, vy));
    x = nx;
    y = ny;
    vx = nvx;
    vy = nvy;
}

// ---------------------------------------------------------------------------
// Packed FP32x2 path: two trajectories per thread held as register pairs, every
// arithmetic operation issued as one f32x2 instruction (fma/mul/add.rn.f32x2).
// Each component sees exactly the operations of the scalar path above, in the
// same order, so the results are bitwise those of the two-trajectory scalar
// kernel; only selects, comparisons and the special functions stay scalar.
// The coefficients come from the same table as the scalar path's, each widened
// to a pair in registers: a table with every value stored twice costs twice the
// loads and more spills (precision sweep, four masses: 6.79 ms with the doubled
// table and 38 B of spill stores, 6.41-6.50 ms with the plain one and 14 B).
// ---------------------------------------------------------------------------
struct f2 {
    unsigned long long v;
};

__device__ __forceinline__ f2 pk(float a, float b)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ float f2lo(f2 a)
{
    float l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(l), "=f"(h) : "l"(a.v));
    return l;
}
__device__ __forceinline__ float f2hi(f2 a)
{
    float l, h;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(l), "=f"(h) : "l"(a.v));
    return h;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 dup(float a) { return pk(a, a); }
// largest of three, NaN if one of them is NaN
__device__ __forceinline__ float max3_nan(float a, float b, float c)
{
    float r;
    asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
    return r;
}

__device__ __forceinline__ f2 rsqrt2(f2 a) { return pk(rsqrt_approx(f2lo(a)), rsqrt_approx(f2hi(a))); }
__device__ __forceinline__ f2 rcp2(f2 a) { return pk(rcp_approx(f2lo(a)), rcp_approx(f2hi(a))); }
__device__ __forceinline__ f2 rcp_neg2(f2 a) { return pk(rcp_approx(-f2lo(a)), rcp_approx(-f2hi(a))); }
__device__ __forceinline__ f2 lg2_2(f2 a) { return pk(lg2_approx(f2lo(a)), lg2_approx(f2hi(a))); }

struct HaloX2 {
    f2 invIc, neg_invR3;
    float R2, R, c;
};

// N(y) and D(y) of the rational g for both halves (see nfw_N16, nfw_D16 and nfw_N8,
// nfw_D8); NARROW selects the fit.
template <bool NARROW>
__device__ __forceinline__ f2 nfw_N(f2 y)
{
    f2 p;
    if constexpr (NARROW) {
        p = dup(-4.539978363e-06f);
        p = fma2(p, y, dup(4.568357544e-04f));
        p = fma2(p, y, dup(4.554858804e-02f));
        p = fma2(p, y, dup(3.421576917e-01f));
        p = fma2(p, y, dup(5.000000000e-01f));
    } else {
        p = dup(3.952767202e-06f);
        p = fma2(p, y, dup(2.387282439e-03f));
        p = fma2(p, y, dup(6.631398201e-02f));
        p = fma2(p, y, dup(3.795046508e-01f));
        p = fma2(p, y, dup(5.000000596e-01f));
    }
    return p;
}
template <bool NARROW>
__device__ __forceinline__ f2 nfw_D(f2 y)
{
    f2 p;
    if constexpr (NARROW) {
        p = dup(1.647129469e-02f);
        p = fma2(p, y, dup(2.829689085e-01f));
        p = fma2(p, y, dup(1.281258702e+00f));
        p = fma2(p, y, dup(2.017652512e+00f));
        p = fma2(p, y, dup(1.0f));
    } else {
        p = dup(5.989100318e-04f);
        p = fma2(p, y, dup(3.099172190e-02f));
        p = fma2(p, y, dup(3.629413843e-01f));
        p = fma2(p, y, dup(1.422382593e+00f));
        p = fma2(p, y, dup(2.092346668e+00f));
        p = fma2(p, y, dup(1.0f));
    }
    return p;
}

// Two force evaluations, one in each half of the pairs: accel_m (FP32) without
// branches, from r^2 on.
//   kRational   the value on the rational branch of the NFW part
//   kSelect     each half's own branch, where none is the logarithm: the bounds Yq
//               are c then, so no y lies between them and c
//   kSelectLog  each half's own branch
//   kOutside    each half's own branch outside the NFW part: the shell, beyond R
enum StepForm { kRational, kSelect, kSelectLog, kOutside };

template <StepForm FORM>
__device__ __forceinline__ float branch_of(float r2, float ys, float Yq, float R2, float c, float mq,
                                           float ml, float ms)
{
    const float mn = FORM == kSelectLog && ys < c ? ml : ms;
    return ys < Yq ? mq : r2 < R2 ? mn : 0.0f;
}

template <bool NARROW, StepForm FORM>
__device__ __forceinline__ f2 m_form(f2 r2, f2 S, float Yq0, float Yq1, f2 T, const HaloX2& hc, f2& ys)
{
    const f2 rinv = rsqrt2(r2);
    const f2 rs = mul2(rinv, S);
    ys = mul2(r2, rs);
    if constexpr (FORM == kOutside) {
        const f2 ms = fma2(mul2(rinv, rinv), rinv, hc.neg_invR3);
        return pk(f2lo(r2) < hc.R2 ? f2lo(ms) : 0.0f, f2hi(r2) < hc.R2 ? f2hi(ms) : 0.0f);
    }
    const f2 mq = fma2(mul2(nfw_N<NARROW>(ys), mul2(rs, T)), rcp2(nfw_D<NARROW>(ys)), hc.neg_invR3);
    if constexpr (FORM == kRational) return mq;
    const f2 rinv2 = mul2(rinv, rinv);
    const f2 ms = fma2(rinv2, rinv, hc.neg_invR3);
    f2 ml = ms;
    if constexpr (FORM == kSelectLog) {
        const f2 u = fma2(r2, rs, dup(1.0f));
        const f2 I = fma2(lg2_2(u), dup(0.693147180559945309f), mul2(ys, rcp_neg2(u)));
        ml = fma2(mul2(I, hc.invIc), mul2(rinv2, rinv), hc.neg_invR3);
    }
    return pk(branch_of<FORM>(f2lo(r2), f2lo(ys), Yq0, hc.R2, hc.c, f2lo(mq), f2lo(ml), f2lo(ms)),
              branch_of<FORM>(f2hi(r2), f2hi(ys), Yq1, hc.R2, hc.c, f2hi(mq), f2hi(ml), f2hi(ms)));
}

// One RK4 step of a lane's trajectories: every value is formed by the operations of
// rk4_step.  The four force evaluations run as two independent pairs: within a step
// the positions of the first two stages depend only on its start state, and those
// of the last two on it and the first pair's forces.
// A kRational step returns false and leaves the state as it was where a lane of the
// warp is on another branch, found out with one vote near the step's end: the
// bounds of the four evaluations do not rise from stage to stage (S falls with z),
// so the largest y against the last stage's bound decides, and a NaN (r^2 out of
// range, far beyond R) decides against it.  A kOutside step does the same where a lane
// is in the NFW part (y < c, the least y decides, NaNs passed over).  Other steps clear
// `rational` where this lane's last evaluation was on another branch.
//
// Two trajectories of a lane: the halves of every pair are theirs.
template <bool OUTSIDE>                                // with kOutside steps
struct TwoTrajectories {
    static constexpr bool kOutsideSteps = OUTSIDE;
    f2 x, y, vx, vy;
    __device__ __forceinline__ void begin(const float4*) {}
    __device__ __forceinline__ TwoTrajectories(const float* x_, const float* y_, const float* vx_,
                                               const float* vy_)
        : x(pk(x_[0], x_[1])), y(pk(y_[0], y_[1])), vx(pk(vx_[0], vx_[1])), vy(pk(vy_[0], vy_[1]))
    {
    }
    __device__ __forceinline__ void store(float* x_, float* y_, float* vx_, float* vy_) const
    {
        x_[0] = f2lo(x); x_[1] = f2hi(x);
        y_[0] = f2lo(y); y_[1] = f2hi(y);
        vx_[0] = f2lo(vx); vx_[1] = f2hi(vx);
        vy_[0] = f2lo(vy); vy_[1] = f2hi(vy);
    }
    // Whether every active trajectory of this lane is finished (see escapes).
    __device__ __forceinline__ bool finished(const bool* act, const HaloX2& hc, float irem) const
    {
        const f2 r2 = fma2(x, x, mul2(y, y));
        const f2 dot = fma2(x, vx, mul2(y, vy));
        const f2 v2 = fma2(vx, vx, mul2(vy, vy));
        return (!act[0] || escapes(f2lo(r2), f2lo(dot), f2lo(v2), hc.R2, hc.R, irem)) &&
               (!act[1] || escapes(f2hi(r2), f2hi(dot), f2hi(v2), hc.R2, hc.R, irem));
    }
    // Whether both trajectories are out of the NFW part, to the rounding: r S >= c.
    __device__ __forceinline__ bool outside(float S, const HaloX2& hc) const
    {
        const f2 r2 = fma2(x, x, mul2(y, y));
        const float S2 = S * S, c2 = hc.c * hc.c;
        return !(f2lo(r2) * S2 < c2) && !(f2hi(r2) * S2 < c2);
    }
    template <bool NARROW, StepForm FORM>
    __device__ __forceinline__ bool step(const float4* row, const float4*, const HaloX2& hc, bool& rational)
    {
        auto r2 = [](f2 a, f2 b) { return fma2(a, a, fma2(b, b, dup(kR2Guard))); };
        const float4 q0 = row[0];                    // MA1 MA2 MA3 W0
        const f2 MA1 = dup(q0.x), MA2 = dup(q0.y), MA3 = dup(q0.z), W0 = dup(q0.w);
        const f2 X2 = fma2(MA1, vx, x), Y2 = fma2(MA1, vy, y);
        const float4 q2 = row[2];                    // W1 W2 S0 S1
        const float4 q3 = row[3];                    // S2 Q0 Q1 Q2
        const float4 q4 = row[4];                    // T0 T1 T2 IREM
        const f2 S1 = dup(q2.w), T1 = dup(q4.y);
        f2 y1, y2, y3, y4;
        const f2 m1 = m_form<NARROW, FORM>(r2(x, y), dup(q2.z), q3.y, q3.y, dup(q4.x), hc, y1);
        const f2 m2 = m_form<NARROW, FORM>(r2(X2, Y2), S1, q3.z, q3.z, T1, hc, y2);
        const float4 q1 = row[1];                    // B1 B2 B4 B3
        const f2 p1 = mul2(dup(q1.x), m1);
        const f2 VX2 = fma2(p1, x, vx), VY2 = fma2(p1, y, vy);
        const f2 p2 = mul2(dup(q1.y), m2);
        const f2 VX3 = fma2(p2, X2, vx), VY3 = fma2(p2, Y2, vy);
        const f2 X3 = fma2(MA2, VX2, x), Y3 = fma2(MA2, VY2, y);
        const f2 X4 = fma2(MA3, VX3, x), Y4 = fma2(MA3, VY3, y);

        const f2 m3 = m_form<NARROW, FORM>(r2(X3, Y3), S1, q3.z, q3.z, T1, hc, y3);
        const f2 m4 = m_form<NARROW, FORM>(r2(X4, Y4), dup(q3.x), q3.w, q3.w, dup(q4.z), hc, y4);
        if constexpr (FORM == kRational) {
            const float a = max3_nan(f2lo(y1), f2hi(y1), f2lo(y2));
            const float b = max3_nan(f2hi(y2), f2lo(y3), f2hi(y3));
            const float y_max = max3_nan(max3_nan(a, b, f2lo(y4)), f2hi(y4), f2hi(y4));
            if (!__all_sync(0xffffffffu, y_max < q3.w)) return false;
        } else if constexpr (FORM == kOutside) {
            const float a = fminf(fminf(f2lo(y1), f2hi(y1)), fminf(f2lo(y2), f2hi(y2)));
            const float b = fminf(fminf(f2lo(y3), f2hi(y3)), fminf(f2lo(y4), f2hi(y4)));
            if (__any_sync(0xffffffffu, fminf(a, b) < hc.c)) return false;
        } else {
            rational = rational && f2lo(y4) < q3.w && f2hi(y4) < q3.w;
        }

        const f2 W1 = dup(q2.x), W2 = dup(q2.y);
        const f2 p3 = mul2(dup(q1.w), m3);
        const f2 VX4 = fma2(p3, X3, vx), VY4 = fma2(p3, Y3, vy);
        const f2 p4 = mul2(dup(q1.z), m4);
        const f2 nx = fma2(W2, VX4, fma2(W1, add2(VX2, VX3), fma2(W0, vx, x)));
        const f2 ny = fma2(W2, VY4, fma2(W1, add2(VY2, VY3), fma2(W0, vy, y)));
        const f2 p2x2 = mul2(p2, dup(2.0f));         // exact doubling
        const f2 third = dup(1.0f / 3.0f);
        const f2 tx = fma2(p3, X3, fma2(p2x2, X2, mul2(p1, x)));
        const f2 ty = fma2(p3, Y3, fma2(p2x2, Y2, mul2(p1, y)));
        vx = fma2(p4, X4, fma2(tx, third, vx));
        vy = fma2(p4, Y4, fma2(ty, third, vy));
        x = nx;
        y = ny;
        return true;
    }
};

// One trajectory of a lane: the halves of a position or velocity are its x and y,
// and those of a force evaluation the two stages of a pair (1 and 2, then 4 and 3).
// So a step takes few more instructions than half of two trajectories' step, which
// is what a scheduler with few warps is bound by.
struct OneTrajectory {
    static constexpr bool kOutsideSteps = false;
    f2 r, v;
    float ma1;                                       // the next step's C_MA1, read a step ahead
    __device__ __forceinline__ void begin(const float4* row) { ma1 = row[0].x; }
    __device__ __forceinline__ OneTrajectory(const float* x, const float* y, const float* vx,
                                             const float* vy)
        : r(pk(x[0], y[0])), v(pk(vx[0], vy[0]))
    {
    }
    __device__ __forceinline__ void store(float* x, float* y, float* vx, float* vy) const
    {
        x[0] = f2lo(r); y[0] = f2hi(r);
        vx[0] = f2lo(v); vy[0] = f2hi(v);
    }
    __device__ __forceinline__ bool finished(const bool* act, const HaloX2& hc, float irem) const
    {
        const float x = f2lo(r), y = f2hi(r), vx = f2lo(v), vy = f2hi(v);
        return !act[0] || escapes(fmaf(x, x, y * y), fmaf(x, vx, y * vy), fmaf(vx, vx, vy * vy), hc.R2,
                                  hc.R, irem);
    }
    template <bool NARROW, StepForm FORM>
    __device__ __forceinline__ bool step(const float4* row, const float4* next, const HaloX2& hc,
                                         bool& rational)
    {
        const f2 R2 = fma2(dup(ma1), v, r);
        const float ma1_next = next[0].x;
        auto r2 = [](f2 a, f2 b) { return pk(guarded_r2(f2lo(a), f2hi(a)), guarded_r2(f2lo(b), f2hi(b))); };
        const float4 q0 = row[0], q1 = row[1], q2 = row[2], q3 = row[3], q4 = row[4];
        f2 y12, y43;
        const f2 m12 = m_form<NARROW, FORM>(r2(r, R2), pk(q2.z, q2.w), q3.y, q3.z, pk(q4.x, q4.y), hc, y12);
        const f2 p12 = mul2(pk(q1.x, q1.y), m12);
        const f2 p1 = dup(f2lo(p12)), p2 = dup(f2hi(p12));
        const f2 V2 = fma2(p1, r, v);
        const f2 V3 = fma2(p2, R2, v);
        const f2 R3 = fma2(dup(q0.y), V2, r);
        const f2 R4 = fma2(dup(q0.z), V3, r);
        const f2 m43 = m_form<NARROW, FORM>(r2(R4, R3), pk(q3.x, q2.w), q3.w, q3.z, pk(q4.z, q4.y), hc, y43);
        if constexpr (FORM == kRational) {
            const float y_max = max3_nan(max3_nan(f2lo(y12), f2hi(y12), f2lo(y43)), f2hi(y43), f2hi(y43));
            if (!__all_sync(0xffffffffu, y_max < q3.w)) return false;
        } else {
            rational = rational && f2lo(y43) < q3.w;
        }
        const f2 p43 = mul2(pk(q1.z, q1.w), m43);
        const f2 p3 = dup(f2hi(p43)), p4 = dup(f2lo(p43));
        const f2 V4 = fma2(p3, R3, v);
        const f2 nr = fma2(dup(q2.y), V4, fma2(dup(q2.x), add2(V2, V3), fma2(dup(q0.w), v, r)));
        const f2 t = fma2(p3, R3, fma2(dup(f2hi(p12) * 2.0f), R2, mul2(p1, r)));
        v = fma2(p4, R4, fma2(t, dup(1.0f / 3.0f), v));
        r = nr;
        ma1 = ma1_next;
        return true;
    }
};

// A warp's window on the coefficient table: two buffers of rows in shared memory,
// one filled by asynchronous copies while the steps of the other run.  Read in
// place, a table row costs its first reader on an SM a wait for L2, with all of a
// step behind it.
constexpr int kRow16 = C_COUNT / 4;                  // 16-byte words of an FP32 row; FP64 twice
constexpr int kRingSteps = 32;                       // FP32 rows of a buffer; FP64 half
constexpr int kRing16 = 2 * kRingSteps * kRow16;     // 16-byte words of a warp's two buffers

__device__ __forceinline__ void copy16_async(float4* dst, const float4* src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     (unsigned)__cvta_generic_to_shared(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int PENDING>
__device__ __forceinline__ void copies_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(PENDING) : "memory");
}

// Copy the rows of ROW words from `first` on, none past s_end, into a buffer.
template <int ROW>
__device__ __forceinline__ void ring_fill(float4* half, const float4* tab, int first, int s_end,
                                          int lane)
{
    const int n16 = min(kRing16 / 2 / ROW, s_end - first) * ROW;
    for (int i = lane; i < n16; i += 32) copy16_async(half + i, tab + (size_t)first * ROW + i);
    copies_commit();
}

// Run body(rows, count) over steps [s_begin, s_end) in windows of a buffer's
// rows until it returns false.  Warp-uniform; all copies are done on return, so
// the buffers can be filled again.
template <int ROW, class Body>
__device__ __forceinline__ void over_ring(float4* ring, const float4* tab, int s_begin, int s_end,
                                          int lane, Body body)
{
    constexpr int kSteps = kRing16 / 2 / ROW;
    ring_fill<ROW>(ring, tab, s_begin, s_end, lane);
    ring_fill<ROW>(ring + kRing16 / 2, tab, s_begin + kSteps, s_end, lane);
    float4* half = ring;
    for (int first = s_begin; first < s_end; first += kSteps) {
        copies_wait<1>();                            // this half has arrived
        __syncwarp();
        if (!body(half, min(kSteps, s_end - first))) break;
        __syncwarp();                                // every lane has read it
        ring_fill<ROW>(half, tab, first + 2 * kSteps, s_end, lane);
        half = half == ring ? ring + kRing16 / 2 : ring;
    }
    copies_wait<0>();
    __syncwarp();
}

// The FP32 step loop of one warp for steps [s_begin, s_end).  NARROW is fixed per
// request (the rational fit its force uses), so the tile chooses the loop once.
//
// With many warps it is bound by register operands and issue: a packed fused
// multiply-add with three different register pairs takes 3 cycles of a scheduler,
// one with a constant operand 2, each other instruction about one more (measured
// with independent chains), and 97 of a packed step's 145 instructions are such
// operations.  With one warp on a scheduler it is bound by that warp's own issue
// (a scalar fused multiply-add every 2 cycles) and the chain of a step.  So the
// instructions of a step count, and no step has more than one vote, off the chain,
// and no branch but its.
// A warp whose lanes all stay on the rational branch runs kRational steps, without
// selects and without the exit test (no lane of it is beyond R).  Where one fails
// it is done again in a form that lets each lane select its branch, and so are the
// following steps: every kSelectEvery of them the warp stops if its lanes are all
// finished, and goes back to kRational steps if they were all on that branch.  With two
// trajectories a lane it takes kOutside steps, half the work, while they are all out of
// the NFW part: precision sweep 5.61 -> 5.37 ms, uneven batch 25.9 -> 25.2, 614,000
// trajectories from beyond R 0.45 -> 0.31 (0.36 in a kernel that skips the force by
// branches).  Where the chain of a step counts, the loop is faster without: one trajectory
// a lane (plain profile 97 us against 104), and up to three CTAs of two on an SM
// (kPackedFew: 12,000 to 38,000 trajectories 109 us against 120-125, 76,000 145-149 against
// 155-164, 114,000 200-207 against 206-215; from four on there is no difference).
// Evaluating the branches of such a warp by votes and warp-uniform paths took 1900
// cycles a step on one scheduler, selecting takes 479 (412 one trajectory a lane).
constexpr int kSelectEvery = 8;

template <bool NARROW, class State>
__device__ __forceinline__ void step_loop(State& s, const float4* tab, int s_begin, int s_end,
                                          const bool* act, bool done, const HaloX2& hc, float4* ring,
                                          int lane)
{
    if (__all_sync(0xffffffffu, done)) return;
    bool rational = true;
    bool select = false;             // the warp runs steps that select
    int k_select = 0;
    over_ring<kRow16>(ring, tab, s_begin, s_end, lane, [&](const float4* rows, int count) {
        const float4* const end = rows + count * kRow16;
        // a bound below c, which comes last in the window first: c > 16, or an NFW
        // edge that lies beyond R
        const bool logarithm = end[3 - kRow16].w < hc.c;
        auto next = [&] { return rows + kRow16 < end ? rows + kRow16 : rows; };
        s.begin(rows);
        while (rows < end) {
            if (!select) {
                for (; rows < end; rows += kRow16)
                    if (!s.template step<NARROW, kRational>(rows, next(), hc, rational)) break;
                if (rows >= end) break;
                select = true;
                k_select = 0;
                rational = false;
            }
            if ((k_select++ & (kSelectEvery - 1)) == 0) {
                done |= s.finished(act, hc, rows[C_IREM / 4].w);
                if (__all_sync(0xffffffffu, done)) return false;
                select = !__all_sync(0xffffffffu, rational);
                rational = true;
                if constexpr (State::kOutsideSteps) {
                    if (__all_sync(0xffffffffu, s.outside(rows[C_S0 / 4].z, hc))) {
                        int n = 0;
                        while (n < kSelectEvery && rows < end &&
                               s.template step<NARROW, kOutside>(rows, next(), hc, rational)) {
                            rows += kRow16;
                            ++n;
                        }
                        if (n == kSelectEvery || rows >= end) {
                            select = true;
                            rational = false;
                            k_select = 0;
                            continue;
                        }
                    }
                }
            }
            if (logarithm)
                s.template step<NARROW, kSelectLog>(rows, next(), hc, rational);
            else
                s.template step<NARROW, kSelect>(rows, next(), hc, rational);
            rows += kRow16;
        }
        return true;
    });
}

// ---------------------------------------------------------------------------
// FP64 step loop: rk4_step with its force evaluations in two independent pairs.  The
// values are those of accel_m; what differs is which lanes compute them.  With one
// warp on a scheduler the pair's chains fill each other's waits, and where the lanes
// of a warp lie on both sides of y = 1, which most warps' do at some steps, the
// evaluations of the pair that need the series are gathered into one pass over the
// warp if they are 32 or fewer, and those that need the logarithm likewise.
// ---------------------------------------------------------------------------
// (A value's series length goes with it into a pass: found again there it would lengthen
// the chain, 25.5 ms instead of 25.15 for six radii of the precision sweep.)
struct PassBuffer {
    double v[32];
    int k[32];
};
struct Compact {                                     // a pair's evaluations that need a pass
    unsigned a, b, below;                            // their lanes; the lanes below this one
    __device__ __forceinline__ Compact(bool need_a, bool need_b, int lane)
        : a(__ballot_sync(0xffffffffu, need_a)), b(__ballot_sync(0xffffffffu, need_b)),
          below((1u << lane) - 1u)
    {
    }
    __device__ __forceinline__ int count() const { return __popc(a) + __popc(b); }
    __device__ __forceinline__ bool one_pass() const { return a && b && count() <= 32; }
    __device__ __forceinline__ int slot_a() const { return __popc(a & below); }
    __device__ __forceinline__ int slot_b() const { return __popc(a) + __popc(b & below); }
    // f(va, ka) where need_a and f(vb, kb) where need_b, in one pass (one_pass())
    template <class F>
    __device__ __forceinline__ void pass(bool need_a, bool need_b, double& va, double& vb, int ka, int kb,
                                         PassBuffer& buf, int lane, F f) const
    {
        if (need_a) {
            buf.v[slot_a()] = va;
            buf.k[slot_a()] = ka;
        }
        if (need_b) {
            buf.v[slot_b()] = vb;
            buf.k[slot_b()] = kb;
        }
        __syncwarp();
        const int from = lane < count() ? lane : 0;
        const double r = f(buf.v[from], buf.k[from]);
        __syncwarp();
        buf.v[lane] = r;
        __syncwarp();
        if (need_a) va = buf.v[slot_a()];
        if (need_b) vb = buf.v[slot_b()];
        __syncwarp();
    }
};

__device__ __forceinline__ void accel_pair(double xa, double ya, double Sa, double Qa, double xb,
                                           double yb, double Sb, double Qb, const HaloF64& hc,
                                           PassBuffer& buf, int lane, double& ma, double& mb)
{
    const unsigned full = 0xffffffffu;
    const double r2a = fma(xa, xa, ya * ya), r2b = fma(xb, xb, yb * yb);
    const bool in_a = less_nonneg(r2a, hc.R2), in_b = less_nonneg(r2b, hc.R2);
    ma = mb = 0.0;
    if (!__any_sync(full, in_a || in_b)) return;
    const double rinva = rsqrt(less_nonneg(r2a, 1e-200) ? 1e-200 : r2a);
    const double rinvb = rsqrt(less_nonneg(r2b, 1e-200) ? 1e-200 : r2b);
    const bool nfw_a = in_a && less_nonneg(r2a, Qa), nfw_b = in_b && less_nonneg(r2b, Qb);
    double sela = 1.0, selb = 1.0;
    if (__any_sync(full, nfw_a || nfw_b)) {
        const double ysa = (r2a * rinva) * Sa, ysb = (r2b * rinvb) * Sb;
        const double ta = quotient(ysa, 1.0 + ysa), tb = quotient(ysb, 1.0 + ysb);
        const bool sa = nfw_a && less_nonneg(ta, 0.5), sb = nfw_b && less_nonneg(tb, 0.5);
        const bool la = nfw_a && !sa, lb = nfw_b && !sb;
        double Ia = ta, Ib = tb;
        const Compact cs(sa, sb, lane);
        if (cs.a | cs.b) {
            const int Ja = series_steps(ta), Jb = series_steps(tb);
            const int J_max = __reduce_max_sync(full, max(sa ? Ja : 0, sb ? Jb : 0));
            if (cs.one_pass()) {
                cs.pass(sa, sb, Ia, Ib, Ja, Jb, buf, lane,
                        [&](double t, int J) { return (t * t) * nfw_series(t, J, J_max); });
            } else if (cs.a && cs.b) {
                double pa, pb;
                nfw_series2(ta, tb, Ja, Jb, J_max, pa, pb);
                Ia = (ta * ta) * pa;
                Ib = (tb * tb) * pb;
            } else if (cs.a) {
                Ia = (ta * ta) * nfw_series(ta, Ja, J_max);
            } else {
                Ib = (tb * tb) * nfw_series(tb, Jb, J_max);
            }
        }
        const Compact cl(la, lb, lane);
        if (cl.a | cl.b) {
            double ga = ysa, gb = ysb;
            if (cl.one_pass()) {
                cl.pass(la, lb, ga, gb, 0, 0, buf, lane, [](double v, int) { return log1p(v); });
            } else {
                if (cl.a) ga = log1p(ysa);
                if (cl.b) gb = log1p(ysb);
            }
            if (la) Ia = ga - ta;
            if (lb) Ib = gb - tb;
        }
        if (nfw_a) sela = Ia * hc.invIc;
        if (nfw_b) selb = Ib * hc.invIc;
    }
    if (in_a) ma = fma(sela, rinva * rinva * rinva, -hc.invR3);
    if (in_b) mb = fma(selb, rinvb * rinvb * rinvb, -hc.invR3);
}

// The loop of one warp.  pair(x, y, S, Q, X, Y, S', Q', m, m') evaluates the forces of
// two points.
template <class Pair>
__device__ __forceinline__ void fp64_loop(double& x, double& y, double& vx, double& vy,
                                          const float4* tab, int s_begin, int s_end, bool done,
                                          const HaloF64& hc, float4* ring, int lane, Pair pair)
{
    if (__all_sync(0xffffffffu, done)) return;
    int k = 0;
    over_ring<2 * kRow16>(ring, tab, s_begin, s_end, lane, [&](const float4* rows, int count) {
        for (int i = 0; i < count; ++i) {
            const double* c = reinterpret_cast<const double*>(rows + i * 2 * kRow16);
            if ((k++ & (kSelectEvery - 1)) == 0) {
                done |= escapes(fma(x, x, y * y), fma(x, vx, y * vy), fma(vx, vx, vy * vy), hc.R2, hc.R,
                                c[C_IREM]);
                if (__all_sync(0xffffffffu, done)) return false;
            }
            const double X2 = fma(c[C_MA1], vx, x), Y2 = fma(c[C_MA1], vy, y);
            double m1, m2;
            pair(x, y, c[C_S0], c[C_Q0], X2, Y2, c[C_S1], c[C_Q1], m1, m2);
            const double p1 = c[C_B1] * m1;
            const double VX2 = fma(p1, x, vx), VY2 = fma(p1, y, vy);
            const double p2 = c[C_B2] * m2;
            const double VX3 = fma(p2, X2, vx), VY3 = fma(p2, Y2, vy);
            const double X3 = fma(c[C_MA2], VX2, x), Y3 = fma(c[C_MA2], VY2, y);
            const double X4 = fma(c[C_MA3], VX3, x), Y4 = fma(c[C_MA3], VY3, y);
            double m3, m4;
            pair(X3, Y3, c[C_S1], c[C_Q1], X4, Y4, c[C_S2], c[C_Q2], m3, m4);
            const double p3 = c[C_B3] * m3;
            const double VX4 = fma(p3, X3, vx), VY4 = fma(p3, Y3, vy);
            const double p4 = c[C_B4] * m4;
            const double nx = fma(c[C_W2], VX4, fma(c[C_W1], VX2 + VX3, fma(c[C_W0], vx, x)));
            const double ny = fma(c[C_W2], VY4, fma(c[C_W1], VY2 + VY3, fma(c[C_W0], vy, y)));
            const double p2x2 = p2 * 2.0;            // exact doubling
            const double third = 1.0 / 3.0;
            const double tx = fma(p3, X3, fma(p2x2, X2, p1 * x));
            const double ty = fma(p3, Y3, fma(p2x2, Y2, p1 * y));
            vx = fma(p4, X4, fma(tx, third, vx));
            vy = fma(p4, Y4, fma(ty, third, vy));
            x = nx;
            y = ny;
        }
        return true;
    });
}

// The pairs of a small launch, whose warps leave half of the schedulers without one:
// two warps integrate the same trajectories, each evaluates one point of a pair and
// hands it to the other.  They hold the same state, so they meet at every barrier.
struct SplitPair {
    const HaloF64& hc;
    double* shared;                                  // [2][2][32]: pairs in turn, points
    int barrier, role, lane, turn;
    __device__ __forceinline__ void operator()(double xa, double ya, double Sa, double Qa, double xb,
                                               double yb, double Sb, double Qb, double& ma, double& mb)
    {
        NoTally none;
        const double m = role ? accel_m(xb, yb, Sb, Qb, 0.0, hc, none) : accel_m(xa, ya, Sa, Qa, 0.0, hc, none);
        double* at = shared + turn * 64;
        at[role * 32 + lane] = m;
        asm volatile("bar.sync %0, 64;" ::"r"(barrier) : "memory");
        ma = at[lane];
        mb = at[32 + lane];
        turn ^= 1;       // written again only after the next pair's barrier, past these reads
    }
};

// ---------------------------------------------------------------------------
// Work queue of a resident launch (see QueueCtl).  Thread 0 of a CTA has
// claimed tile g; it returns g once the host has published it, or -1 when the
// launch ends: the queue was closed (or has expired) with g beyond its last
// published tile, or this CTA's wait ran past the limit and it expired the
// queue itself (by compare-and-swap on the same word the host publishes
// through, so the tile it gave up on can never be published afterwards).
// ---------------------------------------------------------------------------
__device__ __forceinline__ unsigned long long load_acquire_sys(const unsigned long long* p)
{
    unsigned long long v;
    asm volatile("ld.acquire.sys.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned load_acquire_sys(const unsigned* p)
{
    unsigned v;
    asm volatile("ld.acquire.sys.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ unsigned long long globaltimer_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ int queue_wait(QueueCtl* q, unsigned g, int* n_probs)
{
    const unsigned long long t0 = globaltimer_ns();
    bool asked = false;
    for (;;) {
        const unsigned long long w = load_acquire_sys(&q->word);
        const unsigned published = (unsigned)w;
        if (g < published) {
            *n_probs = (int)load_acquire_sys(&q->n_probs);
            return (int)g;
        }
        if ((unsigned)(w >> 32) != kQueueOpen) return -1;
        if (!asked) {
            atomicExch_system(&q->want_work, 1u);
            asked = true;
        }
        if (globaltimer_ns() - t0 > q->wait_limit_ns) {
            const unsigned long long expired = ((unsigned long long)kQueueExpired << 32) | published;
            if (atomicCAS_system(&q->word, w, expired) == w) return -1;
            continue;                          // the host changed the word: look again
        }
        __nanosleep(2000);
    }
}

// Sum of a tile's weighted f values, in an order that depends on the trajectories
// alone: each 64 consecutive ones form a unit, whose lanes add the two halves and
// are then summed by a shuffle tree; units are added by fours, in pairs, and the
// fours of a tile in order.  So every kernel and every split of a request's tiles
// into ones of a unit, two or four gives the same bits.
constexpr int kUnit = 64;

// Sums over the warp of N values a lane (2 kMassGroup), each by warp_sum's tree: at every
// level the lanes of one half hand over the values that the other half goes on with,
// so 8 sums take 9 FP64 additions a lane where one after another they take 40.
// Lane l returns the sum of value l N / 32.
template <int N>
__device__ __forceinline__ double warp_sums(double (&v)[N], int lane)
{
    int step = 16;
#pragma unroll
    for (int n = N / 2; n >= 1; n /= 2, step /= 2) {
        const bool upper = (lane & step) != 0;
#pragma unroll
        for (int j = 0; j < n; ++j) {
            const double give = upper ? v[j] : v[j + n], keep = upper ? v[j + n] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, step);
        }
    }
    double sum = v[0];
#pragma unroll
    for (; step >= 1; step /= 2) sum += __shfl_xor_sync(0xffffffffu, sum, step);
    return sum;
}

// Sum of n (1, 2 or 4) values of a four, those from `have` on being absent.
template <class Load>
__device__ __forceinline__ double sum_of_four(int n, int have, Load load)
{
    auto at = [&](int i) { return i < n && i < have ? load(i) : 0.0; };   // + 0.0 is exact
    return (at(0) + at(1)) + (at(2) + at(3));
}

// Work of one launch: CTAs of a persistent grid claim tiles of `P.tile`
// consecutive trajectories of one radius and integrate them in passes of
// blockDim.x * TPT.  The step loop:
//   kLoopPacked  two trajectories per thread in packed FP32x2, 24 warps per SM (80
//                registers, 5.37 ms on the precision sweep of four masses; 5.61 without
//                kOutside steps; before that and the coefficients' being read ahead 5.75
//                ms, 5.95 with 64 registers, which spill, and 5.74 with 96 and 20 warps,
//                but the uneven batch 27.5 against 27.0 ms);
//   kLoopPackedFew  the same without kOutside steps, for few CTAs on an SM (step_loop);
//   kLoopPackedPasses  kLoopPacked for tiles of more trajectories than a CTA holds
//                (whole_tiles);
//   kLoopRing    one trajectory per thread, for small launches (plan_shape);
//   kLoopRingMasses  the same with an epilogue that takes kMassGroup masses at a time,
//                for launches in which a request reads several: f and its sums in FP64
//                were a fifth of the kernel at 15 masses.  20 radii x 6400 trajectories
//                x 300 steps: 301 -> 261 us with 15 masses, 220 -> 204 with 8, 185 ->
//                177 with 4, the same with 2; the paper's production grid 281 -> 272.
//                For one mass kLoopRing stays (relic-table profile 237 against 243 us);
//                groups of 8 take 263 us on the paper's grid but 102 against 97 us for
//                4 masses of 128,000 short trajectories; two trajectories a lane would
//                spill (precision sweep 5.61 -> 5.79 ms);
//   kLoopFp64    one trajectory per thread;
//   kLoopFp64Split  one trajectory in a lane of two warps (SplitPair): CTAs of four
//                warps and 64 trajectories;
//   kLoopGeneral one trajectory after another with the general force: the counting
//                variant of either mode.
enum StepLoop { kLoopGeneral, kLoopPacked, kLoopPackedFew, kLoopPackedPasses, kLoopRing, kLoopRingMasses,
                kLoopFp64, kLoopFp64Split };
constexpr int kRingThreads = 128;
constexpr int kMassGroup = 4;
template <StepLoop LOOP> constexpr bool kTwo =
    LOOP == kLoopPacked || LOOP == kLoopPackedFew || LOOP == kLoopPackedPasses;

__device__ __forceinline__ int warp_id() { return threadIdx.x >> 5; }

template <typename T, int TPT, bool COUNT, StepLoop LOOP>
__global__ void __launch_bounds__(LOOP == kLoopGeneral ? 512
                                  : LOOP == kLoopRing || LOOP == kLoopRingMasses ? kRingThreads : 256,
                                  kTwo<LOOP> ? 3 : 1)
traj_kernel(const DevProblem* __restrict__ probs, const int* __restrict__ tile_prefix,
            int n_probs, int n_tiles, unsigned* __restrict__ ctrl,
            unsigned long long* __restrict__ tallies, QueueCtl* queue)
{
    using Ctr = typename std::conditional<COUNT, Tally, NoTally>::type;
    Ctr ctr;
    __shared__ int s_tile;
    __shared__ int s_req;
    __shared__ int s_last;
    // the descriptor of the tile's request, read through L2 (requests published
    // into a resident launch are never served from a stale L1 line)
    __shared__ __align__(16) DevProblem s_prob;
    // unit sums of a pass; with one trajectory per thread a unit is two warps, and
    // the second hands its lanes' values to the first
    constexpr int kMasses = LOOP == kLoopRingMasses ? kMassGroup : 1;   // of an epilogue's pass
    __shared__ double s_red[16][2 * kMasses];
    __shared__ double s_half[TPT == 1 ? (kMasses > 1 ? 2 : 8) : 1][2 * kMasses][32];
    __shared__ double s_pair[LOOP == kLoopFp64Split ? 8 : 1][32];
    __shared__ PassBuffer s_pass[LOOP == kLoopFp64 ? 8 : 1];
    // kRing16 words a warp (not kLoopGeneral).  From 16 bytes past a multiple of 32 on the
    // copies into it take longer, seen where little else is done: 614,000 trajectories
    // without a halo 111 us, 83 at 32 and 64 bytes, 76 at 128.
    extern __shared__ __align__(128) float4 s_ring[];
    float4* ring = s_ring + warp_id() * kRing16;

    const int lane = threadIdx.x & 31;
    const int warp = warp_id();
    const int n_warps = blockDim.x >> 5;
    constexpr bool kSplit = LOOP == kLoopFp64Split;
    const int group = kSplit ? warp & 1 : warp;      // of 32 trajectories of a thread's slot
    // trajectory of slot i of this thread within a pass
    auto slot = [&](int i) { return (group * TPT + i) * 32 + lane; };

    for (;;) {
        if (threadIdx.x == 0) {
            const unsigned claimed = atomicAdd(&ctrl[kCtrlNext], 1u);
            int np = n_probs;
            int t = queue ? queue_wait(queue, claimed, &np)
                          : (claimed < (unsigned)n_tiles ? (int)claimed : -1);
            // request that owns global tile t: last p with tile_prefix[p] <= t
            if (t >= 0) {
                int lo = 0, hi = np - 1;
                while (lo < hi) {
                    const int mid = (lo + hi + 1) >> 1;
                    if (__ldcg(&tile_prefix[mid]) <= t) lo = mid; else hi = mid - 1;
                }
                s_req = lo;
            }
            s_tile = t;
        }
        __syncthreads();
        const int g = s_tile;
        if (g < 0) break;
        const int lo = s_req;
        {
            constexpr int kWords = (int)(sizeof(DevProblem) / sizeof(unsigned));
            static_assert(sizeof(DevProblem) % sizeof(unsigned) == 0, "descriptor words");
            const unsigned* src = reinterpret_cast<const unsigned*>(probs + lo);
            unsigned* dst = reinterpret_cast<unsigned*>(&s_prob);
            for (int i = threadIdx.x; i < kWords; i += blockDim.x) dst[i] = __ldcg(&src[i]);
        }
        __syncthreads();
        const DevProblem& P = s_prob;
        const int n_steps = P.n_steps;
        // coefficient table: read through the warp's window, by kLoopGeneral in place
        const T* tab = reinterpret_cast<const T*>(P.coef);

        const int tps = P.tiles_per_seg;
        const int lt = g - __ldcg(&tile_prefix[lo]);
        const int seg = lt / tps;
        const int tis = lt - seg * tps;
        const int n_mu = P.n_mu;
        const int n_seg = P.n_q * n_mu;
        const typename PrecTraits<T>::Halo hc = PrecTraits<T>::halo(P);
        const T x0 = reinterpret_cast<const T*>(P.x0)[seg];

        // steps of this launch: all of them, or one chunk of a served request
        const int s_begin = P.step_begin;
        const int s_end = P.step_end > 0 ? P.step_end : n_steps;
        T* state = reinterpret_cast<T*>(P.state);
        const bool more = state && s_end < n_steps;      // more chunks follow
        const int nm = P.n_mass;
        double* part = P.partials + ((size_t)seg * tps + tis) * 2 * nm;

        // one pass, but for a tile of more trajectories than the CTA holds
        constexpr bool kPasses = LOOP == kLoopGeneral || LOOP == kLoopFp64 || LOOP == kLoopPackedPasses;
        for (int base = 0; base < (kPasses ? P.tile : 1); base += blockDim.x * TPT) {
        T x[TPT], y[TPT], vx[TPT], vy[TPT];
        bool act[TPT];
        bool done = true;            // every trajectory of this lane is finished
#pragma unroll
        for (int i = 0; i < TPT; ++i) {
            const int t = tis * P.tile + base + slot(i);
            act[i] = base + slot(i) < P.tile && t < n_seg;
            done &= !act[i];
            const int tt = act[i] ? t : 0;
            if (state && s_begin > 0) {          // resume a served request
                const T* st = state + ((size_t)seg * n_seg + tt) * 4;
                x[i] = st[0];
                y[i] = st[1];
                vx[i] = st[2];
                vy[i] = st[3];
            } else {                             // Sec. II.C initial conditions
                const int j = tt / n_mu, k = tt - (tt / n_mu) * n_mu;
                const T v0 = reinterpret_cast<const T*>(P.v0)[j];
                x[i] = x0;
                y[i] = T(0);
                vx[i] = v0 * reinterpret_cast<const T*>(P.mu)[k];
                vy[i] = v0 * reinterpret_cast<const T*>(P.smu)[k];
            }
        }

        // A finished trajectory (escapes(): beyond R on a line that never
        // re-enters) keeps its velocity for every later step, and q_i depends
        // on v alone.  A warp stops integrating once all of its lanes are in that state
        // (padding lanes of a ragged tile start finished), and a finished lane
        // that keeps stepping with its warp stays beyond R with its velocity
        // unchanged.  All lanes of the warp reach the votes, so the full mask is
        // valid.
        if constexpr (LOOP == kLoopFp64) {
            fp64_loop(x[0], y[0], vx[0], vy[0], reinterpret_cast<const float4*>(tab), s_begin, s_end,
                      done, hc, ring, lane,
                      [&](double xa, double ya, double Sa, double Qa, double xb, double yb, double Sb,
                          double Qb, double& ma, double& mb) {
                          accel_pair(xa, ya, Sa, Qa, xb, yb, Sb, Qb, hc, s_pass[warp], lane, ma, mb);
                      });
        } else if constexpr (kSplit) {
            SplitPair pair{hc, s_pair[group * 4], 1 + group, warp >> 1, lane, 0};
            fp64_loop(x[0], y[0], vx[0], vy[0], reinterpret_cast<const float4*>(tab), s_begin, s_end,
                      done, hc, ring, lane, pair);
            if (warp >> 1) act[0] = false;               // counted once
        } else if constexpr (LOOP != kLoopGeneral) {
            using State = typename std::conditional<kTwo<LOOP>, TwoTrajectories<LOOP != kLoopPackedFew>,
                                                    OneTrajectory>::type;
            static_assert(TPT == (kTwo<LOOP> ? 2 : 1), "trajectories of a lane");
            const HaloX2 h2{dup(hc.invIc), dup(-hc.invR3), hc.R2, hc.R, hc.c};
            const float4* tab4 = reinterpret_cast<const float4*>(tab);
            State st(x, y, vx, vy);
            if (hc.narrow)
                step_loop<true>(st, tab4, s_begin, s_end, act, done, h2, ring, lane);
            else
                step_loop<false>(st, tab4, s_begin, s_end, act, done, h2, ring, lane);
            st.store(x, y, vx, vy);
        } else {
            bool fin_i[TPT];
#pragma unroll
            for (int i = 0; i < TPT; ++i) fin_i[i] = !act[i];
            for (int n = s_begin; n < s_end; ++n) {
                if (((n - s_begin) & (kExitEvery - 1)) == 0) {
                    bool fin = true;
#pragma unroll
                    for (int i = 0; i < TPT; ++i) {
                        fin_i[i] = !act[i] || escapes(fma(x[i], x[i], y[i] * y[i]),
                                                      fma(x[i], vx[i], y[i] * vy[i]),
                                                      fma(vx[i], vx[i], vy[i] * vy[i]), hc.R2,
                                                      hc.R, tab[(size_t)n * C_COUNT + C_IREM]);
                        fin &= fin_i[i];
                    }
                    done |= fin;
                    if (__all_sync(0xffffffffu, done)) break;
                }
                ctr.ran(TPT);
                T c[C_COUNT];
                const float4* c4 = reinterpret_cast<const float4*>(tab + (size_t)n * C_COUNT);
#pragma unroll
                for (int q = 0; q < (int)(C_COUNT * sizeof(T) / 16); ++q)
                    reinterpret_cast<float4*>(c)[q] = __ldg(&c4[q]);
#pragma unroll
                for (int i = 0; i < TPT; ++i) {
                    ctr.set_live(!fin_i[i] && !done);
                    rk4_step<T, Ctr>(x[i], y[i], vx[i], vy[i], c, hc, ctr);
                }
            }
        }

        if (more) {                              // keep the state
#pragma unroll
            for (int i = 0; i < TPT; ++i) {
                if (!act[i]) continue;
                T* st = state + ((size_t)seg * n_seg + tis * P.tile + base + slot(i)) * 4;
                st[0] = x[i];
                st[1] = y[i];
                st[2] = vx[i];
                st[3] = vy[i];
            }
            continue;
        }

        // Liouville map and the weight of each trajectory in Eq. localdensity,
        // in FP64 from the final state (in the mixed mode its FP32 components
        // widened exactly).  The final momentum is that of the fiducial mass;
        // mass a of a mass-reuse request reads it scaled by s_a (Sec. III).
        double qf[TPT];
#pragma unroll
        for (int i = 0; i < TPT; ++i) {
            const double ux = (double)vx[i], uy = (double)vy[i];
            qf[i] = sqrt(fma(ux, ux, uy * uy)) * P.q_scale;
            if (P.qi && act[i])
                reinterpret_cast<T*>(P.qi)[(size_t)seg * n_seg + tis * P.tile + base + slot(i)] = (T)qf[i];
        }
        // momentum and direction nodes of each trajectory (recomputed here
        // rather than kept live through the step loop)
        int tj[TPT], tk[TPT];
#pragma unroll
        for (int i = 0; i < TPT; ++i) {
            const int t = act[i] ? tis * P.tile + base + slot(i) : 0;
            tj[i] = t / n_mu;
            tk[i] = t - tj[i] * n_mu;
        }
        int a = 0;
        if constexpr (kMasses > 1) {
            const double wm = P.wmu[tk[0]], w = P.wq[tj[0]] * wm, wc = P.wqc[tj[0]] * wm;
            for (; a < nm; a += kMasses) {           // a last group may be short
                double v[2 * kMasses];
#pragma unroll
                for (int m = 0; m < kMasses; ++m) {
                    const bool read = act[0] && a + m < nm;
                    const double f = read ? relic_f_dev(P, qf[0] * P.mass_s[a + m]) : 0.0;
                    v[2 * m] = read ? __dadd_rn(0.0, __dmul_rn(w, f)) : 0.0;
                    v[2 * m + 1] = read ? __dadd_rn(0.0, __dmul_rn(wc, f)) : 0.0;
                }
                if (warp & 1) {
#pragma unroll
                    for (int j = 0; j < 2 * kMasses; ++j) s_half[warp >> 1][j][lane] = v[j];
                }
                __syncthreads();
                if (!(warp & 1)) {
#pragma unroll
                    for (int j = 0; j < 2 * kMasses; ++j) v[j] += s_half[warp >> 1][j][lane];
                    const double sum = warp_sums(v, lane);
                    constexpr int kLanes = 16 / kMasses;         // that return one sum
                    if (lane % kLanes == 0) s_red[warp >> 1][lane / kLanes] = sum;
                }
                __syncthreads();
                if (threadIdx.x < 2 * min(kMasses, nm - a))
                    part[2 * a + threadIdx.x] =
                        sum_of_four(4, kRingThreads / kUnit, [&](int i) { return s_red[i][threadIdx.x]; });
                __syncthreads();
            }
        }
        for (; kMasses == 1 && a < nm; ++a) {
            const double sa = P.mass_s[a];
            double acc = 0.0, accc = 0.0;
#pragma unroll
            for (int i = 0; i < TPT; ++i) {
                if (!act[i]) continue;
                // (no fused multiply-adds: a thread of one trajectory adds in no other way)
                const double f = relic_f_dev(P, qf[i] * sa);
                const double wm = P.wmu[tk[i]];
                acc = __dadd_rn(acc, __dmul_rn(P.wq[tj[i]] * wm, f));
                accc = __dadd_rn(accc, __dmul_rn(P.wqc[tj[i]] * wm, f));
            }
            if constexpr (TPT == 1) {
                if (warp & 1) {
                    s_half[warp >> 1][0][lane] = acc;
                    s_half[warp >> 1][1][lane] = accc;
                }
                __syncthreads();
                if (!(warp & 1) && warp + 1 < n_warps) {
                    acc += s_half[warp >> 1][0][lane];
                    accc += s_half[warp >> 1][1][lane];
                }
            }
            if (TPT == 2 || !(warp & 1)) {
                acc = warp_sum(acc);
                accc = warp_sum(accc);
                if (lane == 0) {
                    s_red[TPT == 2 ? warp : warp >> 1][0] = acc;
                    s_red[TPT == 2 ? warp : warp >> 1][1] = accc;
                }
            }
            __syncthreads();
            if (threadIdx.x < 2) {               // the units of this pass, in order
                double t = base > 0 ? part[2 * a + threadIdx.x] : 0.0;
                const int units = (min((int)blockDim.x * TPT, P.tile - base) + kUnit - 1) / kUnit;
                for (int u = 0; u < units; u += 4)
                    t += sum_of_four(4, units - u, [&](int i) { return s_red[u + i][threadIdx.x]; });
                part[2 * a + threadIdx.x] = t;
            }
            __syncthreads();   // s_red is reused by the next mass
        }
        }   // passes
        if (more) {
            __syncthreads();   // every thread has read s_tile before it is reused
            continue;
        }

        if (threadIdx.x == 0) {
            __threadfence();
            const unsigned prev = atomicAdd(&P.seg_count[seg], 1u);
            s_last = (prev == (unsigned)(tps - 1));
        }
        __syncthreads();

        if (s_last && warp == 0) {   // this CTA finished the radius: add tiles in order
            __threadfence();
            const double* sp = P.partials + (size_t)seg * tps * 2 * nm;
            // P.group tiles make one tile of the request's shape, `per` of them a four
            const int n_whole = (tps + P.group - 1) / P.group;
            const int per = P.group > 1 ? max(1, 4 * kUnit / P.tile) : 1;
            for (int a = 0; a < nm; ++a) {
                double t0 = 0.0, t1 = 0.0;
                for (int k = lane; k < n_whole; k += 32) {
                    double w0 = 0.0, w1 = 0.0;
                    const int end = min((k + 1) * P.group, tps);
                    for (int i = k * P.group; i < end; i += per) {
                        const double* s0 = sp + (size_t)i * 2 * nm + 2 * a;
                        w0 += sum_of_four(per, end - i, [&](int j) { return __ldcg(s0 + j * 2 * nm); });
                        w1 += sum_of_four(per, end - i, [&](int j) { return __ldcg(s0 + j * 2 * nm + 1); });
                    }
                    t0 += w0;
                    t1 += w1;
                }
                t0 = warp_sum(t0);
                t1 = warp_sum(t1);
                if (lane == 0) {
                    const double ratio = t0 * P.norms[2 * a];
                    const double ratio_c = t1 * P.norms[2 * a + 1];
                    P.out[(size_t)a * P.n_radii + seg] = ratio;
                    const double err = fabs(ratio - ratio_c) / (3.0 * fabs(ratio));
                    P.err[(size_t)a * P.n_radii + seg] = err;
                    if (P.host_out) {
                        P.host_out[(size_t)a * P.n_radii + seg] = ratio;
                        P.host_out[(size_t)(nm + a) * P.n_radii + seg] = err;
                    }
                }
            }
            if (lane == 0) {
                P.seg_count[seg] = 0u;              // ready for the next run
                if (P.done_flag) {                  // serving: signal the request's last radius
                    __threadfence_system();
                    if (atomicAdd(P.done_count, 1u) == (unsigned)P.n_radii - 1u) {
                        __threadfence_system();
                        *P.done_flag = 1u;
                    }
                }
            }
        }
        // the next iteration's first __syncthreads orders s_tile/s_last reuse
    }
    // the last CTA to leave makes the counters ready for the next launch
    if (threadIdx.x == 0 && atomicAdd(&ctrl[kCtrlLeft], 1u) == gridDim.x - 1u) {
        ctrl[kCtrlNext] = 0u;
        ctrl[kCtrlLeft] = 0u;
    }
    if constexpr (COUNT) {
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            unsigned long long v = ctr.n[k];
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
            if (lane == 0) atomicAdd(&tallies[k], v);
        }
    }
}

// Force probe: m = Mhat/r^3 from the same device function the integrator
// uses, at radius r[i] on the x axis and RK stage (half-step index) `stage`.
template <typename T>
__global__ void force_probe_kernel(const DevProblem* __restrict__ prob, int stage,
                                   const double* __restrict__ r, int n, double* __restrict__ out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const DevProblem& P = *prob;
    const T* c = reinterpret_cast<const T*>(P.coef);
    // stage 2k -> S0/Q0 of step k; 2k+1 -> S1/Q1 of step k; 2N -> S2/Q2 of step N-1
    const int k = stage >= 2 * P.n_steps ? P.n_steps - 1 : stage / 2;
    const int slot = stage >= 2 * P.n_steps ? 2 : (stage & 1);
    const T S = c[(size_t)k * C_COUNT + C_S0 + slot];
    const T Q = c[(size_t)k * C_COUNT + C_Q0 + slot];
    const T Tq = c[(size_t)k * C_COUNT + C_T0 + slot];
    const typename PrecTraits<T>::Halo hc = PrecTraits<T>::halo(P);
    NoTally none;
    if constexpr (std::is_same<T, double>::value)
        out[i] = accel_m<NoTally, false>(r[i], 0.0, S, Q, Tq, hc, none);
    else
        out[i] = (double)accel_m((T)r[i], T(0), S, Q, Tq, hc, none);
}

int launch_force_probe(int precision, const DevProblem* d_prob, int stage, const double* d_r, int n,
                       double* d_out, void* stream)
{
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    const int grid = (n + 127) / 128;
    if (precision == NU_FP64)
        force_probe_kernel<double><<<grid, 128, 0, s>>>(d_prob, stage, d_r, n, d_out);
    else
        force_probe_kernel<float><<<grid, 128, 0, s>>>(d_prob, stage, d_r, n, d_out);
    if (cudaGetLastError() != cudaSuccess) return NU_ECUDA;
    count_launch();
    return NU_OK;
}

// The kernel, the threads of a CTA and the tiles of a launch whose sums are to be
// those of tiles of `tile`.
//   Mixed precision: one trajectory a lane or two (packed), each in CTAs of four
// warps, one for each scheduler of an SM.  As a CTA is one warp more on every scheduler of
// its SM, a step of a launch that fits the chip takes the time of the SM with most CTAs:
// with w of them (more than four one a lane take turns), about max(440, 280 + 115 w)
// cycles one trajectory a lane and max(540, 250 + 240 w) packed.  The cheaper one is taken.
// Measured, one a lane / packed, us for 400 steps of the sweep's halo over
//    12k    25k    38k    51k    65k    77k    92k   102k   116k   153k   184k   208k   233k
//  90/109 102/111 104/110 125/143 153/150 160/151 166/204 174/202 197/205 248/258 293/305 321/355 346/357
// trajectories.  At 97 to 116k packed is taken: one a lane is up to 20 % faster on many
// halos, and up to 15 % slower on the heaviest.  From 233k on (more packed CTAs than fit
// the chip) it is taken too: 250k 354/361, 271k 383/369, 307k 422/397, with one a lane 5 to
// 30 % faster where most trajectories leave, and up to 12 % slower where none does.
//   FP64: one trajectory a lane, in the smallest CTAs there are sums for, and of
// those the fewest on an SM that give each scheduler a warp: one keeps its FP64
// unit busy, and work not yet started can go to an SM that is done early.  Six radii of
// the precision sweep take 25.5 ms with 4 warps on an SM, 26.0 with 6 and 30.5 with 8;
// 26.1 in CTAs of 4 warps; in tiles of 96 26.6 with 6 warps and 31.7 with 3.
//   A second pair of warps takes half of the force evaluations where each SM has a tile
// at most (16 to 144 tiles of the plain workload 3.75-3.79 ms instead of 5.7-6.4).  The
// split kernel has one CTA on an SM, so further tiles wait for one to end, which costs
// nothing while fast trajectories leave their tiles early.  At 100 steps, split against
// whole: 160 to 225 tiles of the plain and the sweep grid 1.00-1.08 ms against 1.53-1.69,
// 248 to 253 1.0-1.8 against 1.6-1.7, 256 to 260 1.1-1.8, 272 to 320 1.7-1.95 against
// 1.5-1.7.  So it is taken up to 5/3 tiles an SM.  Where nothing leaves (relics of 0.3 eV
// and more, the heaviest halos) it costs up to 15 % from 185 tiles on; and with one or two
// tiles a radius each tile holds slow momenta, and nothing ends early on any halo (200
// tiles 1.71 against 1.56 ms), so from two waves on those run whole.
constexpr int kFp64WarpsPerSm = 4;
constexpr int kPackedTile = 256;
constexpr int kPackedCtas = 6;                       // on an SM
constexpr int kPackedFewCtas = 3;                    // on an SM: the loop without kOutside
constexpr int kDevices = 32;                         // whose properties are kept

int sm_count()
{
    static std::atomic<int> kept[kDevices];
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return 0;
    if (dev < kDevices && (n = kept[dev].load(std::memory_order_relaxed)) > 0) return n;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) return 0;
    if (dev < kDevices) kept[dev].store(n, std::memory_order_relaxed);
    return n;
}

LaunchShape plan_shape(int precision, int tile, const LaunchSize& size)
{
    if (size.n_traj > (1LL << 35)) return whole_tiles(precision, tile);   // few enough to count
    const long long sms = std::max(1, sm_count());
    LaunchShape s;
    s.tile = tile;
    if (precision == NU_FP64) {
        const bool split = tile % kUnit == 0 &&
                           (size.tiles64 <= sms ||
                            (size.tiles64 * 3 <= sms * 5 && size.tiles64 >= 3 * size.radii));
        s.kernel = split ? kFp64Split : kFp64;
        s.tile = tile % kUnit == 0 ? kUnit : tile;
        s.threads = split ? 2 * kUnit : std::min(s.tile, 256);
    } else {
        const long long w1 = (size.tiles128 + sms - 1) / sms, w2 = (size.tiles256 + sms - 1) / sms;
        const bool one = tile % kRingThreads == 0 && w2 <= kPackedCtas &&
                         std::max(440LL, 280 + 115 * w1) < std::max(540LL, 250 + 240 * w2);
        s.kernel = !one ? (w2 <= kPackedFewCtas ? kPackedFew : kPacked)
                        : size.most_masses > 1 ? kRingMasses : kRing;
        for (int t : {one ? kRingThreads : kPackedTile, 128, 64})
            if (tile % t == 0) {
                s.tile = t;
                break;
            }
        s.threads = one ? s.tile : (s.tile + kUnit - 1) / kUnit * 32;
    }
    s.group = tile / s.tile;
    return s;
}

// The same with CTAs that claim whole tiles, for callers without room for the sums
// of smaller ones.  A mixed tile of more than 512 trajectories is integrated in passes
// of four units, which leaves 24 warps on an SM: 300 radii x 262144 trajectories x 20
// steps take 10.8 ms in tiles of 576 and 9.3 in tiles of 1024; one trajectory after
// another with the branching force took 24.0 and 17.4.
LaunchShape whole_tiles(int precision, int tile)
{
    LaunchShape s;
    s.tile = tile;
    s.group = 1;
    if (precision == NU_FP64) {
        s.kernel = kFp64;
        s.threads = std::min(tile, 256);
    } else if (tile <= 512) {
        s.kernel = kPacked;
        s.threads = (tile + kUnit - 1) / kUnit * 32;
    } else {
        s.kernel = kPackedPasses;
        s.threads = kPackedTile / 2;
    }
    return s;
}

typedef void (*TrajKernel)(const DevProblem*, const int*, int, int, unsigned*, unsigned long long*,
                           QueueCtl*);

static TrajKernel kernel_of(int kernel)
{
    switch (kernel) {
    case kPacked: return traj_kernel<float, 2, false, kLoopPacked>;
    case kRing: return traj_kernel<float, 1, false, kLoopRing>;
    case kRingMasses: return traj_kernel<float, 1, false, kLoopRingMasses>;
    case kFp64: return traj_kernel<double, 1, false, kLoopFp64>;
    case kFp64Split: return traj_kernel<double, 1, false, kLoopFp64Split>;
    case kPackedFew: return traj_kernel<float, 2, false, kLoopPackedFew>;
    case kPackedPasses: return traj_kernel<float, 2, false, kLoopPackedPasses>;
    case kCountF32: return traj_kernel<float, 2, true, kLoopGeneral>;
    default: return traj_kernel<double, 2, true, kLoopGeneral>;
    }
}

// Shared memory of a CTA: its warps' windows on the table.
static size_t ring_bytes(const LaunchShape& shape)
{
    return (size_t)(shape.threads / 32) * kRing16 * sizeof(float4);   // (not the counting kernels)
}

int launch_traj(const LaunchShape& shape, int grid, const DevProblem* d_probs, const int* d_prefix,
                int n_probs, int n_tiles, unsigned* d_counter, void* stream, QueueCtl* d_queue)
{
    cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
    kernel_of(shape.kernel)<<<grid, shape.threads, ring_bytes(shape), s>>>(d_probs, d_prefix, n_probs, n_tiles,
                                                           d_counter, nullptr, d_queue);
    if (cudaGetLastError() != cudaSuccess) return NU_ECUDA;
    cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &cs) == cudaSuccess && cs == cudaStreamCaptureStatusNone)
        count_launch();   // captured launches are counted when the graph is replayed
    return NU_OK;
}

int launch_traj_tally(int precision, const LaunchShape& shape, int grid, const DevProblem* d_probs,
                      const int* d_prefix, int n_probs, int n_tiles, unsigned* d_counter,
                      unsigned long long* d_tallies, void* stream)
{
    // the branches and needed steps are trajectory facts: every kernel integrates the same
    // values.  The lane-steps run are this launch's own.
    const int threads = std::min((shape.tile + kUnit - 1) / kUnit * 32, 512);
    kernel_of(precision == NU_FP64 ? kCountF64 : kCountF32)
        <<<grid, threads, 0, reinterpret_cast<cudaStream_t>(stream)>>>(
            d_probs, d_prefix, n_probs, n_tiles, d_counter, d_tallies, nullptr);
    if (cudaGetLastError() != cudaSuccess) return NU_ECUDA;
    count_launch();
    return NU_OK;
}

int max_ctas_per_sm(const LaunchShape& shape, int* out)
{
    // asked for by every run: kept for each device
    static std::atomic<int> kept[kDevices][kKernelKinds][512 / 32 + 1];
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return NU_ECUDA;
    std::atomic<int>* known = dev < kDevices ? &kept[dev][shape.kernel][shape.threads / 32] : nullptr;
    if (known && (*out = known->load(std::memory_order_relaxed)) > 0) return NU_OK;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(out, kernel_of(shape.kernel), shape.threads,
                                                      ring_bytes(shape)) != cudaSuccess)
        return NU_ECUDA;
    if (shape.kernel == kFp64 || shape.kernel == kFp64Split)
        *out = std::min(*out, (kFp64WarpsPerSm * 32 + shape.threads - 1) / shape.threads);
    if (known) known->store(*out, std::memory_order_relaxed);
    return NU_OK;
}

}  // namespace nuprof
