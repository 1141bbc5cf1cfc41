// Monte Carlo photon-packet walk (Sec. 2.1-2.3 of the paper), one persistent
// kernel per run.
//
// Scheduling: a persistent grid (a few CTAs per SM). Each lane owns one
// packet in registers. Whenever enough lanes of a warp are idle, the warp
// takes a contiguous block of packet ids with ONE atomicAdd on a global work
// counter (ballot + popc + shuffle) and the idle lanes emit those packets;
// this is the server-worker scheme of Sec. 2.3.2 at warp granularity. After
// the counter runs out, a CTA packs its running packets into full warps, and
// its last few packets are each walked by a group of lanes (see run_model and
// transport_tail.cuh).
//
// Per iteration a lane advances its packet by one event in the current
// cell: with x_com = x_lab - n.V/b (Sec. 2.2.1) and alpha = alpha0
// H(a, x_com) (Sec. 2.1), it either scatters inside the cell (tau < alpha
// s_exit) or crosses the nearest face. A scattering draws u_par from the
// velocity sampler (Sec. 2.1.1), u_perp from a Gaussian, an isotropic new
// direction and x_out = x_in + u_par (g - 1) + u_perp sin(gamma)
// (Eq. riia-scatter); with probability epsilon (Eq. eps) the photon is
// destroyed instead. Leaving a non-periodic face is an escape, binned in the
// lab-frame spectrum.
//
// Random numbers: Philox4x32-10 with counter (id_lo, id_hi, event, block)
// and key (seed_lo, seed_hi); a 32-bit word r becomes ((r >> 9) + 1/2) 2^-23,
// exact in FP32 and FP64. Event 0 is the emission, event e >= 1 the e-th
// scattering; the slots of each event are fixed (see emit / scatter), so a
// packet's stream depends only on (seed, id).
//
// Tallies: scattering counts and excitation are summed in registers over a
// cell visit and flushed with one atomic when the packet leaves the cell;
// the mean-intensity and emissivity tallies (Eq. scat-line) are added per
// segment. Spectrum and counters go to FP64 / 64-bit integers.
//
// Precision: R = float is the production walk (FP32 arithmetic in cell-local
// coordinates, so positions keep 2^-24 of a cell width at any optical depth);
// R = double runs the same steps in FP64 for lockstep checks.
#pragma once

#include <math.h>
#include <stdint.h>

#include <type_traits>

#include "krl_internal.cuh"

namespace krl {

namespace {

constexpr unsigned kFull = 0xffffffffu;

// Table placement PH = 4 (a measurement variant of profile mode 2, chosen
// by krl_tune.table_space): the Voigt slice and the sampler's nodes and ln
// CDF read from __constant__ memory (60 KB, copied in before each launch)
// instead of shared memory; the search guides stay in shared memory. The
// arrays exist only in the translation unit that instantiates that mode.
#ifdef KRL_TABLES_IN_CONSTANT
__constant__ float c_voigt[kVoigtN];
__constant__ float c_usx[kUsNx];
__constant__ float c_uslncdf[kUsNx * kUsNu];
#endif

// ---------------------------------------------------------------- Philox4x32-10

struct Words {
    uint32_t w[4];
};

__device__ __forceinline__ Words philox(uint32_t c0, uint32_t c1, uint32_t c2, uint32_t c3, const RoundKeys& K)
{
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint32_t m0 = 0xD2511F53u, m1 = 0xCD9E8D57u;
        uint32_t h0 = __umulhi(m0, c0), l0 = m0 * c0;
        uint32_t h1 = __umulhi(m1, c2), l1 = m1 * c2;
        uint32_t n0 = h1 ^ c1 ^ K.k[0][r];
        uint32_t n2 = h0 ^ c3 ^ K.k[1][r];
        c0 = n0;
        c1 = l1;
        c2 = n2;
        c3 = l0;
    }
    return Words{{c0, c1, c2, c3}};
}

// ---------------------------------------------------------------- precision policy

template <typename R>
struct Ops;

template <>
struct Ops<float> {
    // ((r >> 9) + 1/2) 2^-23 without an int-to-float conversion: the bits
    // give 1 + (r >> 9) 2^-23, and subtracting 1 - 2^-24 is exact (Sterbenz)
    static __device__ __forceinline__ float uni(uint32_t r)
    {
        return __uint_as_float((r >> 9) + 0x3f800000u) - 0x1.fffffep-1f;
    }
    static __device__ __forceinline__ float ln(float v) { return __logf(v); }
    static __device__ __forceinline__ float ex(float v) { return __expf(v); }
    // sqrt(v) for v >= 0 as v * rsqrt(v) (one MUFU op, 2 ulp)
    static __device__ __forceinline__ float sq(float v) { return v > 0.0f ? v * rsqrtf(v) : 0.0f; }
    static __device__ __forceinline__ float dv(float a, float b) { return __fdividef(a, b); }
    // 1/a to about 1 ulp (one MUFU op; used for the exit distances only)
    static __device__ __forceinline__ float rcp(float a)
    {
        float r;
        asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
        return r;
    }
    // sin and cos of 2 pi u for u in (0, 1): shift to [-pi, pi] where the
    // hardware approximation is accurate, then reflect.
    static __device__ __forceinline__ void sc2pi(float u, float* s, float* c)
    {
        float ss, cc;
        __sincosf(6.28318530717958648f * (u - 0.5f), &ss, &cc);
        *s = -ss;
        *c = -cc;
    }
    static __device__ __forceinline__ float big() { return 3.0e38f; }
    // min(1, max(0, p + d n)): one saturating FMA
    static __device__ __forceinline__ float step01(float p, float d, float n) { return __saturatef(fmaf(d, n, p)); }
    // position of |x| on the Voigt table, (log10|x| - L0) (N - 1) / (L1 - L0),
    // as one FMA on log2|x|
    static __device__ __forceinline__ float vt(float ax)
    {
        constexpr double C = (kVoigtN - 1) / (kVoigtL1 - kVoigtL0);
        return fmaf(__log2f(ax), (float)(C * 0.30102999566398119521), (float)(-kVoigtL0 * C));
    }
};

template <>
struct Ops<double> {
    static __device__ __forceinline__ double uni(uint32_t r) { return (double)(r >> 9) * 0x1p-23 + 0x1p-24; }
    static __device__ __forceinline__ double ln(double v) { return log(v); }
    static __device__ __forceinline__ double ex(double v) { return exp(v); }
    static __device__ __forceinline__ double sq(double v) { return sqrt(v); }
    static __device__ __forceinline__ double dv(double a, double b) { return a / b; }
    static __device__ __forceinline__ double rcp(double a) { return 1.0 / a; }
    static __device__ __forceinline__ void sc2pi(double u, double* s, double* c) { sincospi(2.0 * u, s, c); }
    static __device__ __forceinline__ double big() { return 1.0e300; }
    static __device__ __forceinline__ double step01(double p, double d, double n) { return fmin(1.0, fmax(0.0, p + d * n)); }
    static __device__ __forceinline__ double vt(double ax)
    {
        return (log10(ax) - (double)kVoigtL0) * ((kVoigtN - 1) / (kVoigtL1 - kVoigtL0));
    }
};

// ---------------------------------------------------------------- paired FP32 draws
//
// The FP32 walk pairs the independent single-precision work of a scattering
// in the paired instructions of sm_100 and later (FFMA2 / FADD2 / FMUL2;
// each half rounds as the scalar operation would): the uniforms, the logs,
// the two angles, the square roots' products and the Box-Muller and
// direction products, and the two sampler rows' inversions.

__device__ __forceinline__ float lg2_approx(float x)
{
    float r;
    asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// a - b for two values as fma(b, -1, a): exact product, one rounding
__device__ __forceinline__ float2 sub2f(float2 a, float2 b)
{
    return __ffma2_rn(b, make_float2(-1.0f, -1.0f), a);
}

// two uniforms ((r >> 9) + 1/2) 2^-23, as Ops<float>::uni
__device__ __forceinline__ float2 uni2(uint32_t a, uint32_t b)
{
    return __fadd2_rn(make_float2(__uint_as_float((a >> 9) + 0x3f800000u), __uint_as_float((b >> 9) + 0x3f800000u)),
                      make_float2(-0x1.fffffep-1f, -0x1.fffffep-1f));
}

// One scattering's draws from its two Philox blocks (slots as in advance):
// the guide bin and L = ln(xi) of the velocity sampler, the Box-Muller
// radius and phase (cos, sin), the new isotropic direction, the next free
// path.
struct DrawsF {
    float L, rad, bc, bs, mx, my, mz, tau;
    int gm;
};

__device__ __forceinline__ DrawsF draws_f32(const Words& w0, const Words& w1)
{
    constexpr float kLn2 = 0.69314718055994531f;
    DrawsF D;
    const float2 ua = uni2(w0.w[0], w0.w[1]);          // xi of u_par, Box-Muller radius
    const float2 ub = uni2(w0.w[2], w0.w[3]);          // Box-Muller phase, free path
    const float2 uc = uni2(w1.w[0], w1.w[1]);          // mu, azimuth
    // -ln of the radius and free-path uniforms; ln xi and ln(1 - xi)
    const float2 nl = __fmul2_rn(make_float2(lg2_approx(ua.y), lg2_approx(ub.y)), make_float2(-kLn2, -kLn2));
    const float2 lx = __fmul2_rn(make_float2(lg2_approx(ua.x), lg2_approx(1.0f - ua.x)), make_float2(kLn2, kLn2));
    D.L = fminf(lx.x, -1e-30f);
    int m = (int)((D.L - lx.y + (float)kGuideW) * (float)(kGuideN / (2.0 * kGuideW)));
    D.gm = m < 0 ? 0 : (m > kGuideN - 1 ? kGuideN - 1 : m);
    D.tau = fmaxf(0.0f, nl.y);
    // square roots v rsqrt(v) of the radius^2 and of 1 - mu^2 (0 for v <= 0)
    const float rr = fmaxf(0.0f, nl.x);
    const float mu = fmaf(2.0f, uc.x, -1.0f);
    const float ss = fmaxf(0.0f, fmaf(-mu, mu, 1.0f));
    const float2 rt = __fmul2_rn(make_float2(rr, ss), make_float2(rsqrtf(rr), rsqrtf(ss)));
    D.rad = rr > 0.0f ? rt.x : 0.0f;
    const float st = ss > 0.0f ? rt.y : 0.0f;
    // sin and cos of 2 pi u through the shifted angle 2 pi (u - 1/2) in
    // [-pi, pi] (negated back), for the phase and the azimuth
    const float2 ang = __fmul2_rn(__fadd2_rn(make_float2(ub.x, uc.y), make_float2(-0.5f, -0.5f)),
                                  make_float2(6.28318530717958648f, 6.28318530717958648f));
    float sb, cb, sp, cp;
    __sincosf(ang.x, &sb, &cb);
    __sincosf(ang.y, &sp, &cp);
    D.bc = -cb;
    D.bs = -sb;
    const float2 mxy = __fmul2_rn(make_float2(st, st), make_float2(-cp, -sp));
    D.mx = mxy.x;
    D.my = mxy.y;
    D.mz = mu;
    return D;
}

// ---------------------------------------------------------------- table lookups (shared memory)

// H(a, x) from the ph_mode 2 slice: ln H linear in log10|x| between nodes;
// H(a, 0) below |x| = 1e-4 and the wing series above 1e3. The table path is
// evaluated for every x (finite for any x); the two outer ranges, which a
// walk rarely reaches, replace it in a branch of their own.
template <typename R>
__device__ __forceinline__ R voigt(R x, const float* sv, R a, R H0)
{
    using O = Ops<R>;
    const R ax = fabs(x);
    const R t = O::vt(ax);
    int i = (int)t;
    i = i < 0 ? 0 : (i > kVoigtN - 2 ? kVoigtN - 2 : i);
    const R f = t - (R)i;
    const R l0 = (R)sv[i], l1 = (R)sv[i + 1];
    R lh;
    if constexpr (sizeof(R) == 4) lh = fmaf(f, l1, __fmul_rn(1.0f - f, l0));
    else lh = ((R)1 - f) * l0 + f * l1;
    R h = O::ex(lh);
    if (ax < (R)1e-4 || ax > (R)1e3) {
        const R ax2 = ax * ax;
        R wing;
        if constexpr (sizeof(R) == 4) {
            const float r = Ops<float>::rcp(ax2);                 // one reciprocal: a r (1 + 3r/2) / sqrt(pi)
            wing = (a * 0.56418958354775628f) * r * fmaf(1.5f, r, 1.0f);
        } else {
            wing = a / ((R)1.7724538509055160 * ax2) * ((R)1 + (R)1.5 / ax2);
        }
        h = ax < (R)1e-4 ? H0 : wing;
    }
    return h;
}

// Line-profile mode 1: ln H bilinear in (log10 a, log10|x|) on the global
// two-dimensional table; the rows v2_row, v2_row + 1 and the weight v2_w of
// this a come with the launch. |x| below the first node takes the first
// node; the wing series above |x| = 1e3.
template <typename R>
__device__ __forceinline__ R voigt2d(const TransportArgs& A, R x, R a)
{
    using O = Ops<R>;
    const R ax = fabs(x);
    constexpr double C = (kV2Nx - 1) / (kVoigtL1 - kVoigtL0);
    R t;
    if constexpr (sizeof(R) == 4) {
        t = fmaf(__log2f(fmaxf(ax, 1e-4f)), (float)(C * 0.30102999566398119521), (float)(-kVoigtL0 * C));
    } else {
        t = (log10(ax < 1e-4 ? 1e-4 : ax) - kVoigtL0) * C;
    }
    t = t < (R)0 ? (R)0 : t;
    int i = (int)t;
    i = i > kV2Nx - 2 ? kV2Nx - 2 : i;
    const R f = t - (R)i;
    const float* r0 = A.voigt2d + (size_t)A.v2_row * kV2Nx;
    const float* r1 = r0 + kV2Nx;
    const R l0 = ((R)1 - f) * (R)__ldg(r0 + i) + f * (R)__ldg(r0 + i + 1);
    const R l1 = ((R)1 - f) * (R)__ldg(r1 + i) + f * (R)__ldg(r1 + i + 1);
    const R w = (R)A.v2_w;
    const R tab = O::ex(((R)1 - w) * l0 + w * l1);
    const R ax2 = ax * ax;
    const R wing = O::dv(a, (R)1.7724538509055160 * ax2) * ((R)1 + O::dv((R)1.5, ax2));
    return ax > (R)1e3 ? wing : tab;
}

// Line-profile mode 3: (1 - w) exp(-x^2) + w a / (sqrt(pi) (x^2 + a^2)) with
// w = [1 + tanh(2|x| - 2 u0)] / 2 = 1 / (1 + exp(4 (u0 - |x|))).
template <typename R>
__device__ __forceinline__ R blend(const TransportArgs& A, R x, R a)
{
    using O = Ops<R>;
    const R ax = fabs(x);
    const R w = O::dv((R)1, (R)1 + O::ex((R)4 * ((R)A.u0 - ax)));
    const R core = O::ex(-ax * ax);
    const R wing = O::dv(a, (R)1.7724538509055160 * (ax * ax + a * a));
    return ((R)1 - w) * core + w * wing;
}

template <typename R, int PH>
__device__ __forceinline__ R profile(const TransportArgs& A, R x, const float* sv, R a, R H0)
{
    // (PH 4 is mode 2 with its tables in constant memory: the slice below)
    if constexpr (PH == 1) return voigt2d<R>(A, x, a);
    else if constexpr (PH == 3) return blend<R>(A, x, a);
    else return voigt<R>(x, sv, a, H0);
}

// The sampling tables as the walk reads them (shared memory in profile mode
// 2). rb and rx serve the FP32 walk. Per bin of the row guide, two vectors:
// {node x_i+1, or infinity in the last row; i; x_i, 1 / (x_i+1 - x_i)} and
// {x_i+1, 1 / (x_i+2 - x_i+1); -, -}. Per row, {x_i, 1 / (x_i+1 - x_i)}.
struct Tabs {
    const float* sv;
    const float* sx;
    const float* sc;
    const unsigned char* sg;
    const unsigned char* rg;
    const float4* rb;
    const float2* rx;
    unsigned long long* segw;       // this warp's next slot of the segment buffer
};

__device__ __forceinline__ int row_bin(float f)
{
    const int t = (int)(__float_as_uint(f) >> 19) - (int)kRowGuideBase;
    return t < 0 ? 0 : (t > kRowGuideN - 1 ? kRowGuideN - 1 : t);
}

// The same bin with the clamp on ax itself, which shortens the way from ax to
// the address (a group's walk waits for it).
__device__ __forceinline__ int row_bin_in(float ax)
{
    const float f = fminf(fmaxf(ax, 0.25f), 511.0f);
    return (int)(__float_as_uint(f) >> 19) - (int)kRowGuideBase;
}

// Largest row i in [0, 38] with X[i] <= ax, and the two bracketing nodes:
// the row guide's entry for the bin of ax (a node at or below ax), then one
// step up if the next node is also <= ax. The FP64 walk takes the bin of ax
// rounded toward zero, so the entry stays at or below ax there too.
__device__ __forceinline__ int us_row2(double ax, const Tabs& T, double& x0, double& x1)
{
    const float* sx = T.sx;
    const int i = T.rg[row_bin(__double2float_rz(ax))];
    const double g0 = (double)sx[i], g1 = (double)sx[i + 1];
    const double gp = (double)sx[i < kUsNx - 2 ? i + 2 : kUsNx - 1];
    const bool up = i < kUsNx - 2 && g1 <= ax;
    x0 = up ? g1 : g0;
    x1 = up ? gp : g1;
    return i + (up ? 1 : 0);
}

// The same row for the FP32 walk: one 8-byte read.
__device__ __forceinline__ int us_row(float ax, const Tabs& T)
{
    const float2 g = *reinterpret_cast<const float2*>(T.rb + 2 * row_bin(ax));
    return __float_as_int(g.y) + (g.x <= ax ? 1 : 0);
}

// Weight of row i + 1 at ax (the FP32 walk): (ax - x_i) / (x_i+1 - x_i) as a
// product with the row's approximate reciprocal, which is what __fdividef
// evaluates (equal for every ax of every row).
__device__ __forceinline__ float us_weight(float ax, int i, const Tabs& T)
{
    const float2 r = T.rx[i];
    return __fmul_rn(ax - r.x, r.y);
}

// The FP32 walk's sums and products that two pieces of code share (a lane's
// walk and a group's, transport_tail.cuh) are written with explicit fused
// operations: their rounding then does not depend on what the compiler fuses
// around them, and a packet takes the same path in both.

// u of the two rows interpolated in |x| (for x >= 0; u is odd in x).
template <typename R>
__device__ __forceinline__ R us_lerp(R t, R ua, R ub)
{
    if constexpr (sizeof(R) == 4) return fmaf(1.0f - t, ua, __fmul_rn(t, ub));
    else return ((R)1 - t) * ua + t * ub;
}

// u_par for incoming gas-frame frequency x (|x| <= 300), given L = ln(xi)
// and the guide bin m of logit(xi). Each bracketing row is inverted at L:
// the largest node j with c[j] <= L (the guide entry starts at or next to
// it; the bounded walks make the result exactly the bisection's), then u is
// linear between nodes j and j + 1; the two rows' u are interpolated in |x|.
// The two rows are walked together so their shared-memory loads overlap.
template <typename R>
__device__ __forceinline__ R us_sample(R x, R L, int m, const Tabs& T)
{
    using O = Ops<R>;
    const R ax = fabs(x);
    R t;
    int i;
    if constexpr (sizeof(R) == 4) {
        i = us_row(ax, T);
        t = us_weight(ax, i, T);
    } else {
        R x0, x1;
        i = us_row2(ax, T, x0, x1);
        t = O::dv(ax - x0, x1 - x0);
    }
    const float* ra = T.sc + i * kUsNu;
    const float* rb = ra + kUsNu;
    int ja = T.sg[i * kGuideN + m];
    int jb = T.sg[(i + 1) * kGuideN + m];
    R a0 = (R)ra[ja], a1 = (R)ra[ja + 1];
    R b0 = (R)rb[jb], b1 = (R)rb[jb + 1];
    // Every row starts at the floor ln 1e-30 < L and ends at ln 1 = 0 > L
    // (L is the log of a uniform in [2^-24, 1 - 2^-24]), so both walks stop
    // inside the row without bound checks.
    for (;;) {
        const bool da = a0 > L;
        const bool db = b0 > L;
        if (!(da || db)) break;
        if (da) { --ja; a1 = a0; a0 = (R)ra[ja]; }
        if (db) { --jb; b1 = b0; b0 = (R)rb[jb]; }
    }
    for (;;) {
        const bool ua = a1 <= L;
        const bool ub = b1 <= L;
        if (!(ua || ub)) break;
        if (ua) { ++ja; a0 = a1; a1 = (R)ra[ja + 1]; }
        if (ub) { ++jb; b0 = b1; b1 = (R)rb[jb + 1]; }
    }
    R ua_, ub_;
    if constexpr (sizeof(R) == 4) {
        // both rows at once: u_j + du (L - c_j) / (c_j+1 - c_j)
        const float2 num = sub2f(make_float2(L, L), make_float2(a0, b0));
        const float2 den = sub2f(make_float2(a1, b1), make_float2(a0, b0));
        const float2 fr = __fmul2_rn(num, make_float2(O::rcp(den.x), O::rcp(den.y)));
        float2 u2 = __ffma2_rn(make_float2((float)kUsDu, (float)kUsDu), make_float2((float)ja, (float)jb),
                               make_float2((float)kUsU0, (float)kUsU0));
        u2 = __ffma2_rn(make_float2((float)kUsDu, (float)kUsDu), fr, u2);
        ua_ = u2.x;
        ub_ = u2.y;
    } else {
        ua_ = (R)kUsU0 + (R)kUsDu * (R)ja + (R)kUsDu * O::dv(L - a0, a1 - a0);
        ub_ = (R)kUsU0 + (R)kUsDu * (R)jb + (R)kUsDu * O::dv(L - b0, b1 - b0);
    }
    const R u = us_lerp<R>(t, ua_, ub_);
    return x < (R)0 ? -u : u;
}

// Guide bin of logit(xi) and L = ln(xi) (< 0 strictly: node 250, ln CDF = 0,
// always bounds the search).
template <typename R>
__device__ __forceinline__ int us_bin(R xi, R& L)
{
    using O = Ops<R>;
    L = fmin(O::ln(xi), (R)-1e-30);
    const R w = L - O::ln((R)1 - xi);
    int m = (int)((w + (R)kGuideW) * (R)(kGuideN / (2.0 * kGuideW)));
    return m < 0 ? 0 : (m > kGuideN - 1 ? kGuideN - 1 : m);
}

// ---------------------------------------------------------------- packet state

// Per-lane event counters (summed over the CTA at the end of a model).
struct LaneStats {
    unsigned esc, des, stuck, absorbed;     // packets of one lane (every emitted one ends in one of these)
    unsigned scat, cross;                   // kept below 2^31 (end_packet)
};

template <typename R>
struct Pkt {
    int cx, cy, cz, c;
    R px, py, pz;
    R nx, ny, nz;
    R ix, iy, iz;          // 1 / n
    R x, tau;
    float4 rec;            // current cell record
    uint32_t nscat, ncross;
    unsigned long long id;
    uint32_t vis_scat;     // scatterings in this cell visit
    R vis_exc;             // sum w ds H over this cell visit
    R wgt;                 // packet weight (continuum absorption; 1 otherwise)
    R vis_abs;             // weight absorbed by the continuum over this visit
    bool prev_scat;        // last event was a scattering (draw the next one early)
    uint32_t cellsum;      // FP64 walk: sum of the cells of its scatterings (mod 2^32)
};

// n . V/b of a cell, always evaluated in this one fixed order (explicit
// fused multiply-adds): the comoving frequency x_lab - n.V/b then recovers
// exactly the value that x_lab was built from (e.g. 0 for line-centre
// emission), whose sign the velocity sampler's symmetry depends on.
template <typename R>
__device__ __forceinline__ R vdot(R nx, R ny, R nz, const float4& rec)
{
    if constexpr (sizeof(R) == 4) return fmaf(nz, rec.w, fmaf(ny, rec.z, __fmul_rn(nx, rec.y)));
    else return fma(nz, (R)rec.w, fma(ny, (R)rec.z, nx * (R)rec.y));
}

// The FP64 walk keeps 1 / n with the direction (its face distances are
// taken every event, as the oracle takes them); the FP32 walk forms them
// only when a packet crosses a face.
template <typename R>
__device__ __forceinline__ void set_dir(Pkt<R>& p, R nx, R ny, R nz)
{
    p.nx = nx;
    p.ny = ny;
    p.nz = nz;
    if constexpr (sizeof(R) == 8) {
        p.ix = Ops<R>::rcp(nx);
        p.iy = Ops<R>::rcp(ny);
        p.iz = Ops<R>::rcp(nz);
    }
}

// Distance (in cell widths) to the face ahead along one axis, from the
// in-cell coordinate q in [0, 1] and the direction component n with 1/n.
template <typename R>
__device__ __forceinline__ R face_dist(R q, R n, R in)
{
    if constexpr (sizeof(R) == 4) {
        return fmaf(-q, in, in > 0.0f ? in : 0.0f);      // (1 - q)/n or -q/n
    } else {
        return n > 0.0 ? (1.0 - q) * in : (n < 0.0 ? -q * in : 1.0e300);
    }
}

template <typename R>
__device__ __forceinline__ void iso_dir(R umu, R uphi, R& nx, R& ny, R& nz)
{
    R mu = (R)2 * umu - (R)1;
    R st = Ops<R>::sq(fmax((R)0, (R)1 - mu * mu));
    R s, c;
    Ops<R>::sc2pi(uphi, &s, &c);
    nx = st * c;
    ny = st * s;
    nz = mu;
}

__device__ __forceinline__ int spectrum_bin(const TransportArgs& A, double x)
{
    if (x < A.spec_lo) return 0;
    if (x >= A.spec_hi) return A.spec_n + 1;
    const int b = 1 + (int)floor((x - A.spec_lo) / (A.spec_hi - A.spec_lo) * A.spec_n);
    return b > A.spec_n ? A.spec_n : b;
}

// The FP32 walk finds the bin in single precision and takes the FP64 form
// (whose divide alone keeps an SM's FP64 pipe busy for some 400 cycles) only
// where the place in the bin is within the single-precision error of an
// edge: q = x sc + off has an error below 2e-7 (|x sc| + |off|), the margin
// is 1e-6 of that sum. Inf and NaN fail both tests.
template <typename R>
__device__ __forceinline__ void spectrum_add(const TransportArgs& A, R x, R w)
{
    int b = -1;
    if constexpr (sizeof(R) == 4) {
        const float q = fmaf(x, A.spec_sc, A.spec_off);
        const float m = fmaf(fabsf(x), A.spec_msc, A.spec_moff);
        const float fl = floorf(q), fr = q - fl;
        if (fr > m && fr < 1.0f - m) b = fl < 0.0f ? 0 : (fl >= (float)A.spec_n ? A.spec_n + 1 : 1 + (int)fl);
    }
    if (b < 0) b = spectrum_bin(A, (double)x);
    atomicAdd(A.spec_w + b, (double)w);
    atomicAdd(A.spec_c + b, 1ull);
}

template <typename R>
__device__ __forceinline__ void write_record(const TransportArgs& A, const Pkt<R>& p, uint16_t status)
{
    if (!A.rec) return;
    krl_packet_record& r = A.rec[p.id - A.first];       // (cell0 is written at emission)
    r.x = (float)p.x;
    r.nscat = p.nscat;
    r.ncross = p.ncross;
    r.status = status;
    r.pad = 0;
    r.scat_cells = sizeof(R) == 8 ? p.cellsum : 0u;
}

// X = dim u, u = (2 (r >> 9) + 1) 2^-24 the uniform of word r: the product is
// exact in 64-bit integers. Its cell and the place in the cell, as floor(X)
// and X - floor(X) give them.
template <typename R>
__device__ __forceinline__ void place_uniform(int dim, uint32_t r, int& c, R& q, bool& on)
{
    const unsigned long long v = (unsigned long long)(unsigned)dim * (2u * (r >> 9) + 1u);
    const unsigned low = (unsigned)v & 0xffffffu;
    c = (int)(v >> 24);
    q = (R)low * (R)0x1p-24;
    on = low == 0u;
}

// First cell with cdf > uc, uc = (2 K + 1) 2^-49 with K the 48 bits of two
// words. The guide's bin (the top 16 bits of uc) bounds it between two
// neighbouring entries; CDF values are not negative, so their order is that
// of their bits as integers. Uses no FP64 instruction.
__device__ __forceinline__ int pick_cell(const TransportArgs& A, uint32_t w0, uint32_t w1)
{
    const unsigned long long v = ((unsigned long long)(w0 >> 8) << 25) | (2u * (w1 >> 8) + 1u);
    const int top = 63 - __clzll((long long)v);                  // uc = 1.x 2^(top - 49)
    const unsigned long long uc =
        ((unsigned long long)(1023 + top - 49) << 52) | ((v << (52 - top)) & 0xfffffffffffffull);
    const unsigned bin = w0 >> (32 - kCdfGuideBits);
    int l = __ldg(A.src_guide + bin), h = __ldg(A.src_guide + bin + 1);
    const long long* cdf = reinterpret_cast<const long long*>(A.src_cdf);
    while (l < h) {
        const int m = (int)(((unsigned)l + (unsigned)h) >> 1);
        if (__ldg(cdf + m) > (long long)uc) h = m;
        else l = m + 1;
    }
    return l;
}

// Emission (event 0). Slots: block 0 = {mu, phi, tau, freq1},
// block 1 = {freq2, pos_a, pos_b, pos_c}, block 2 = {cell_hi, cell_lo}.
// Returns false if the source point lies outside the domain (the packet
// then leaves at once). The position is formed without FP64 arithmetic
// (except a beam's band): a warp emits for the few lanes that are idle, and
// where packets have tens of events the FP64 pipe, at 16 cycles per warp
// instruction, was the bound of the whole walk (70 % busy on the 128^3
// cloud, 86 events per packet).
template <typename R, unsigned F>
__device__ __forceinline__ bool emit(const TransportArgs& A, const RoundKeys& K, Pkt<R>& p)
{
    using O = Ops<R>;
    const uint32_t lo = (uint32_t)p.id, hi = (uint32_t)(p.id >> 32);
    Words b0 = philox(lo, hi, 0u, 0u, K);
    const bool need1 = A.src_kind != KRL_SRC_POINT || A.src_profile == KRL_PROFILE_GAUSSIAN;
    Words b1 = {{0u, 0u, 0u, 0u}};
    if (need1) b1 = philox(lo, hi, 0u, 1u, K);
    const int dims[3] = {A.nx, A.ny, A.nz};
    R n[3], pp[3];
    int ci[3];
    bool on[3];                 // exactly on the cell's lower face
    if (A.src_kind == KRL_SRC_VOLUME) {
        iso_dir<R>(O::uni(b0.w[0]), O::uni(b0.w[1]), n[0], n[1], n[2]);
        const Words b2 = philox(lo, hi, 0u, 2u, K);
        const int l = pick_cell(A, b2.w[0], b2.w[1]);
        const int row = l / A.nx;
        ci[0] = l - row * A.nx;
        ci[2] = row / A.ny;
        ci[1] = row - ci[2] * A.ny;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            pp[d] = O::uni(b1.w[1 + d]);
            on[d] = false;
        }
    } else if (A.src_kind == KRL_SRC_BEAM) {
        int q = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            const bool along = d == A.src_axis;
            n[d] = along ? (R)1 : (R)0;
            ci[d] = 0;
            pp[d] = (R)0;
            on[d] = along;
            if (!along) {
                const uint32_t r = q == 0 ? b1.w[1] : b1.w[2];
                if (d == A.band_axis) {
                    const double X = A.band_lo + (A.band_hi - A.band_lo) * (double)O::uni(r);
                    const double f = floor(X);
                    ci[d] = (int)f;
                    pp[d] = (R)(X - f);
                    on[d] = X - f == 0.0;
                } else {
                    place_uniform<R>(dims[d], r, ci[d], pp[d], on[d]);
                }
                ++q;
            }
        }
    } else {
        iso_dir<R>(O::uni(b0.w[0]), O::uni(b0.w[1]), n[0], n[1], n[2]);
        int q = 0;
#pragma unroll
        for (int d = 0; d < 3; ++d) {
            ci[d] = A.src_c[d];
            pp[d] = (R)A.src_q[d];
            on[d] = (A.src_on >> d) & 1u;
            if (A.src_kind == KRL_SRC_PLANE && d != A.src_axis)
                place_uniform<R>(dims[d], q++ == 0 ? b1.w[1] : b1.w[2], ci[d], pp[d], on[d]);
        }
    }
    set_dir(p, n[0], n[1], n[2]);
    bool inside = true;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        int c = ci[d];
        if (on[d] && n[d] < (R)0) {
            c -= 1;
            pp[d] = (R)1;
        }
        if (((A.periodic >> d) & 1u) && (c < 0 || c >= dims[d])) {
            c %= dims[d];
            if (c < 0) c += dims[d];
        }
        if (c < 0 || c >= dims[d]) inside = false;
        ci[d] = c;
    }
    p.tau = fmax((R)0, -O::ln(O::uni(b0.w[2])));
    R xcom = (R)0;
    if (A.src_profile == KRL_PROFILE_GAUSSIAN) {
        R s, c;
        O::sc2pi(O::uni(b1.w[0]), &s, &c);
        xcom = O::sq(fmax((R)0, -O::ln(O::uni(b0.w[3])))) * c;
    }
    p.nscat = 0;
    p.ncross = 0;
    p.cellsum = 0;
    p.vis_scat = 0;
    p.vis_exc = (R)0;
    p.wgt = (R)1;
    p.vis_abs = (R)0;
    p.prev_scat = true;
    if (!inside) {
        p.x = xcom;
        if (A.rec) A.rec[p.id - A.first].cell0 = 0xFFFFFFFFu;
        return false;
    }
    p.cx = ci[0];
    p.cy = ci[1];
    p.cz = ci[2];
    p.px = pp[0];
    p.py = pp[1];
    p.pz = pp[2];
    p.c = (ci[2] * A.ny + ci[1]) * A.nx + ci[0];
    if (A.rec) A.rec[p.id - A.first].cell0 = (uint32_t)p.c;
    p.rec = __ldg(A.cells + p.c);
    R vdn = (F & F_VEL) ? vdot<R>(p.nx, p.ny, p.nz, p.rec) : (R)0;
    p.x = xcom + vdn;
    return true;
}

// Camera m's share of one segment's emissivity (Eq. scat-line with the
// trilinear R_IIA table, Eq. riia-table, or Eq. riia-inf for |x_in| >= 120):
// the channels k with |x_out,k - x_com| <= 10, x_out,k = -(x0 + (k + 1/2) dx)
// - n_cam.V/b, each receive base R(x_out,k - x_com; x_com, g), g = n.n_cam.
// emiss_setup holds what depends on the segment and camera only: the channel
// range, n_cam.V/b and either the table cell (g node kg, x node j, packed as
// kg << 8 | j, and the four (g, x) corner weights) or, in the wing limit
// (cell < 0), the Gaussian's normalisation (w00) and 1 / (2 var) (w01).
template <typename R>
struct EmSetup {
    int k0, k1;            // channel range; empty when k0 > k1
    int cell;              // kg << 8 | j, or -1
    R vc, sgn;             // n_cam.V/b; sign of x_com (R(D; -x, g) = R(-D; x, g))
    R w00, w01, w10, w11;
    R x0, dx;              // channel origin and width in x units
};

template <typename R, bool VEL>
__device__ __forceinline__ EmSetup<R> emiss_setup(const TransportArgs& A, int m, const float4& rec, R nx, R ny, R nz,
                                                  R xcom)
{
    EmSetup<R> S;
    S.x0 = (R)A.ch_x0;
    S.dx = (R)A.ch_dx;
    const R axc = fabs(xcom);
    S.sgn = xcom < (R)0 ? (R)-1 : (R)1;
    const R cx = (R)A.cam[m][0], cy = (R)A.cam[m][1], cz = (R)A.cam[m][2];
    R g = nx * cx + ny * cy + nz * cz;
    g = fmin((R)1, fmax((R)-1, g));
    S.vc = VEL ? vdot<R>(cx, cy, cz, rec) : (R)0;
    // channels with |x_out,k - x_com| <= 10
    const R ctr = Ops<R>::dv(-S.x0 - S.vc - xcom, S.dx) - (R)0.5;
    const R span = Ops<R>::dv((R)kRdMax, S.dx);
    const int k0 = (int)ceil(ctr - span) - 1;
    const int k1 = (int)floor(ctr + span) + 1;
    S.k0 = k0 < 0 ? 0 : k0;
    S.k1 = k1 > A.n_ch - 1 ? A.n_ch - 1 : k1;
    if (axc >= (R)kRxMax) {
        const R v = fmax((R)1 - g, (R)(kRsMin * kRsMin));
        S.cell = -1;
        S.w00 = (R)1 / Ops<R>::sq((R)6.283185307179586 * v);
        S.w01 = (R)0.5 / v;
        S.w10 = S.w11 = (R)0;
        return S;
    }
    const R fx = axc * (R)((kRnX - 1) / kRxMax);
    const R fg = (g + (R)1) * (R)((kRnG - 1) / 2.0);
    int j = (int)fx;
    int kg = (int)fg;
    j = j > kRnX - 2 ? kRnX - 2 : j;
    kg = kg > kRnG - 2 ? kRnG - 2 : kg;
    const R wx = fx - (R)j, wg = fg - (R)kg;
    S.cell = kg << 8 | j;
    S.w00 = ((R)1 - wg) * ((R)1 - wx);
    S.w01 = ((R)1 - wg) * wx;
    S.w10 = wg * ((R)1 - wx);
    S.w11 = wg * wx;
    return S;
}

// x_out,k - x_com of channel k (kf = k as R).
template <typename R>
__device__ __forceinline__ R emiss_delta(const EmSetup<R>& S, R xcom, R kf)
{
    const R xo = -(S.x0 + (kf + (R)0.5) * S.dx) - S.vc;
    return xo - xcom;
}

// The table's interval of Delta = Dd and the weight of its upper node.
template <typename R>
__device__ __forceinline__ void emiss_node(R Dd, int& i, R& wd)
{
    const R fd = (Dd + (R)kRdMax) * (R)(1.0 / kRdStep);
    if constexpr (sizeof(R) == 4) {
        // floor(fd) for 0 <= fd < 2^23 by a round-down add of 2^23 (exact),
        // clamped to the last interval, without float/int conversions
        const float t = __fadd_rd(fd, 8388608.0f) - 8388608.0f;
        const float fi = fminf(fmaxf(t, 0.0f), (float)(kRnD - 2));
        i = __float_as_int(fi + 8388608.0f) - 0x4B000000;
        wd = fd - fi;
    } else {
        i = (int)floor(fd);
        i = i < 0 ? 0 : (i > kRnD - 2 ? kRnD - 2 : i);
        wd = fd - (R)i;
    }
}

// Channel k of a segment's camera share, added to out[k] (the cell's row of
// that camera's cube) by one thread, from the plain table.
template <typename R>
__device__ __forceinline__ void emiss_channel(const TransportArgs& A, float* out, const EmSetup<R>& S, R xcom, R base,
                                              int k, R kf)
{
    const R D = emiss_delta<R>(S, xcom, kf);
    if (fabs(D) > (R)kRdMax) return;
    if (S.cell < 0) {
        atomicAdd(out + k, (float)(base * S.w00 * Ops<R>::ex(-D * D * S.w01)));
        return;
    }
    int i;
    R wd;
    emiss_node<R>(S.sgn * D, i, wd);
    const int kg = S.cell >> 8, j = S.cell & 255;
    const float* r00 = A.rtab + ((size_t)kg * kRnX + j) * kRnD;
    const float* r01 = r00 + kRnD;
    const float* r10 = r00 + (size_t)kRnX * kRnD;
    const float* r11 = r10 + kRnD;
    const R a0 = S.w00 * (R)__ldg(r00 + i) + S.w01 * (R)__ldg(r01 + i) + S.w10 * (R)__ldg(r10 + i) +
                 S.w11 * (R)__ldg(r11 + i);
    const R a1 = S.w00 * (R)__ldg(r00 + i + 1) + S.w01 * (R)__ldg(r01 + i + 1) + S.w10 * (R)__ldg(r10 + i + 1) +
                 S.w11 * (R)__ldg(r11 + i + 1);
    const R val = ((R)1 - wd) * a0 + wd * a1;
    atomicAdd(out + k, (float)(base * val));
}

// Camera m's share deposited by one thread (inside the walk).
template <typename R, bool VEL>
__device__ __forceinline__ void emiss_camera(const TransportArgs& A, int m, int c, const float4& rec, R nx, R ny,
                                             R nz, R xcom, R base)
{
    const EmSetup<R> S = emiss_setup<R, VEL>(A, m, rec, nx, ny, nz, xcom);
    if (S.k0 > S.k1) return;
    float* out = A.emiss + ((size_t)m * A.ncell + c) * A.n_ch;
    R kf = (R)S.k0;
    for (int k = S.k0; k <= S.k1; ++k, kf += (R)1) emiss_channel<R>(A, out, S, xcom, base, k, kf);
}

// Marks segment records [i, i + n) as empty.
__device__ __forceinline__ void clear_segments(const TransportArgs& A, unsigned long long i, unsigned n)
{
    for (unsigned k = 0; k < n; ++k)
        if (i + k < A.seg_cap) A.seg[2 * (i + k)] = make_float4(__int_as_float(-1), 0.0f, 0.0f, 0.0f);
}

// First stage of the two-stage emissivity deposit (FP32 walk): the segment
// (cell, base weight, x_com, direction) goes to the run's segment buffer, one
// slot range per converged group of lanes. A warp takes slots from a chunk of
// seg_chunk records of its own (*word: the next one; at a multiple of the
// chunk there is none), so that the buffer's counter takes one atomic per
// chunk: one per group made that single address the bound of the walk (0.8e6
// atomics, each waited for, in a 3 ms run). What a chunk has left when a
// group does not fit is marked empty. seg_chunk 0 (a buffer too small to
// leave each warp a chunk): every group takes its slots from the counter.
// Returns false when the buffer is full; the caller then deposits the segment
// itself.
__device__ __forceinline__ bool append_segment(const TransportArgs& A, unsigned long long* word, int c, float base,
                                               float xcom, float nx, float ny, float nz)
{
    const unsigned mask = __activemask();
    const unsigned lane = threadIdx.x & 31u;
    const int leader = __ffs(mask) - 1;
    unsigned long long first = 0;
    if ((int)lane == leader) {
        const unsigned cnt = (unsigned)__popc(mask), chunk = A.seg_chunk;
        if (chunk == 0u) {
            first = atomicAdd(A.seg_count, (unsigned long long)cnt);
        } else {
            // another group of this warp may take slots in between: the swap
            // then fails and the new word is looked at (at most 31 times)
            unsigned long long old = *reinterpret_cast<volatile unsigned long long*>(word);
            for (;;) {
                if (old >= A.seg_cap) {         // the buffer is full: nothing to take
                    first = old;
                    break;
                }
                const unsigned left = (unsigned)(0ull - old) & (chunk - 1u);
                const bool fits = cnt <= left;
                first = fits ? old : atomicAdd(A.seg_count, (unsigned long long)chunk);
                const unsigned long long seen = atomicCAS(word, old, first + cnt);
                if (seen == old) {
                    if (!fits) clear_segments(A, old, left);
                    break;
                }
                if (!fits) clear_segments(A, first, chunk);
                old = seen;
            }
        }
    }
    first = __shfl_sync(mask, first, leader);
    const unsigned long long i = first + __popc(mask & ((1u << lane) - 1u));
    if (i >= A.seg_cap) return false;
    A.seg[2 * i] = make_float4(__int_as_float(c), base, xcom, nx);
    A.seg[2 * i + 1] = make_float4(ny, nz, 0.0f, 0.0f);
    return true;
}

// Per-segment tallies of the rich mode: mean intensity by comoving channel
// and the camera-directed emissivity (Eq. scat-line). With a segment buffer
// (FP32 walk) the emissivity is deposited by the second stage instead.
template <typename R, unsigned F>
__device__ void rich_segment(const TransportArgs& A, const Tabs& T, int c, const float4& rec, R nx, R ny, R nz, R ds, R xcom, R H, R w)
{
    if ((A.rich & KRL_TALLY_J) && A.n_ch > 0) {
        R q = Ops<R>::dv(-xcom - (R)A.ch_x0, (R)A.ch_dx);
        if (q >= (R)0 && q < (R)A.n_ch) atomicAdd(A.J + (size_t)c * A.n_ch + (int)q, (double)(w * ds));
    }
    if (!(A.rich & KRL_TALLY_EMISS) || A.n_ch <= 0) return;
    const R base = w * ds * (R)rec.x * H * (R)0.079577471545947668;   // 1 / 4 pi
    if constexpr (sizeof(R) == 4) {
        if (A.seg && append_segment(A, T.segw, c, base, xcom, nx, ny, nz)) return;
    }
    for (int m = 0; m < A.n_cam; ++m) emiss_camera<R, (F & F_VEL) != 0>(A, m, c, rec, nx, ny, nz, xcom, base);
}

// Second stage of the emissivity deposit. A warp takes 32 consecutive
// segment records (one per lane, coalesced). Per camera each lane works out
// its own segment's setup, trimmed to the channels within reach, and puts it
// into shared memory; the warp then goes over all (segment, channel) items of
// the 32 segments, 16 at a time, two lanes per item: each of the two reads one
// Delta node of the regrouped R_IIA table (16 of the same 32 bytes), the even
// one combines them and adds. What bounds this is the L1 data pipe, a
// wavefront per table line touched (the channels of a segment lie several
// nodes apart): with one lane per item reading both nodes every line was
// touched twice, and a segment filled 5 to 19 of the warp's 32 lanes (128^3
// envelope, 64 channels, 3 cameras, 1.3e7 segments: 4.9 -> 4.3 ms; 5 CTAs per
// SM, of 4: 4.6, 6: 5.0). The record count is read on the device (no host
// round trip between the stages).
constexpr int kDepositBlock = 256;

struct DepositItems {
    float4 a[32];       // {first channel, table cell (kg << 8 | j, or -1), x_com, base}
    float4 w[32];       // corner weights (or the wing limit's two numbers)
    float4 b[32];       // {n_cam.V/b, sign of x_com, grid cell, first item}
};

template <bool VEL>
__global__ void __launch_bounds__(kDepositBlock, 5) k_emiss_deposit(const __grid_constant__ TransportArgs A)
{
    __shared__ DepositItems items[kDepositBlock / 32];
    DepositItems& it = items[threadIdx.x >> 5];
    const unsigned long long cnt = *A.seg_count;
    const unsigned long long n = cnt < A.seg_cap ? cnt : A.seg_cap;
    const int lane = (int)(threadIdx.x & 31u);
    const unsigned long long stride = ((unsigned long long)gridDim.x * blockDim.x) & ~31ull;
    for (unsigned long long w = ((unsigned long long)blockIdx.x * blockDim.x + threadIdx.x) & ~31ull; w < n;
         w += stride) {
        const unsigned long long i = w + (unsigned long long)lane;
        float4 r0 = make_float4(__int_as_float(-1), 0.0f, 0.0f, 0.0f), r1 = r0;
        if (i < n) {
            r0 = __ldg(A.seg + 2 * i);
            r1 = __ldg(A.seg + 2 * i + 1);
        }
        const bool valid = __float_as_int(r0.x) >= 0;       // (not an empty record)
        const int c = valid ? __float_as_int(r0.x) : 0;
        const float4 rec = (VEL && valid) ? __ldg(A.cells + c) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        const float base = r0.y, xcom = r0.z;
        for (int m = 0; m < A.n_cam; ++m) {
            EmSetup<float> S = emiss_setup<float, VEL>(A, m, rec, r0.w, r1.x, r1.y, xcom);
            // the range has up to two channels too many at each end
            for (int q = 0; q < 2; ++q) {
                if (S.k0 <= S.k1 && fabsf(emiss_delta<float>(S, xcom, (float)S.k0)) > (float)kRdMax) ++S.k0;
                if (S.k0 <= S.k1 && fabsf(emiss_delta<float>(S, xcom, (float)S.k1)) > (float)kRdMax) --S.k1;
            }
            const int mine = valid && S.k0 <= S.k1 ? S.k1 - S.k0 + 1 : 0;
            int sum = mine;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int v = __shfl_up_sync(kFull, sum, o);
                if (lane >= o) sum += v;
            }
            const int first = sum - mine, total = __shfl_sync(kFull, sum, 31);
            const unsigned some = __ballot_sync(kFull, mine > 0);
            if (mine > 0) {
                const int r = __popc(some & ((1u << lane) - 1u));
                it.a[r] = make_float4(__int_as_float(S.k0), __int_as_float(S.cell), xcom, base);
                it.w[r] = make_float4(S.w00, S.w01, S.w10, S.w11);
                it.b[r] = make_float4(S.vc, S.sgn, __int_as_float(c), __int_as_float(first));
            }
            __syncwarp();
            const float4* quads = A.rquad;
            float* cube = A.emiss + (size_t)m * A.ncell * A.n_ch;
            const int slot = lane >> 1;
            int started = 0;            // segments that begin before this window of 16 items
            for (int e0 = 0; e0 < total; e0 += 16) {
                const unsigned bit = mine > 0 && first >= e0 && first < e0 + 16 ? 1u << (first - e0) : 0u;
                const unsigned begins = __reduce_or_sync(kFull, bit);
                const int e = e0 + slot;
                const bool on = e < total;
                const int s = on ? started + __popc(begins & ((2u << slot) - 1u)) - 1 : 0;
                started += __popc(begins);
                const float4 sa = it.a[s], sw = it.w[s], sb = it.b[s];
                EmSetup<float> T;
                T.x0 = S.x0;
                T.dx = S.dx;
                T.vc = sb.x;
                T.sgn = sb.y;
                T.cell = __float_as_int(sa.y);
                const int k = __float_as_int(sa.x) + (e - __float_as_int(sb.w));
                const float kf = __int_as_float(0x4B000000 + k) - 8388608.0f;      // (float)k, k < 2^23
                const float D = emiss_delta<float>(T, sa.z, kf);
                const bool near = on && !(fabsf(D) > (float)kRdMax);       // (NaN counts, as in emiss_channel)
                float val = 0.0f;
                const bool table = near && T.cell >= 0;
                int node = 0;
                float wd = 0.0f;
                emiss_node<float>(T.sgn * D, node, wd);
                float4 q = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
                if (table) {
                    const int kg = T.cell >> 8, j = T.cell & 255;
                    q = __ldg(quads + ((size_t)kg * (kRnX - 1) + j) * kRnD + node + (lane & 1));
                }
                const float av = sw.x * q.x + sw.y * q.y + sw.z * q.z + sw.w * q.w;
                const float a1 = __shfl_down_sync(kFull, av, 1);        // the odd lane's
                val = (1.0f - wd) * av + wd * a1;
                if (near && T.cell < 0) val = sw.x * Ops<float>::ex(-D * D * sw.y);
                if (near && !(lane & 1)) atomicAdd(cube + (size_t)__float_as_int(sb.z) * A.n_ch + k, sa.w * val);
            }
            __syncwarp();
        }
    }
}

// lead: whether this lane writes (false in the other lanes of a group that
// walks one packet together).
template <typename R, unsigned F>
__device__ __forceinline__ void flush_visit(const TransportArgs& A, Pkt<R>& p, bool lead = true)
{
    if constexpr (sizeof(R) == 8) p.cellsum += p.vis_scat * (uint32_t)p.c;
    if (lead) {
        if ((F & F_SCAT) && p.vis_scat && A.scat) atomicAdd(A.scat + p.c, (unsigned long long)p.vis_scat);
        if ((F & F_RICH) && (A.rich & KRL_TALLY_EXC) && p.vis_exc != (R)0) atomicAdd(A.exc + p.c, (double)p.vis_exc);
        if ((F & F_RICH) && A.tau_abs && p.vis_abs != (R)0) atomicAdd(A.absw + p.c, (double)p.vis_abs);
    }
    p.vis_scat = 0;
    p.vis_exc = (R)0;
    p.vis_abs = (R)0;
}

template <typename T>
__device__ __forceinline__ T warp_sum(T v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
    return v;
}

// Launch shape per instantiation, two CTAs per SM each (shared memory holds
// two CTAs' tables). F_WIDE: the lean FP32 walk in 512-thread CTAs (64
// registers each) and the rich one without per-segment tallies in 384 (80
// registers), for throughput; all others, and these two where a launch is set
// by its longest packets, in 256 (up to 128 registers, which the walk of the
// last packets uses: a step of its frequency chain takes 136 cycles, 173 with
// 64 registers). On the 128^3 cloud (86 events per packet; 16 warps per SM
// issued in half the cycles) 384 threads took the Lambda cycle from 79 to
// 66 ms, 512 (with spills) 75.
constexpr int kLeanBlock = 512, kLightBlock = 384;
template <typename R, unsigned F>
constexpr int max_block()
{
    return sizeof(R) == 8 || !(F & F_WIDE) ? 256 : ((F & F_RICH) ? kLightBlock : kLeanBlock);
}

// ---------------------------------------------------------------- tail compaction
//
// Dynamic shared memory after the tables: a control block (the CTA's "ids
// ran out" flag and per-warp packet counts, double-buffered by round) and a
// stash that holds one packet per thread, field-major (one 32-bit word per
// field and slot, so consecutive slots fall in consecutive banks).
constexpr size_t kCtlOff = (kSmemBytes + 15) / 16 * 16;
constexpr int kCtlInts = 4 + 2 * 32 + 2 * 16;         // ... and a 64-bit word per warp
constexpr size_t kStashOff = kCtlOff + (size_t)kCtlInts * sizeof(int);
// Events a lane runs between two compaction checks in the tail.
constexpr int kTailRound = 32;
// Bulk-phase iterations between two reads of the CTA's stop flag by a warp
// with no idle lane.
constexpr int kBulkCheck = 16;

// Words per stashed packet: cell (c, cx, cy, cz), nscat, ncross, id
// (2 words), the scattering-cell sum (FP64 walk), and px, py, pz, nx, ny, nz,
// x, tau (and the weight in the rich walk) in R.
template <typename R, unsigned F>
constexpr int stash_words() { return 8 + (sizeof(R) == 8 ? 1 : 0) + ((F & F_RICH) ? 9 : 8) * (int)(sizeof(R) / 4); }

// (the stash, or the buffers of the last packets' walk in its place)
template <typename R, unsigned F>
constexpr size_t smem_bytes(int block, int tail_warps);

template <typename R>
__device__ __forceinline__ void put_r(uint32_t* w, int& f, int n, int slot, R v)
{
    if constexpr (sizeof(R) == 4) {
        w[(f++) * n + slot] = __float_as_uint(v);
    } else {
        w[(f++) * n + slot] = (uint32_t)__double2loint(v);
        w[(f++) * n + slot] = (uint32_t)__double2hiint(v);
    }
}

template <typename R>
__device__ __forceinline__ R get_r(const uint32_t* w, int& f, int n, int slot)
{
    if constexpr (sizeof(R) == 4) {
        return __uint_as_float(w[(f++) * n + slot]);
    } else {
        const uint32_t lo = w[(f++) * n + slot];
        const uint32_t hi = w[(f++) * n + slot];
        return __hiloint2double((int)hi, (int)lo);
    }
}

// Moves a packet into / out of stash slot `slot`. The visit tallies are
// flushed before (they belong to the cell visit, not the packet), and the
// derived fields (1/n, the cell record) are recomputed from the stored ones
// by the same functions, so a restored packet continues bit for bit as it
// would have in its old lane.
template <typename R, unsigned F>
__device__ __forceinline__ void stash_put(uint32_t* w, int n, int slot, const Pkt<R>& p)
{
    int f = 0;
    w[(f++) * n + slot] = (uint32_t)p.c;
    w[(f++) * n + slot] = (uint32_t)p.cx;
    w[(f++) * n + slot] = (uint32_t)p.cy;
    w[(f++) * n + slot] = (uint32_t)p.cz;
    w[(f++) * n + slot] = p.nscat;
    w[(f++) * n + slot] = p.ncross;
    w[(f++) * n + slot] = (uint32_t)p.id;
    w[(f++) * n + slot] = (uint32_t)(p.id >> 32);
    if constexpr (sizeof(R) == 8) w[(f++) * n + slot] = p.cellsum;
    put_r<R>(w, f, n, slot, p.px);
    put_r<R>(w, f, n, slot, p.py);
    put_r<R>(w, f, n, slot, p.pz);
    put_r<R>(w, f, n, slot, p.nx);
    put_r<R>(w, f, n, slot, p.ny);
    put_r<R>(w, f, n, slot, p.nz);
    put_r<R>(w, f, n, slot, p.x);
    put_r<R>(w, f, n, slot, p.tau);
    if (F & F_RICH) put_r<R>(w, f, n, slot, p.wgt);
}

template <typename R, unsigned F>
__device__ __forceinline__ void stash_get(const TransportArgs& A, const uint32_t* w, int n, int slot, Pkt<R>& p)
{
    int f = 0;
    p.c = (int)w[(f++) * n + slot];
    p.cx = (int)w[(f++) * n + slot];
    p.cy = (int)w[(f++) * n + slot];
    p.cz = (int)w[(f++) * n + slot];
    p.nscat = w[(f++) * n + slot];
    p.ncross = w[(f++) * n + slot];
    const uint32_t lo = w[(f++) * n + slot];
    const uint32_t hi = w[(f++) * n + slot];
    p.id = ((unsigned long long)hi << 32) | lo;
    if constexpr (sizeof(R) == 8) p.cellsum = w[(f++) * n + slot];
    p.px = get_r<R>(w, f, n, slot);
    p.py = get_r<R>(w, f, n, slot);
    p.pz = get_r<R>(w, f, n, slot);
    const R nx = get_r<R>(w, f, n, slot);
    const R ny = get_r<R>(w, f, n, slot);
    const R nz = get_r<R>(w, f, n, slot);
    set_dir(p, nx, ny, nz);
    p.x = get_r<R>(w, f, n, slot);
    p.tau = get_r<R>(w, f, n, slot);
    p.wgt = (F & F_RICH) ? get_r<R>(w, f, n, slot) : (R)1;
    p.rec = __ldg(A.cells + p.c);
    p.vis_scat = 0;
    p.vis_exc = (R)0;
    p.vis_abs = (R)0;
    p.prev_scat = true;
}

// ---------------------------------------------------------------- one event

// Continuum absorption over a segment of optical depth dt (Eq. scat-line):
// ab = 1 - exp(-dt) is the absorbed fraction of the weight, and the
// returned factor (1 - exp(-dt))/dt the segment's mean weight per unit
// starting weight (its series below dt = 1e-4).
template <typename R>
__device__ __forceinline__ R seg_factor(R dt, R& ab)
{
    if constexpr (sizeof(R) == 4) ab = -expm1f(-dt);
    else ab = -expm1(-dt);
    if (dt < (R)1e-4) return (R)1 - dt * ((R)0.5 - dt * ((R)(1.0 / 6.0) - dt * (R)(1.0 / 24.0)));
    return ab / dt;
}

// Whether the point q lies inside the unit cell ([0, 1] on every axis; false
// for a NaN).
__device__ __forceinline__ bool in_cell(float2 qxy, float qz)
{
    const float2 hxy = __fadd2_rn(qxy, make_float2(-0.5f, -0.5f));
    return fabsf(hxy.x) <= 0.5f && fabsf(hxy.y) <= 0.5f && fabsf(qz - 0.5f) <= 0.5f;
}

// FP32: distance to the nearest face ahead, the axis and 1/n of that face;
// the packet is moved there. A zero component counts as +1e-30 (the packet
// then crosses that face only from exactly on it), so that 1/n is finite and
// its sign alone selects the face ahead.
__device__ __forceinline__ float to_face(Pkt<float>& p, int& axis, float& nd)
{
    using O = Ops<float>;
    const float ix = O::rcp(p.nx != 0.0f ? p.nx : 1e-30f);
    const float iy = O::rcp(p.ny != 0.0f ? p.ny : 1e-30f);
    const float iz = O::rcp(p.nz != 0.0f ? p.nz : 1e-30f);
    float s = face_dist<float>(p.px, p.nx, ix);
    nd = ix;
    axis = 0;
    const float ty = face_dist<float>(p.py, p.ny, iy);
    const float tz = face_dist<float>(p.pz, p.nz, iz);
    if (ty < s) { s = ty; axis = 1; nd = iy; }
    if (tz < s) { s = tz; axis = 2; nd = iz; }
    p.px = O::step01(p.px, s, p.nx);
    p.py = O::step01(p.py, s, p.ny);
    p.pz = O::step01(p.pz, s, p.nz);
    return s;
}

// A packet's end: status 1 escaped, 2 destroyed, 3 budget, 4 absorbed.
template <typename R>
__device__ __forceinline__ void end_packet(const TransportArgs& A, const Pkt<R>& p, uint16_t status,
                                           unsigned& counter, LaneStats& st)
{
    ++counter;
    if ((p.nscat | p.ncross | st.scat | st.cross) >> 30) {      // counts in 32 bits only while the sums fit
        atomicAdd(A.stats + ST_SCAT, (unsigned long long)st.scat + p.nscat);
        atomicAdd(A.stats + ST_CROSS, (unsigned long long)st.cross + p.ncross);
        st.scat = st.cross = 0u;
    } else {
        st.scat += p.nscat;
        st.cross += p.ncross;
    }
    write_record(A, p, status);
}

// The packet, moved to the face on `axis` at distance s, enters the next
// cell. Returns false if it leaves the domain.
template <typename R, unsigned F>
__device__ __forceinline__ bool cross_face(const TransportArgs& A, Pkt<R>& p, R alpha, R s, int axis, R nd,
                                           LaneStats& st, bool lead = true)
{
    if constexpr (sizeof(R) == 4) p.tau = fmaxf(0.0f, fmaf(-alpha, s, p.tau));   // (the two tests may part at a tie)
    else p.tau -= alpha * s;
    ++p.ncross;
    flush_visit<R, F>(A, p, lead);
    const int dim = axis == 0 ? A.nx : (axis == 1 ? A.ny : A.nz);
    const int stride = axis == 0 ? 1 : (axis == 1 ? A.nx : A.nx * A.ny);
    const int cur = axis == 0 ? p.cx : (axis == 1 ? p.cy : p.cz);
    // side from the sign of 1/n, which selected the face
    const int step = nd > (R)0 ? 1 : -1;
    int nc = cur + step;
    int dc = step * stride;
    const R pnew = step > 0 ? (R)0 : (R)1;
    if (axis == 0) p.px = pnew;
    else if (axis == 1) p.py = pnew;
    else p.pz = pnew;
    if (nc < 0 || nc >= dim) {
        if (!((A.periodic >> axis) & 1u)) {
            if (lead) {
                spectrum_add(A, p.x, p.wgt);
                end_packet(A, p, 1, st.esc, st);
            }
            return false;
        }
        if (nc < 0) { nc += dim; dc += dim * stride; }
        else { nc -= dim; dc -= dim * stride; }
    }
    if (axis == 0) p.cx = nc;
    else if (axis == 1) p.cy = nc;
    else p.cz = nc;
    p.c += dc;
    p.rec = __ldg(A.cells + p.c);
    return true;
}

// Cosine g of the scattering angle as g - 1, and sin(gamma).
template <typename R>
__device__ __forceinline__ void scatter_angle(R nx, R ny, R nz, R mx, R my, R mz, R& gm1, R& sg)
{
    R g, s2;
    if constexpr (sizeof(R) == 4) {
        g = fmaf(nz, mz, fmaf(nx, mx, __fmul_rn(ny, my)));
        s2 = fmaf(-g, g, 1.0f);
    } else {
        g = nx * mx + ny * my + nz * mz;
        s2 = (R)1 - g * g;
    }
    sg = Ops<R>::sq(fmax((R)0, s2));
    gm1 = g - (R)1;
}

// x_out = x_in + u_par (g - 1) + u_perp sin(gamma) (Eq. riia-scatter).
template <typename R>
__device__ __forceinline__ R scatter_x(R xcom, R upar, R gm1, R z1, R sg)
{
    if constexpr (sizeof(R) == 4) return fmaf(z1, sg, fmaf(upar, gm1, xcom));
    else return xcom + upar * gm1 + z1 * sg;
}

// Advances an active packet by one event in its current cell (a scattering
// inside the cell or a crossing of the nearest face). Returns false when the
// packet has ended (escape, destruction or event budget).
template <typename R, unsigned F, int PH>
__device__ __forceinline__ bool advance(const TransportArgs& A, const RoundKeys& K, Pkt<R>& p, const Tabs& T, R a, R H0,
                                        LaneStats& st)
{
    using O = Ops<R>;
    if (p.nscat + p.ncross >= A.max_iters32) {
        flush_visit<R, F>(A, p);
        end_packet(A, p, 3, st.stuck, st);
        return false;
    }
    // Draw the next scattering's random numbers up front, for every lane of
    // the converged group, when any of them last scattered (the common case
    // deep in the line core): the lanes then share one pass through Philox
    // instead of the few lanes that follow a face crossing drawing again in
    // a divergent branch, and the chains overlap the lookup's latency. A
    // lane whose event turns out to be a crossing discards its draw.
    const uint32_t idlo = (uint32_t)p.id, idhi = (uint32_t)(p.id >> 32);
    Words w0 = {{0u, 0u, 0u, 0u}}, w1 = {{0u, 0u, 0u, 0u}};
    const bool spec = __any_sync(__activemask(), p.prev_scat);
    if (spec) {
        w0 = philox(idlo, idhi, p.nscat + 1u, 0u, K);
        w1 = philox(idlo, idhi, p.nscat + 1u, 1u, K);
    }
    const R vdn = (F & F_VEL) ? vdot<R>(p.nx, p.ny, p.nz, p.rec) : (R)0;
    const R xcom = p.x - vdn;
    const R H = profile<R, PH>(A, xcom, T.sv, a, H0);
    R alpha;
    if constexpr (sizeof(R) == 4) alpha = __fmul_rn(p.rec.x, H);
    else alpha = (R)p.rec.x * H;
    bool scat;
    R ds, sx_ = (R)0, nd = (R)0;
    int axis = 0;
    if constexpr (sizeof(R) == 4) {
        // FP32: the packet scatters in this cell iff the point at distance
        // tau / alpha along n lies inside the cell ([0, 1] on every axis; a
        // line-free cell gives an infinite or NaN distance: outside). The
        // face distances are needed only for a crossing.
        ds = O::dv(p.tau, alpha);
        const float2 qxy = __ffma2_rn(make_float2(ds, ds), make_float2(p.nx, p.ny), make_float2(p.px, p.py));
        const float qz = fmaf(ds, p.nz, p.pz);
        scat = in_cell(qxy, qz);
        if (scat) {
            p.px = qxy.x;
            p.py = qxy.y;
            p.pz = qz;
        } else {
            sx_ = to_face(p, axis, nd);
            ds = sx_;
        }
    } else {
        // FP64 (the lockstep walk): nearest face first, as the oracle does
        const R tx = face_dist<R>(p.px, p.nx, p.ix);
        const R ty = face_dist<R>(p.py, p.ny, p.iy);
        const R tz = face_dist<R>(p.pz, p.nz, p.iz);
        sx_ = tx;
        nd = p.ix;
        if (ty < sx_) { sx_ = ty; axis = 1; nd = p.iy; }
        if (tz < sx_) { sx_ = tz; axis = 2; nd = p.iz; }
        scat = p.tau < alpha * sx_;
        ds = scat ? O::dv(p.tau, alpha) : sx_;
        p.px = O::step01(p.px, ds, p.nx);
        p.py = O::step01(p.py, ds, p.ny);
        p.pz = O::step01(p.pz, ds, p.nz);
    }
    if (F & F_RICH) {
        // segment tallies at the mean weight along the segment; the weight
        // then decays by the continuum's absorption over it
        R wseg = p.wgt, ab = (R)0;
        if (A.tau_abs) wseg = p.wgt * seg_factor<R>((R)__ldg(A.tau_abs + p.c) * ds, ab);
        if (A.rich & KRL_TALLY_EXC) p.vis_exc = fma(wseg * ds, H, p.vis_exc);
        if ((F & F_SEG) && (A.rich & (KRL_TALLY_J | KRL_TALLY_EMISS))) rich_segment<R, F>(A, T, p.c, p.rec, p.nx, p.ny, p.nz, ds, xcom, H, wseg);
        if (A.tau_abs) {
            p.vis_abs = fma(p.wgt, ab, p.vis_abs);
            p.wgt = p.wgt * ((R)1 - ab);
            if (p.wgt < (R)kWeightCut) {
                flush_visit<R, F>(A, p);
                end_packet(A, p, 4, st.absorbed, st);
                return false;
            }
        }
    }
    p.prev_scat = scat;
    if (scat) {
        // ---- scattering (event e = nscat): block 0 = {u_par, bm_r, bm_phi, tau},
        //      block 1 = {mu, phi, eps_test, -}
        ++p.nscat;
        ++p.vis_scat;
        if (!spec) {
            w0 = philox(idlo, idhi, p.nscat, 0u, K);
            w1 = philox(idlo, idhi, p.nscat, 1u, K);
        }
        if ((F & F_RICH) && (A.rich & kRichEps)) {
            if (O::uni(w1.w[2]) < (R)__ldg(A.eps + p.c)) {
                flush_visit<R, F>(A, p);
                end_packet(A, p, 2, st.des, st);
                return false;
            }
        }
        // independent long-latency work first: Box-Muller, new direction,
        // the sampler's logs; then the table walk
        R bs, bc, rad, mx, my, mz, L, tau_new, z1, z2;
        int gm;
        if constexpr (sizeof(R) == 4) {
            const DrawsF D = draws_f32(w0, w1);
            bs = D.bs;
            bc = D.bc;
            rad = D.rad;
            mx = D.mx;
            my = D.my;
            mz = D.mz;
            L = D.L;
            gm = D.gm;
            tau_new = D.tau;
            const float2 z = __fmul2_rn(make_float2(rad, rad), make_float2(bc, bs));
            z1 = z.x;
            z2 = z.y;
        } else {
            O::sc2pi(O::uni(w0.w[2]), &bs, &bc);
            rad = O::sq(fmax((R)0, -O::ln(O::uni(w0.w[1]))));
            iso_dir<R>(O::uni(w1.w[0]), O::uni(w1.w[1]), mx, my, mz);
            gm = us_bin<R>(O::uni(w0.w[0]), L);
            tau_new = fmax((R)0, -O::ln(O::uni(w0.w[3])));
            z1 = rad * bc;
            z2 = rad * bs;
        }
        const R us = us_sample<R>(xcom, L, gm, T);   // finite for any x; unused beyond 300
        const R upar = fabs(xcom) > (R)300 ? z2 : us;
        R gm1, sg;
        scatter_angle<R>(p.nx, p.ny, p.nz, mx, my, mz, gm1, sg);
        const R xout = scatter_x<R>(xcom, upar, gm1, z1, sg);
        set_dir(p, mx, my, mz);
        const R vdo = (F & F_VEL) ? vdot<R>(mx, my, mz, p.rec) : (R)0;
        p.x = xout + vdo;
        p.tau = tau_new;
        return true;
    }
    return cross_face<R, F>(A, p, alpha, sx_, axis, nd, st);
}

#include "transport_tail.cuh"

template <typename R, unsigned F>
constexpr size_t smem_bytes(int block, int tail_warps)
{
    const size_t stash = (size_t)stash_words<R, F>() * 4u * (size_t)block, tail = tail_bytes(block, tail_warps);
    return kStashOff + (sizeof(R) == 4 && tail > stash ? tail : stash);
}
// (the splits of an SM's 256 KB: ... 164, 196 or 228 KB of shared memory, of
// which each CTA takes 1 KB more than it asks for)
static_assert(2 * (smem_bytes<float, F_RICH | F_SEG>(256, kTailWarpsL1) + 1024) <= 196 * 1024,
              "two CTAs with an emissivity tally leave L1 60 KB");

// One model's walk by the whole CTA: stage the model's tables in shared
// memory, run packets until the model's id counter is exhausted and every
// lane has finished, then add the counters. Every thread of the CTA calls it.
//
// Bulk phase: each lane owns a packet; a warp refills its idle lanes with one
// atomic on the id counter (ballot + popc + shuffle). The first warp of the
// CTA that finds the counter exhausted raises a CTA flag, and every warp
// leaves the bulk phase at its next iteration.
//
// Tail phase (the remaining, typically longest packets): rounds of
// kTailRound events per lane; after each round the CTA counts its running
// packets and, if they occupy more warps than they would fill, moves them
// (through the shared-memory stash) to the lowest threads. Emptied warps
// then wait at the round barrier without issuing, so the surviving packets
// run in full warps instead of sharing the issue slots with idle lanes. The
// FP32 walk's last packets (tail_starts) go to groups of lanes, walk_tail,
// if most of them scatter at least twice per crossing: a group's chain ends at
// each crossing, and a walk of crossings (the optically thin fill, 12 of 13
// events) took 4 % longer with it.
//
// Line-profile mode PH (2: the slice; 1: the global 2-D table, with the
// sampler also read from global memory; 3: the core-wing blend) selects the
// profile and where the sampler's tables are read from.
template <typename R, unsigned F, int PH>
__device__ __forceinline__ void run_model(const TransportArgs& A, const RoundKeys& K, float* sm)
{
    int* ctl = reinterpret_cast<int*>(reinterpret_cast<char*>(sm) + kCtlOff);
    uint32_t* stash = reinterpret_cast<uint32_t*>(reinterpret_cast<char*>(sm) + kStashOff);
    unsigned char* sgw = reinterpret_cast<unsigned char*>(sm + kSmemFloats);
    if constexpr (PH == 2) {
        for (int i = threadIdx.x; i < kVoigtN; i += blockDim.x) sm[kSmemVoigt + i] = A.voigt_lnH[i];
    }
    if constexpr (PH == 2 || PH == 3) {
        for (int i = threadIdx.x; i < kUsNx; i += blockDim.x) sm[kSmemUsX + i] = A.us_x[i];
        for (int i = threadIdx.x; i < kUsNx * kUsNu; i += blockDim.x) sm[kSmemUsC + i] = A.us_lncdf[i];
    }
    if constexpr (PH != 1) {
        for (int i = threadIdx.x; i < kUsNx * kGuideN; i += blockDim.x) sgw[i] = A.us_guide[i];
    }
    if (threadIdx.x == 0) ctl[0] = 0;
    unsigned long long* segw = reinterpret_cast<unsigned long long*>(ctl + 4 + 2 * 32) + (threadIdx.x >> 5);
    if ((threadIdx.x & 31u) == 0u) *segw = 0ull;
    __syncthreads();
    Tabs T;
    T.sv = sm + kSmemVoigt;
    T.sx = PH == 1 ? A.us_x : sm + kSmemUsX;
    T.sc = PH == 1 ? A.us_lncdf : sm + kSmemUsC;
#ifdef KRL_TABLES_IN_CONSTANT
    if constexpr (PH == 4) {
        T.sv = c_voigt;
        T.sx = c_usx;
        T.sc = c_uslncdf;
    }
#endif
    T.sg = PH == 1 ? A.us_guide : sgw;
    // the sampler's row guide, from the staged nodes (all profile modes)
    unsigned char* rgw = reinterpret_cast<unsigned char*>(sm) + kSmemRowGuide;
    float4* rbw = reinterpret_cast<float4*>(reinterpret_cast<char*>(sm) + kSmemRowBins);
    float2* rxw = reinterpret_cast<float2*>(rbw + 2 * kRowGuideN);
    auto rrow = [&](int i) { return make_float2(T.sx[i], Ops<float>::rcp(T.sx[i + 1] - T.sx[i])); };
    for (int t = threadIdx.x; t < kRowGuideN; t += blockDim.x) {
        const float edge = __uint_as_float((unsigned)(t + (int)kRowGuideBase) << 19);
        int i = 0;
        while (i < kUsNx - 2 && T.sx[i + 1] <= edge) ++i;
        if constexpr (sizeof(R) == 8) {
            rgw[t] = (unsigned char)i;
        } else {
            const float2 r0 = rrow(i), r1 = i < kUsNx - 2 ? rrow(i + 1) : r0;
            rbw[2 * t] = make_float4(i < kUsNx - 2 ? T.sx[i + 1] : INFINITY, __int_as_float(i), r0.x, r0.y);
            rbw[2 * t + 1] = make_float4(r1.x, r1.y, 0.0f, 0.0f);
        }
    }
    if constexpr (sizeof(R) == 4) {
        for (int i = threadIdx.x; i < kUsNx - 1; i += blockDim.x) rxw[i] = rrow(i);
    }
    __syncthreads();
    T.rg = rgw;
    T.rb = rbw;
    T.rx = rxw;
    T.segw = segw;

    const R a = (R)A.a;
    const R H0 = (R)__ldg(A.H0);
    const unsigned lane = threadIdx.x & 31u;
    const int warp = (int)(threadIdx.x >> 5);
    const int nwarps = (int)(blockDim.x >> 5);
    Pkt<R> p;
    bool active = false;
    LaneStats st = {0u, 0u, 0u, 0u, 0u, 0u};

    // Both phases run in one loop so that the event code is inlined once.
    const int n = (int)blockDim.x;
    bool bulk = true;
    int round = 0, it = 0, quiet = 0;
    int refill = 1, taken = 0, iters = 0;   // idle lanes to wait for; ids taken; bulk iterations
    for (;;) {
        // ---- bulk phase: refill idle lanes, leave when the ids run out. A
        // warp whose lanes are all busy skips this bookkeeping, except every
        // kBulkCheck-th iteration, when it looks at the CTA's stop flag (the
        // other warps may be waiting for it at the tail barrier).
        ++iters;
        const unsigned idle = bulk ? __ballot_sync(kFull, !active) : 0u;
        if (bulk && (idle != 0u || ++quiet == kBulkCheck)) {
            quiet = 0;
            const int nidle = __popc(idle);
            // lane 0 reads the flag and broadcasts it: every lane of the warp
            // must take the same decision (the leave path has a CTA barrier),
            // and lanes that read it themselves could see it before and after
            // another warp's write
            int stop = 0;
            if (lane == 0) stop = *reinterpret_cast<volatile int*>(ctl);
            bool leave = __shfl_sync(kFull, stop, 0) != 0;
            if (!leave && (nidle == 32 || (nidle > 0 && nidle >= (A.refill_min > 0 ? A.refill_min : refill)))) {
                unsigned long long base = 0, top = A.n;
                if (A.even_fill) {
                    // no more packets than lanes: every CTA takes an equal
                    // share of the ids and every warp an equal share of the
                    // CTA's, so that the longest packets meet little company
                    const unsigned long long b0 = A.n * blockIdx.x / gridDim.x, b1 = A.n * (blockIdx.x + 1ull) / gridDim.x;
                    base = b0 + (b1 - b0) * (unsigned)warp / (unsigned)nwarps;
                    top = b0 + (b1 - b0) * (unsigned)(warp + 1) / (unsigned)nwarps;
                    leave = true;
                } else {
                    if (lane == 0) base = atomicAdd(A.next, (unsigned long long)nidle);
                    base = __shfl_sync(kFull, base, 0);
                    leave = base + (unsigned long long)nidle >= A.n;
                    if (leave && lane == 0) *reinterpret_cast<volatile int*>(ctl) = 1;
                }
                // The emission runs for the idle lanes alone and costs about as
                // much as four events of the whole warp: with lambda lanes
                // ending per iteration, waiting for m idle lanes costs m / 2
                // lanes and saves all but 1 / m of the emissions' time, best
                // near m = sqrt(64 x 4 lambda). 1 for long walks.
                taken += nidle;
                if (iters >= 32) {
                    const int m = (int)sqrtf(256.0f * (float)(taken - 32) / (float)iters);
                    refill = m < 1 ? 1 : (m > 16 ? 16 : m);
                }
                if (!active) {
                    const unsigned long long k = base + __popc(idle & ((1u << lane) - 1u));
                    if (k < top) {
                        p.id = A.first + k;
                        if (emit<R, F>(A, K, p)) {
                            active = true;
                        } else {
                            spectrum_add(A, p.x, (R)1);
                            ++st.esc;
                            write_record(A, p, 1);
                        }
                    }
                }
            }
            if (leave) {                      // warp-uniform; once per warp
                bulk = false;
                __syncthreads();
            }
        } else if (!bulk && (it >= kTailRound || !__any_sync(kFull, active))) {
            // ---- tail phase, end of a round: count and compact
            const unsigned m = __ballot_sync(kFull, active);
            int* cnt = ctl + 4 + 32 * (round & 1);
            const unsigned ms = __ballot_sync(kFull, active && p.nscat >= 2u * p.ncross);
            if (lane == 0) cnt[warp] = __popc(m) | __popc(ms) << 16;
            __syncthreads();
            int total = 0, before = 0, busy = 0, scatters = 0;
            for (int w = 0; w < nwarps; ++w) {
                const int c = cnt[w] & 0xffff;
                scatters += cnt[w] >> 16;
                total += c;
                before += w < warp ? c : 0;
                busy += c > 0 ? 1 : 0;
            }
            if (total == 0) break;            // CTA-uniform
            if constexpr (sizeof(R) == 4 && (PH == 2 || PH == 4)) {
                const int tw = nwarps < A.tail_warps ? nwarps : A.tail_warps;
                if (tail_starts(total, tw) && 2 * scatters > total) {     // CTA-uniform
                    // the last packets, dealt over tw warps: group g of warp
                    // w walks packet g tw + w
                    if (active) {
                        flush_visit<R, F>(A, p);
                        stash_put<R, F>(stash, n, before + __popc(m & ((1u << lane) - 1u)), p);
                    }
                    __syncthreads();
                    const int G = total <= tw * kTailWide ? 32 / kTailWide : 16 / kTailWide;
                    const int q = (int)lane / G * tw + warp;
                    active = warp < tw && q < total;
                    if (active) stash_get<R, F>(A, stash, n, q, p);
                    else if (warp < tw) stash_get<R, F>(A, stash, n, 0, p);      // a state to compute on, not walked
                    __syncthreads();                  // the buffers take the stash's place
                    if (warp < tw) {
                        walk_tail<F, PH>(A, K, p, active, G, reinterpret_cast<TailBuf*>(stash) + warp, T, a, H0, st);
                    }
                    break;
                }
            }
            if (busy > (total + 31) / 32) {   // CTA-uniform
                if (active) {
                    flush_visit<R, F>(A, p);
                    stash_put<R, F>(stash, n, before + __popc(m & ((1u << lane) - 1u)), p);
                }
                __syncthreads();
                // the stash is next written after a later round's count
                // barrier, which every thread reaches only after this read
                active = (int)threadIdx.x < total;
                if (active) stash_get<R, F>(A, stash, n, (int)threadIdx.x, p);
            }
            ++round;
            it = 0;
        }
        if (!bulk) ++it;
        if (active) active = advance<R, F, PH>(A, K, p, T, a, H0, st);
    }

    if constexpr (sizeof(R) == 4 && (F & F_SEG) != 0) {
        // the rest of the warp's last chunk of segment records
        if (A.seg && A.seg_chunk) {
            __syncwarp();
            const unsigned long long i = *segw;
            const unsigned left = (unsigned)(0ull - i) & (A.seg_chunk - 1u);
            for (unsigned k = lane; k < left; k += 32u) clear_segments(A, i + k, 1u);
        }
    }
    using u64 = unsigned long long;
    const u64 ended = (u64)st.esc + st.des + st.stuck + st.absorbed;
    const u64 tot[7] = {warp_sum(ended),        warp_sum((u64)st.esc),   warp_sum((u64)st.des),     warp_sum((u64)st.stuck),
                        warp_sum((u64)st.scat), warp_sum((u64)st.cross), warp_sum((u64)st.absorbed)};
    if (lane == 0) {
#pragma unroll
        for (int k = 0; k < 7; ++k)
            if (tot[k]) atomicAdd(A.stats + k, tot[k]);
    }
}

template <typename R, unsigned F, int PH>
__global__ void __launch_bounds__(max_block<R, F>(), 2) k_transport(const __grid_constant__ TransportArgs A)
{
    extern __shared__ float sm[];
    run_model<R, F, PH>(A, A.keys, sm);
}

// The lowest-numbered model that still has unassigned packet ids, or -1.
// The shared cursor only moves forward, so the loop ends within n_models
// steps.
__device__ int next_model(const BatchArgs& B)
{
    int m = atomicAdd(B.cursor, 0);
    while (m < B.n_models) {
        const unsigned long long used = atomicAdd(B.models[m].next, 0ull);
        if (used < B.models[m].n) return m;
        atomicCAS(B.cursor, m, m + 1);
        const int m2 = atomicAdd(B.cursor, 0);
        m = m2 > m ? m2 : m + 1;
    }
    return -1;
}

// Many independent models (grids) in one persistent launch: each CTA takes
// the lowest model that still has packets, stages that model's tables,
// runs its warps on it until its ids run out, drains, and takes the next.
// CTAs finish models at different times, so one model's tail overlaps the
// next model's bulk instead of idling the device as separate launches do.
// The batched launch runs 256-thread CTAs (smaller CTAs move on to the next
// model sooner; the autotuner found them faster on uneven model sets).
constexpr int kBatchBlock = 256;

template <typename R, unsigned F>
__global__ void __launch_bounds__(kBatchBlock, 2) k_transport_batch(const __grid_constant__ BatchArgs B)
{
    extern __shared__ float sm[];
    __shared__ TransportArgs sA;
    __shared__ int s_model;
    for (;;) {
        if (threadIdx.x == 0) s_model = next_model(B);
        __syncthreads();
        const int m = s_model;
        if (m < 0) break;
        {
            const int* src = reinterpret_cast<const int*>(B.models + m);
            int* dst = reinterpret_cast<int*>(&sA);
            for (int i = threadIdx.x; i < (int)(sizeof(TransportArgs) / sizeof(int)); i += blockDim.x) dst[i] = src[i];
        }
        __syncthreads();
        run_model<R, F, 2>(sA, B.keys, sm);
        __syncthreads();     // every warp done before the tables are replaced
    }
}

template <typename R, unsigned F, int PH>
cudaError_t launch_one(const TransportArgs& A, int grid, int block, cudaStream_t s)
{
    if (block > max_block<R, F>()) return cudaErrorInvalidConfiguration;
    auto kern = k_transport<R, F, PH>;
    // the shared-memory opt-in is an attribute of the kernel on the current
    // device: set it on every launch (a host-side call of about a
    // microsecond), so that a launch on any device of the process has it
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem_bytes<R, F>(max_block<R, F>(), kTailWarps));
    if (e != cudaSuccess) return e;
    kern<<<grid, block, smem_bytes<R, F>(block, A.tail_warps), s>>>(A);
    return cudaGetLastError();
}

template <typename R, unsigned F>
cudaError_t launch_batch_one(const BatchArgs& B, int grid, int block, cudaStream_t s)
{
    if (block > kBatchBlock) return cudaErrorInvalidConfiguration;
    auto kern = k_transport_batch<R, F>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)smem_bytes<R, F>(kBatchBlock, kTailWarps));   // per device: every launch
    if (e != cudaSuccess) return e;
    kern<<<grid, block, smem_bytes<R, F>(block, B.tail_warps), s>>>(B);
    return cudaGetLastError();
}

template <typename R, unsigned F, int PH>
int occupancy_one(int block)
{
    if (block > max_block<R, F>()) return 0;
    auto kern = k_transport<R, F, PH>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<R, F>(max_block<R, F>(), kTailWarps));
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, smem_bytes<R, F>(block, kTailWarps)) != cudaSuccess) return 0;
    return n;
}

template <typename R, unsigned F>
int batch_occupancy_one(int block)
{
    if (block > kBatchBlock) return 0;
    auto kern = k_transport_batch<R, F>;
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<R, F>(kBatchBlock, kTailWarps));
    int n = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&n, kern, block, smem_bytes<R, F>(block, kTailWarps)) != cudaSuccess) return 0;
    return n;
}

// Calls fn with the instantiation of the features f. The narrow lean walk and
// the rich walk without per-segment tallies have instantiations of their own
// in the FP32 production walk only (SPLIT).
template <bool SPLIT, typename Fn>
auto with_features(unsigned f, Fn fn)
{
    using std::integral_constant;
    constexpr unsigned W = F_WIDE, L = F_RICH, S = F_RICH | F_SEG;
    if constexpr (SPLIT) {
        switch (f & (F_RICH | F_SEG | F_WIDE | 3u)) {
        case 0: return fn(integral_constant<unsigned, 0u>());
        case 1: return fn(integral_constant<unsigned, 1u>());
        case 2: return fn(integral_constant<unsigned, 2u>());
        case 3: return fn(integral_constant<unsigned, 3u>());
        case L: return fn(integral_constant<unsigned, L>());
        case L | 1u: return fn(integral_constant<unsigned, L | 1u>());
        case L | 2u: return fn(integral_constant<unsigned, L | 2u>());
        case L | 3u: return fn(integral_constant<unsigned, L | 3u>());
        case L | W: return fn(integral_constant<unsigned, L | W>());
        case L | W | 1u: return fn(integral_constant<unsigned, L | W | 1u>());
        case L | W | 2u: return fn(integral_constant<unsigned, L | W | 2u>());
        case L | W | 3u: return fn(integral_constant<unsigned, L | W | 3u>());
        default: break;
        }
    }
    switch (f & 7u) {
    case 0: return fn(integral_constant<unsigned, W>());
    case 1: return fn(integral_constant<unsigned, W | 1u>());
    case 2: return fn(integral_constant<unsigned, W | 2u>());
    case 3: return fn(integral_constant<unsigned, W | 3u>());
    case 4: return fn(integral_constant<unsigned, S>());
    case 5: return fn(integral_constant<unsigned, S | 1u>());
    case 6: return fn(integral_constant<unsigned, S | 2u>());
    default: return fn(integral_constant<unsigned, S | 3u>());
    }
}

template <typename R, int PH>
constexpr bool split() { return sizeof(R) == 4 && PH == 2; }

template <typename R, int PH>
cudaError_t dispatch(const TransportArgs& A, unsigned f, int grid, int block, cudaStream_t s)
{
    return with_features<split<R, PH>()>(f, [&](auto F) { return launch_one<R, decltype(F)::value, PH>(A, grid, block, s); });
}

template <typename R, int PH>
int occ_dispatch(unsigned f, int block)
{
    return with_features<split<R, PH>()>(f, [&](auto F) { return occupancy_one<R, decltype(F)::value, PH>(block); });
}

template <typename R>
cudaError_t dispatch_batch(const BatchArgs& B, unsigned f, int grid, int block, cudaStream_t s)
{
    return with_features<false>(f, [&](auto F) { return launch_batch_one<R, decltype(F)::value>(B, grid, block, s); });
}

template <typename R>
int batch_occ_dispatch(unsigned f, int block)
{
    return with_features<false>(f, [&](auto F) { return batch_occupancy_one<R, decltype(F)::value>(block); });
}

}  // namespace
}  // namespace krl
