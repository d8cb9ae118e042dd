// Device-side building blocks of libxs: physical constants, the Faddeeva
// function w(z) = exp(-z^2) erfc(-iz) by tiers (Sec. 2.1.1), and small helpers.
//
// Faddeeva tiers.  H = Re w is needed to a relative accuracy of ~1e-7 (FP32) or
// ~1e-15 (FP64) everywhere, including the Gaussian-to-Lorentzian transition at
// small a where Re w is far smaller than |w|.  Each tier keeps the real part free
// of cancellation:
//   * |z| large: the asymptotic series of Eq. asywofz,
//       w ~ i/(sqrt(pi) z) * (1 + sum_{k>=1} (2k-1)!! (1/(2 z^2))^k),
//     truncated at K terms chosen per |z| band (bands measured against an
//     arbitrary-precision reference); with z = x + ia and 1/z = (x - ia)/|z|^2
//     the real part is (a Re p - x Im p)/(sqrt(pi)|z|^2) with both terms of one
//     sign, so it keeps its relative accuracy as a -> 0.
//   * |z| small: the exponentially convergent series behind Eq. algo916 /
//     algo916L (Zaghloul & Ali 2011).  Written with E_n^-+ = exp(-(nh -+ x)^2):
//       Re w = e^{-x^2} [K(a) cos 2ax + (2h/pi) sin(ax) sin(ax)/a] + (a h/pi) Sc
//       Im w = e^{-x^2} [-K(a) sin 2ax + (h/pi) sin(2ax)/a]       + (h/pi) Ss
//       Sc = sum_n (E_n^- + E_n^+)/(n^2h^2 + a^2),  Ss = sum_n nh (E_n^- - E_n^+)/(n^2h^2 + a^2)
//       K(a) = erfcx(a) - (2ah/pi) sum_n e^{-n^2h^2}/(n^2h^2 + a^2)   (per line, precomputed)
//     Every E_n is a product of factors with small exponents about the term nearest
//     the peak (nothing passes through e^{-x^2} e^{2nhx}, which would lose digits).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace xsd {

// CODATA 2018 (cgs) and the second radiation constant c2 as printed in Sec. 2.2.
constexpr double kB = 1.380649e-16;
constexpr double hP = 6.62607015e-27;
constexpr double cL = 2.99792458e10;
constexpr double amu = 1.66053906660e-24;
constexpr double c2 = 1.4387773;
constexpr double Tref = 296.0;
constexpr double bar_per_atm = 1.01325;
constexpr double PI = 3.14159265358979323846;
constexpr double SQRTPI = 1.77245385090551602730;
constexpr double INV_SQRTPI = 0.56418958354775628695;
constexpr double SQRT2 = 1.41421356237309504880;

// Scale applied to line strengths in the FP32 path so that partial sums of the
// cross-section (1e-35 .. 1e-12 cm^2) sit well inside the normal float range.
constexpr int MIXED_SCALE_LOG2 = 80;
constexpr double MIXED_SCALE = 1208925819614629174706176.0; // 2^80
constexpr double MIXED_UNSCALE = 8.27180612553027674871e-25; // 2^-80

// cos x at compile time, 0 <= x <= pi/2 (Taylor series)
constexpr double cos_quadrant(double x)
{
    double s = 0.0;
    for (int k = 14; k >= 1; --k) s = -(1.0 + s) * x * x / ((2.0 * k - 1.0) * (2.0 * k));
    return 1.0 + s;
}

// Chebyshev nodes t_m = cos((2m + 1) pi/(2n)) and T_k(t_m) = cos(k (2m + 1) pi/(2n)),
// built at compile time.
template <int n>
struct ChebTable {
    double T[n][n]; // [k][m]; T[1] are the nodes
};
template <int n>
constexpr ChebTable<n> make_cheb()
{
    ChebTable<n> c{};
    for (int k = 0; k < n; ++k)
        for (int m = 0; m < n; ++m) {
            int j = (k * (2 * m + 1)) % (4 * n); // angle j pi/(2n), one period
            double s = 1.0;
            if (j > 2 * n) j = 4 * n - j;
            if (j > n) {
                j = 2 * n - j;
                s = -1.0;
            }
            c.T[k][m] = (j == n) ? 0.0 : s * cos_quadrant(PI * j / (2.0 * n));
        }
    return c;
}

template <class R> struct vec4;
template <> struct vec4<float> { using type = float4; };
template <> struct vec4<double> { using type = double4_32a; };

// Per-precision Faddeeva tier table.
template <class R> struct Tier;
template <> struct Tier<float> {
    // The FP32 path evaluates w only through the wing forms (|z| >= 16.5), the
    // polynomial in 1/|z|^2 (6 <= |z| < 16.5) and the series below |z| = 6
    // (series_sums); these are the series' parameters.
    static constexpr float z2_series = 64.0f;  // K(a) is precomputed for lines with a^2 below this
    static constexpr float h = 0.7f;           // series step (error ~1e-8 relative)
};
template <> struct Tier<double> {
    static constexpr double z2_far = 22500.0;  // |z| >= 150: K = 3
    static constexpr double z2_k4 = 4900.0;    // |z| >= 70 : K = 4
    static constexpr double z2_mid = 1600.0;   // |z| >= 40 : K = 5
    static constexpr double z2_k7 = 441.0;     // |z| >= 21 : K = 7
    static constexpr double z2_series = 100.0; // |z| >= 10 : K = 12, below: series
    // Below this a leaf's nearest |z|^2 to a line has the line's series data staged: it and a
    // point's own |z|^2 round differently (by up to 1e-9 at an ulp of nu).
    static constexpr double z2_stage = z2_series * (1.0 + 1e-6);
    static constexpr double h = 0.5;           // series step (error ~1e-17)
};

// Bounds-checked build (nvcc -DXS_CHECKED): index checks guard the kernels'
// global and shared accesses.  A failed check records its source line in this
// translation unit's device status word (the largest line wins) and the access is
// skipped, so a bad index never faults or traps; xs_check_status reads the words.
// In the normal build XS_CHECK(c) is the constant true and costs nothing.
#ifdef XS_CHECKED
static __device__ int g_xs_check_line = 0;
__device__ __forceinline__ bool xs_check(bool ok, int line)
{
    if (!ok) atomicMax(&g_xs_check_line, line);
    return ok;
}
#define XS_CHECK(c) ::xsd::xs_check((c), __LINE__)
// host accessor of this translation unit's word (read, then cleared if asked)
#define XS_CHECK_ACCESSOR(name)                                                                      \
    namespace xsi {                                                                                  \
    int check_status_##name(int clear)                                                               \
    {                                                                                                \
        int v = 0;                                                                                   \
        if (cudaMemcpyFromSymbol(&v, ::xsd::g_xs_check_line, sizeof(int)) != cudaSuccess) return -1; \
        if (clear) {                                                                                 \
            const int z = 0;                                                                         \
            if (cudaMemcpyToSymbol(::xsd::g_xs_check_line, &z, sizeof(int)) != cudaSuccess) return -1; \
        }                                                                                            \
        return v;                                                                                    \
    }                                                                                                \
    }
#else
#define XS_CHECK(c) true
#define XS_CHECK_ACCESSOR(name)                 \
    namespace xsi {                             \
    int check_status_##name(int) { return 0; } \
    }
#endif

__device__ __forceinline__ float rcp_fast(float x)
{
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// x = |d| c with d = dh + dl and c = ch + cl as unevaluated float pairs:
// returns x as a pair (xh, xl), xh = fl(|dh| ch).
__device__ __forceinline__ void scaled_pair(float dh, float dl, float ch, float cl, float* xh, float* xl)
{
    // renormalise d = dh + dl first (Fast2Sum, |dl| << |dh| or both tiny) so that
    // xh, which the asymptotic tiers use alone, carries all of d's leading bits
    const float d = dh + dl;
    const float e = (dh - d) + dl;
    const float p = d * ch;
    const float r = fmaf(d, ch, -p) + fmaf(d, cl, e * ch);
    *xh = fabsf(p);
    *xl = __int_as_float(__float_as_int(r) ^ (__float_as_int(d) & 0x80000000)); // r with d's sign taken out
}
__device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }

// e^v in FP64, table-driven (Tang 1989): 2^(i/64) as hi + lo from a table, the rest
// (|r| <= ln2/128) by the series to r^5 (next term 4e-17): 12 operations, within 0.52 ulp
// of the exact value.  Beyond +-700 exp.
struct Exp2Entry {
    double hi, lo;
};
__device__ const Exp2Entry EXP2_64[64] = {
    {1.0, 0.0}, {1.0108892860517005, -1.5234778603368577e-17},
    {1.0218971486541166, 5.109225028973444e-17}, {1.0330248790212284, 7.600838874027088e-18},
    {1.0442737824274138, 8.551889705537965e-17}, {1.0556451783605572, 1.759325738772092e-18},
    {1.0671404006768237, -7.899853966841582e-17}, {1.0787607977571199, -6.656660436056593e-17},
    {1.0905077326652577, -3.046782079812471e-17}, {1.102382583307841, 5.2660368715706944e-17},
    {1.1143867425958924, 1.0410278456845571e-16}, {1.1265216186082418, 5.165856758795457e-17},
    {1.1387886347566916, 8.912812676025408e-17}, {1.1511892299529827, 3.250710218863827e-17},
    {1.1637248587775775, 3.8292048369240935e-17}, {1.1763969916502812, 5.554203254218079e-17},
    {1.189207115002721, 3.982015231465646e-17}, {1.202156731452703, 6.644981499252301e-17},
    {1.215247359980469, -7.712630692681488e-17}, {1.22848053610687, -1.89878163130253e-17},
    {1.241857812073484, 4.658027591836937e-17}, {1.255380757024691, -6.7113898212968784e-18},
    {1.2690509571917332, 2.667932131342186e-18}, {1.2828700160787783, 1.713594918243561e-17},
    {1.2968395546510096, 2.5382502794888315e-17}, {1.3109612115247644, -7.181536135519454e-17},
    {1.3252366431597413, -2.8587312100388614e-17}, {1.339667524053303, 8.927282594831732e-17},
    {1.3542555469368927, 7.70094837980299e-17}, {1.3690024229745905, 9.593797919118849e-17},
    {1.383909881963832, -6.770511658794786e-17}, {1.3989796725383112, -9.614213209051323e-17},
    {1.4142135623730951, -9.667293313452913e-17}, {1.42961333839197, -1.2031642489053655e-17},
    {1.4451808069770467, -3.0237581349939873e-17}, {1.460917794180647, -5.600377186075216e-17},
    {1.4768261459394993, -3.483994556892796e-17}, {1.4929077282912648, 1.4192920154284036e-17},
    {1.5091644275934228, -1.016455327754295e-16}, {1.5255981507445384, -1.1024941712342561e-16},
    {1.5422108254079407, 7.949834809697621e-17}, {1.559004400237837, 3.7812070533575275e-17},
    {1.5759808451078865, -1.0136916471278304e-17}, {1.593142151342267, -1.0094406542311964e-16},
    {1.6104903319492543, 2.4707192569797888e-17}, {1.6280274218573478, -6.712955084707084e-17},
    {1.645755478153965, -1.0125679913674773e-16}, {1.6636765803267364, 5.8909926967131e-17},
    {1.681792830507429, 8.199010020581497e-17}, {1.7001063537185235, -8.0237193703977e-18},
    {1.718619298122478, -1.851380418263111e-17}, {1.7373338352737062, 3.164389299292957e-17},
    {1.7562521603732995, 2.960140695448873e-17}, {1.7753764925265212, 6.429731796556572e-17},
    {1.7947090750031072, 1.8227458427912087e-17}, {1.8142521755003989, -9.969531538920349e-17},
    {1.8340080864093424, 3.283107224245627e-17}, {1.8539791250833855, 9.761887490727594e-17},
    {1.8741676341103, -6.122763413004143e-17}, {1.8945759815869656, 3.4034035352165297e-17},
    {1.9152065613971474, -1.0619946056195963e-16}, {1.9360617934922943, 1.0332385960676326e-16},
    {1.9571441241754002, 8.960767791036668e-17}, {1.978456026387951, 4.0388753109278167e-17}};

__device__ __forceinline__ double exp_tab(double v)
{
    if ((__double2hiint(v) & 0x7fffffff) >= 0x4085e000) return exp(v); // |v| >= 700, infinities, NaN
    const double magic = 6755399441055744.0; // 1.5 2^52
    // ln 2 = its float value (products with k are exact) + the rest
    const double ln2_hi = (double)0.693147182f, ln2_lo = -0.000000001904654299957767878541823;
    const double t = fma(v, 64.0 / 0.69314718055994530942, magic), kd = t - magic;
    const int k = __double2loint(t);
    const double r = fma(kd, -ln2_lo / 64, fma(kd, -ln2_hi / 64, v));
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(r, p, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    p = fma(r * r, p, r);
    const Exp2Entry h = EXP2_64[k & 63];
    const double s = h.hi + fma(h.hi, p, h.lo);
    return __hiloint2double(__double2hiint(s) + ((k >> 6) << 20), __double2loint(s));
}

// 1/x in FP64 to about an ulp, x normal: the hardware's approximation and two steps of
// Newton's iteration, five operations
__device__ __forceinline__ double rcp64(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    y = fma(y, fma(-x, y, 1.0), y);
    return fma(y, fma(-x, y, 1.0), y);
}

// the same for any x: 0, infinities and what overflows as a division gives them
__device__ __forceinline__ double rcp64_any(double x)
{
    const int e = __double2hiint(x) & 0x7ff00000;
    return (e < 0x00200000 || e >= 0x7fd00000) ? 1.0 / x : rcp64(x);
}

// exp(-x^2) with x^2 split into hi + lo so the rounding of x*x does not enter.
__device__ __forceinline__ float exp_negsq(float x, float xl) // x + xl, |xl| << |x|
{
    float hi = x * x;
    float lo = fmaf(2.0f * x, xl, fmaf(x, x, -hi));
    return fmaf(expf(-hi), -lo, expf(-hi));
}
__device__ __forceinline__ double exp_negsq(double x)
{
    double hi = x * x;
    double lo = fma(x, x, -hi);
    const double e = exp_tab(-hi);
    return fma(e, -lo, e);
}

// Per-line table for series_sums: d[n + SER_OFF] = 1/(n^2 h^2 + a^2) for n != 0 and 0
// for n = 0, n = -SER_OFF .. SER_TAB - 1 - SER_OFF.  The odd row length keeps the lanes
// that fill 32 rows on different banks.
constexpr int SER_OFF = 6;   // terms on each side of the peak
constexpr int SER_N0 = 16;   // largest peak index: x <= SER_X
constexpr int SER_TAB = SER_N0 + 2 * SER_OFF + 1; // 29
constexpr float SER_X = 11.5f;

__device__ __forceinline__ void series_table(float a, float* d)
{
    const float h = Tier<float>::h;
    const float a2 = a * a;
    d[SER_OFF] = 0.0f;
#pragma unroll 4
    for (int n = 1; n < SER_TAB - SER_OFF; ++n) {
        const float nh = (float)n * h;
        const float v = rcp_fast(fmaf(nh, nh, a2));
        d[SER_OFF + n] = v;
        if (n <= SER_OFF) d[SER_OFF - n] = v;
    }
}

__device__ __forceinline__ float exp2_fast(float x)
{
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// sin v and, if want_c, cos v, both up to the sign (-1)^k of the multiple of pi taken out:
// Taylor series on |r| <= pi/2 (next terms below 7e-10)
__device__ __forceinline__ void sin_cos_mod_pi(float v, bool want_c, float* s, float* c)
{
    constexpr float MAGIC = 12582912.0f;
    const float k = fmaf(v, (float)(1.0 / PI), MAGIC) - MAGIC;
    const float r = fmaf(-k, (float)(PI - (double)(float)PI), fmaf(-k, (float)PI, v));
    const float t = r * r;
    float p = 1.0f / 6227020800.0f;
    p = fmaf(p, t, -1.0f / 39916800.0f);
    p = fmaf(p, t, 1.0f / 362880.0f);
    p = fmaf(p, t, -1.0f / 5040.0f);
    p = fmaf(p, t, 1.0f / 120.0f);
    p = fmaf(p, t, -1.0f / 6.0f);
    *s = fmaf(p * t, r, r);
    if (want_c) {
        float q = -1.0f / 87178291200.0f;
        q = fmaf(q, t, 1.0f / 479001600.0f);
        q = fmaf(q, t, -1.0f / 3628800.0f);
        q = fmaf(q, t, 1.0f / 40320.0f);
        q = fmaf(q, t, -1.0f / 720.0f);
        q = fmaf(q, t, 1.0f / 24.0f);
        q = fmaf(q, t, -0.5f);
        *c = fmaf(q, t, 1.0f);
    }
}

// FP32 small-|z| series, 0 <= x <= SER_X, written as one sum over all integers n != 0 of
// exp(-(nh - x)^2) d_|n| (the E_n^+ of the head of this file are its negative n).  From
// the term nearest the peak, n0 = round(x/h), where n0 h - x = delta is small,
//   exp(-((n0 +- k)h - x)^2) = e^{-delta^2} Q_k e^{-+2kh delta},  Q_k = e^{-(kh)^2},
// so each side is a polynomial in e^{-+2h delta}: no digits are lost to e^{-x^2} e^{2nhx}.
// Terms with |k| > 6 are below 1e-9 of the peak term.  The two sides go as packed pairs,
// with the line's table d (series_table).  sin and cos of ax enter as sin^2 and sin cos
// only, so ax is reduced modulo pi and its sign dropped.  inv_a = 1/a.  Issue-bound:
// about 100 instructions a pair of line and point with its loop.
//
// Derivatives (DERIV): w' = -2 z w + 2i/sqrt(pi) loses 2|z|^2 of its accuracy when it is
// taken from w.  With 1/sqrt(pi) = (h/pi) sum_n E_n the sums cancel term by term instead:
//   Re w' = -2 Re(z g) + (2 a h/pi) S1,   Im w' = -2 Im(z g) + (2h/pi)(e^{-x^2} + x S1 + S2),
//   S_i = sum_{n != 0} E_n d_n (nh - x)^i,
// g the part of w with e^{-x^2}; S1 and S2 come from the first and second derivatives of
// the Horner polynomials.
struct SeriesSums {
    float s0, s1, s2;
};

template <bool DERIV>
__device__ __forceinline__ SeriesSums series_sums(float xh, float xl, const float* dt)
{
    const float h = Tier<float>::h;
    constexpr float L2E = 1.44269504f, MAGIC = 12582912.0f; // 1.5 2^23: rounds to an integer
    const float tm = fmaf(xh, 1.0f / h, MAGIC);
    const float n0f = tm - MAGIC;
    const int n0 = __float_as_int(tm) & 31;
    if (!XS_CHECK(n0 <= SER_N0)) return {0.0f, 0.0f, 0.0f};
    const float delta = (n0f * h - xh) - xl;
    const float E0 = exp2_fast(-L2E * delta * delta);
    const float u = 2.0f * h * L2E * delta;
    const float2 f = make_float2(exp2_fast(-u), exp2_fast(u)); // e^{-2h delta}, e^{2h delta}
    const float* d0 = dt + (n0 + SER_OFF);
    const float Q[SER_OFF + 1] = {1.0f, 0.612626433f, 0.140858427f, 0.0121551799f, 0.00039366915f, 4.78511947e-06f,
                                  2.18295906e-08f};
    // p = sum_k w_k f^k and, for the factors k and k^2, p' and p''/2
    float2 p = __fmul2_rn(make_float2(d0[SER_OFF], d0[-SER_OFF]), make_float2(Q[SER_OFF], Q[SER_OFF]));
    float2 p1 = make_float2(0.0f, 0.0f), p2 = p1;
#pragma unroll
    for (int k = SER_OFF - 1; k >= 0; --k) {
        if (DERIV) {
            p2 = __ffma2_rn(p2, f, p1);
            p1 = __ffma2_rn(p1, f, p);
        }
        // the centre term, k = 0, belongs to the first of the pair
        const float2 w = k ? __fmul2_rn(make_float2(d0[k], d0[-k]), make_float2(Q[k], Q[k])) : make_float2(d0[0], 0.0f);
        p = __ffma2_rn(p, f, w);
    }
    SeriesSums r;
    const float s0 = p.x + p.y;
    r.s0 = E0 * s0;
    r.s1 = r.s2 = 0.0f;
    if (DERIV) {
        const float2 k1 = __fmul2_rn(p1, f);                                         // sum k w f^k
        const float2 k2 = __ffma2_rn(__fmul2_rn(p2, f), make_float2(2.0f * f.x, 2.0f * f.y), k1); // sum k^2 w f^k
        const float m1 = h * (k1.x - k1.y), m2 = h * h * (k2.x + k2.y); // sums of kh and (kh)^2, sides signed
        r.s1 = E0 * fmaf(delta, s0, m1);
        r.s2 = E0 * fmaf(delta, fmaf(delta, s0, 2.0f * m1), m2);
    }
    return r;
}

// Re w
__device__ __forceinline__ float w_series_re(float xh, float xl, float a, float inv_a, float Kc, const float* dt)
{
    const SeriesSums q = series_sums<false>(xh, xl, dt);
    const float ex = exp_negsq(xh, xl);
    float sax, cax;
    sin_cos_mod_pi(a * xh, false, &sax, &cax);
    const float c2v = fmaf(-2.0f * sax, sax, 1.0f); // cos 2ax
    const float hpi = Tier<float>::h * (float)(1.0 / PI);
    return ex * fmaf(2.0f * hpi * inv_a * sax, sax, Kc * c2v) + a * hpi * q.s0;
}

// Re w, Re w' and Im w'
__device__ __forceinline__ void w_series_deriv(float xh, float xl, float a, float inv_a, float Kc, const float* dt,
                                               float* wr, float* dr, float* di)
{
    const SeriesSums q = series_sums<true>(xh, xl, dt);
    const float x = xh, ex = exp_negsq(xh, xl);
    float sax, cax;
    sin_cos_mod_pi(a * x, true, &sax, &cax);
    const float c2v = fmaf(-2.0f * sax, sax, 1.0f), s2 = 2.0f * sax * cax;
    const float hpi = Tier<float>::h * (float)(1.0 / PI);
    const float s2_a = a > 0.0f ? s2 * inv_a : 2.0f * x;
    const float gr = ex * fmaf(2.0f * hpi * inv_a * sax, sax, Kc * c2v);
    const float gi = ex * fmaf(hpi, s2_a, -Kc * s2);
    const float ah = a * hpi;
    *wr = fmaf(ah, q.s0, gr);
    *dr = 2.0f * fmaf(ah, q.s1, a * gi - x * gr);
    *di = 2.0f * fmaf(hpi, ex + fmaf(x, q.s1, q.s2), -fmaf(x, gi, a * gr));
}

// The same in FP64, h = 1/2 and 13 terms on each side (the next are below 1e-19 of the
// peak): n0 = round(x/h) <= SER64_N0 for x <= 10.  (A loop of an exponential a term
// before, 27 and more of them; some 150 operations now, 220 with derivatives.)
constexpr int SER64_OFF = 13, SER64_N0 = 20, SER64_TAB = SER64_N0 + 2 * SER64_OFF + 1; // 47
// e^{-(k h)^2}, k = 1 .. 13
__device__ const double KC_E64[SER64_OFF] = {0.77880078307140488, 0.36787944117144233, 0.10539922456186433,
                                             0.018315638888734179, 0.0019304541362277093, 0.00012340980408667956,
                                             4.7851173921290088e-06, 1.1253517471925912e-07, 1.6052280551856116e-09,
                                             1.3887943864964021e-11, 7.2877240958196922e-14, 2.3195228302435691e-16,
                                             4.4777324417183015e-19};

__device__ __forceinline__ void series_table64(double a, double* d)
{
    const double a2 = a * a;
    d[SER64_OFF] = 0.0;
#pragma unroll 1
    for (int n = 1; n < SER64_TAB - SER64_OFF; ++n) {
        const double v = rcp64(fma(0.25 * n, (double)n, a2));
        d[SER64_OFF + n] = v;
        if (n <= SER64_OFF) d[SER64_OFF - n] = v;
    }
}

struct SeriesSums64 {
    double s0, s1, s2;
};
template <bool DERIV>
__device__ __forceinline__ SeriesSums64 series_sums64(double x, const double* dt)
{
    const int n0 = __double2int_rn(2.0 * x);
    if (!XS_CHECK(n0 >= 0 && n0 <= SER64_N0)) return {0.0, 0.0, 0.0};
    const double delta = 0.5 * n0 - x; // exact
    const double E0 = exp_tab(-delta * delta);
    const double f = exp_tab(-delta), g = rcp64(f); // e^{-2h delta}, e^{2h delta}
    const double* d0 = dt + (n0 + SER64_OFF);
    double p = KC_E64[SER64_OFF - 1] * d0[SER64_OFF], q = KC_E64[SER64_OFF - 1] * d0[-SER64_OFF];
    double p1 = 0.0, p2 = 0.0, q1 = 0.0, q2 = 0.0;
#pragma unroll
    for (int k = SER64_OFF - 1; k >= 0; --k) {
        if (DERIV) {
            p2 = fma(p2, f, p1);
            p1 = fma(p1, f, p);
            q2 = fma(q2, g, q1);
            q1 = fma(q1, g, q);
        }
        p = fma(p, f, k ? KC_E64[k ? k - 1 : 0] * d0[k] : d0[0]);
        q = k ? fma(q, g, KC_E64[k ? k - 1 : 0] * d0[-k]) : q * g; // the centre term belongs to the first
    }
    SeriesSums64 r;
    const double s0 = p + q;
    r.s0 = E0 * s0;
    r.s1 = r.s2 = 0.0;
    if (DERIV) {
        const double k1 = p1 * f, l1 = q1 * g;                          // sums of k w f^k
        const double k2 = fma(p2 * f, 2.0 * f, k1), l2 = fma(q2 * g, 2.0 * g, l1); // of k^2 w f^k
        const double m1 = 0.5 * (k1 - l1), m2 = 0.25 * (k2 + l2);
        r.s1 = E0 * fma(delta, s0, m1);
        r.s2 = E0 * fma(delta, fma(delta, s0, 2.0 * m1), m2);
    }
    return r;
}

__device__ __forceinline__ double w_series_re(double x, double a, double inv_a, double Kc, const double* dt)
{
    const SeriesSums64 q = series_sums64<false>(x, dt);
    const double sax = sin(a * x);
    const double hpi = 0.5 / PI;
    return exp_negsq(x) * fma(2.0 * hpi * inv_a * sax, sax, Kc * fma(-2.0 * sax, sax, 1.0)) + a * hpi * q.s0;
}

__device__ __forceinline__ void w_series_deriv(double x, double a, double inv_a, double Kc, const double* dt, double* wr,
                                               double* dr, double* di)
{
    const SeriesSums64 q = series_sums64<true>(x, dt);
    double sax, cax;
    sincos(a * x, &sax, &cax);
    const double ex = exp_negsq(x), hpi = 0.5 / PI;
    const double c2v = fma(-2.0 * sax, sax, 1.0), s2 = 2.0 * sax * cax;
    const double s2_a = a > 0.0 ? s2 * inv_a : 2.0 * x;
    const double gr = ex * fma(2.0 * hpi * inv_a * sax, sax, Kc * c2v);
    const double gi = ex * fma(hpi, s2_a, -Kc * s2);
    const double ah = a * hpi;
    *wr = fma(ah, q.s0, gr);
    *dr = 2.0 * fma(ah, q.s1, a * gi - x * gr);
    *di = 2.0 * fma(hpi, ex + fma(x, q.s1, q.s2), -fma(x, gi, a * gr));
}

// ------------------------------------------------------------------ wing polynomials
//
// The asymptotic series of Eq. asywofz, truncated after the term k = ASY_K, as a
// polynomial in u = 1/|z|^2 with per-line coefficients (FP32, |z| >= 6, a < WIDE_A).
// Term k is c_k Re(i z^-(2k+1))/sqrt(pi) = c_k Im(z^(2k+1)) u^(2k+1)/sqrt(pi),
// c_k = (2k-1)!!/2^k.  Writing z^m = x alpha_m + i beta_m with alpha_m, beta_m
// homogeneous polynomials in r = |z|^2 and a (x^2 = r - a^2), multiplication by
// z^2 = (r - 2a^2) + 2iax gives
//   alpha_{m+2} = (r - 2a^2) alpha_m - 2a beta_m,   beta_{m+2} = (r - 2a^2) beta_m + 2a (r - a^2) alpha_m,
// alpha_1 = 1, beta_1 = a.  With beta_{2k+1} = a r^k sum_j q_kj t^j (t = a^2/r):
//   H = sum_n C_n u^(n+1),  C_n = (a/sqrt(pi)) sum_{k+j=n} c_k q_kj a^(2j).
// For the adjoint, Euler's relation for the homogeneous terms (degree -(2k+1))
// gives H + x H_x + a H_a = -sum_k 2k T_k, and differentiating a^(2j+1) u^p at
// fixed x gives
//   a H_a = sum_n E_n u^(n+1) - 2 a^2 sum_n (n+1) C_n u^(n+2),  E_n = (1/sqrt(pi)) sum_{k+j=n} (2j+1) c_k q_kj a^(2j+1).
// With ASY_K = 6 the truncation and FP32 rounding stay below 4e-7 of H for |z| >= 6.
// To keep every coefficient inside the FP32 range (powers up to a^13, a^15 in the adjoint;
// a < WIDE_A, scaled strengths up to 1e18) the polynomials are written in v = ASY_S u (v < 1 for |z| >= 6):
// the table holds c_k q_kj / ASY_S^k and a^(2j) enters as (a^2/ASY_S)^j, so that
// H = u sum_n C'_n v^n with C'_n = C_n / ASY_S^n (a power of two: exact).
constexpr int ASY_K = 6;
constexpr int ASY_N = 2 * ASY_K + 1; // powers u^1 .. u^13
constexpr float ASY_S = 32.0f;
// Lines from this a on have |z| >= 100 at every point and take the K = 1 wing form where
// the lines beside them need the polynomial.
constexpr float WIDE_A = 100.0f;

struct AsyTable {
    float cq[ASY_K + 1][ASY_K + 1]; // c_k q_kj / ASY_S^k (j <= k)
};

constexpr AsyTable make_asy_table()
{
    // integer coefficients b[s] of beta_m = sum_s b[s] r^s a^(m-2s) and c[s] of
    // alpha_m = sum_s c[s] r^s a^(m-1-2s), advanced m -> m + 2
    long long b[ASY_K + 2] = {}, c[ASY_K + 2] = {};
    b[0] = 1;
    c[0] = 1;
    AsyTable t{};
    double ck = 1.0;
    for (int k = 0; k <= ASY_K; ++k) {
        if (k > 0) {
            long long nb[ASY_K + 2] = {}, nc[ASY_K + 2] = {};
            for (int s = 0; s <= k; ++s) {
                const long long bs1 = s > 0 ? b[s - 1] : 0, cs1 = s > 0 ? c[s - 1] : 0;
                nc[s] = cs1 - 2 * c[s] - 2 * b[s];
                nb[s] = bs1 - 2 * b[s] + 2 * cs1 - 2 * c[s];
            }
            for (int s = 0; s <= k; ++s) {
                b[s] = nb[s];
                c[s] = nc[s];
            }
            ck *= (2.0 * k - 1.0) / 2.0;
        }
        // beta_{2k+1} = sum_s b[s] r^s a^(2k+1-2s) = a r^k sum_j b[k-j] t^j
        double sk = 1.0;
        for (int i = 0; i < k; ++i) sk /= (double)ASY_S;
        for (int j = 0; j <= k; ++j) t.cq[k][j] = (float)(ck * (double)b[k - j] * sk);
    }
    return t;
}

__constant__ const AsyTable ASY = make_asy_table();

// C'_n (n = 0 .. ASY_N - 1) of H = u sum_n C'_n v^n, times amp.
__device__ __forceinline__ void asy_coeffs(float a, float amp, float (&C)[ASY_N])
{
    const float a2 = a * a * (1.0f / ASY_S);
    float ap[ASY_K + 1]; // amp a^(2j+1) / sqrt(pi)
    ap[0] = amp * a * (float)INV_SQRTPI;
#pragma unroll
    for (int j = 1; j <= ASY_K; ++j) ap[j] = ap[j - 1] * a2;
#pragma unroll
    for (int n = 0; n < ASY_N; ++n) C[n] = 0.0f;
#pragma unroll
    for (int k = 0; k <= ASY_K; ++k)
#pragma unroll
        for (int j = 0; j <= k; ++j) C[k + j] = fmaf(ASY.cq[k][j], ap[j], C[k + j]);
}

// Adjoint: f_T = u sum_n F_n v^n and f_b = u sum_n G_n v^n (n = 0 .. ASY_N) for
// f_T = aS V0 + hT D_beta + nn D_gamma and f_b = D_gamma, with V0 = amp H,
// D_beta = -amp (H + x H_x + a H_a), D_gamma = amp a H_a.
__device__ __forceinline__ void asy_coeffs_adj(float a, float amp, float aS, float hT, float nn,
                                               float (&F)[ASY_N + 1], float (&G)[ASY_N + 1])
{
    const float a2 = a * a * (1.0f / ASY_S); // a^2 / ASY_S
    float ap[ASY_K + 1];
    ap[0] = amp * a * (float)INV_SQRTPI;
#pragma unroll
    for (int j = 1; j <= ASY_K; ++j) ap[j] = ap[j - 1] * a2;
    float C[ASY_N], D[ASY_N], E[ASY_N];
#pragma unroll
    for (int n = 0; n < ASY_N; ++n) {
        C[n] = 0.0f;
        D[n] = 0.0f;
        E[n] = 0.0f;
    }
#pragma unroll
    for (int k = 0; k <= ASY_K; ++k)
#pragma unroll
        for (int j = 0; j <= k; ++j) {
            const float v = ASY.cq[k][j] * ap[j];
            C[k + j] += v;
            D[k + j] = fmaf(2.0f * (float)k, v, D[k + j]);
            E[k + j] = fmaf(2.0f * (float)j + 1.0f, v, E[k + j]);
        }
    // coefficient of u v^n: V0: C'_n, D_beta: D'_n, D_gamma: E'_n - 2 (a^2/ASY_S) n C'_{n-1}
#pragma unroll
    for (int n = 0; n <= ASY_N; ++n) {
        const float cn = n < ASY_N ? C[n] : 0.0f;
        const float dn = n < ASY_N ? D[n] : 0.0f;
        const float en = n < ASY_N ? E[n] : 0.0f;
        const float gm = en - (n > 0 ? 2.0f * a2 * (float)n * C[n - 1] : 0.0f);
        G[n] = gm;
        F[n] = fmaf(aS, cn, fmaf(hT, dn, nn * gm));
    }
}

// The FP64 path: the same polynomials in u, unscaled, truncated after K = 3, 4, 5, 7
// or 12 correction terms (2K + 1 coefficients) by |z| (Tier<double>).
constexpr int ASY64_K = 12;
struct AsyTable64 {
    double cq[ASY64_K + 1][ASY64_K + 1]; // c_k q_kj (j <= k)
};
constexpr AsyTable64 make_asy_table64()
{
    long long b[ASY64_K + 2] = {}, c[ASY64_K + 2] = {}; // as make_asy_table
    b[0] = 1;
    c[0] = 1;
    AsyTable64 t{};
    double ck = 1.0;
    for (int k = 0; k <= ASY64_K; ++k) {
        if (k > 0) {
            long long nb[ASY64_K + 2] = {}, nc[ASY64_K + 2] = {};
            for (int s = 0; s <= k; ++s) {
                const long long bs1 = s > 0 ? b[s - 1] : 0, cs1 = s > 0 ? c[s - 1] : 0;
                nc[s] = cs1 - 2 * c[s] - 2 * b[s];
                nb[s] = bs1 - 2 * b[s] + 2 * cs1 - 2 * c[s];
            }
            for (int s = 0; s <= k; ++s) {
                b[s] = nb[s];
                c[s] = nc[s];
            }
            ck *= (2.0 * k - 1.0) / 2.0;
        }
        for (int j = 0; j <= k; ++j) t.cq[k][j] = ck * (double)b[k - j];
    }
    return t;
}
__constant__ const AsyTable64 ASY64 = make_asy_table64();

// C_n (n = 0 .. 2K) of H = u sum_n C_n u^n, times amp
template <int K>
__device__ __forceinline__ void asy64_coeffs(double a, double amp, double (&C)[2 * K + 1])
{
    const double a2 = a * a;
    double ap = amp * a * INV_SQRTPI;
#pragma unroll
    for (int n = 0; n <= 2 * K; ++n) C[n] = 0.0;
#pragma unroll
    for (int j = 0; j <= K; ++j) {
#pragma unroll
        for (int k = j; k <= K; ++k) C[k + j] = fma(ASY64.cq[k][j], ap, C[k + j]);
        ap *= a2;
    }
}

// From the moments r_n = sum lambda u^(n+1) (n = 0 .. 2K + 1) of a line: the sums of
// lambda V0, lambda D_beta and lambda D_gamma (see asy_coeffs_adj).
template <int K>
__device__ __forceinline__ void asy64_adjoint(double a, double amp, const double (&r)[2 * K + 2], double* V0, double* Db,
                                              double* Dg)
{
    const double a2 = a * a;
    double ap = amp * a * INV_SQRTPI, v0 = 0.0, db = 0.0, dg = 0.0;
#pragma unroll
    for (int j = 0; j <= K; ++j) {
        double s = 0.0, sk = 0.0, sn = 0.0; // over k of c q r_n, k c q r_n, (n + 1) c q r_{n+1}
#pragma unroll
        for (int k = j; k <= K; ++k) {
            const double v = ASY64.cq[k][j] * r[k + j];
            s += v;
            sk = fma((double)k, v, sk);
            sn = fma(ASY64.cq[k][j] * (double)(k + j + 1), r[k + j + 1], sn);
        }
        v0 = fma(ap, s, v0);
        db = fma(ap, 2.0 * sk, db);
        dg = fma(ap, fma((double)(2 * j + 1), s, -2.0 * a2 * sn), dg);
        ap *= a2;
    }
    *V0 = v0;
    *Db = db;
    *Dg = dg;
}

} // namespace xsd
