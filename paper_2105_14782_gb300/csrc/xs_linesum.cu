// Line-by-line cross-section on sm_103a: per-line/per-layer parameters, the
// direct line-profile sum (Eq. crosssec summed over lines, Sec. 3.1) and its
// reverse-mode adjoint.
//
// Near and far.  Seen from a short interval of the grid, a line outside a few of the
// interval's half-widths is a smooth function: its profile's poles lie at
// centre +- i gamma, so a polynomial of low degree through Chebyshev nodes carries it
// to working precision.  The grid is cut into leaves of 32 points and, four at a
// time, into intervals of 128, 512 and 2,048 points.  A line is summed at the nodes
// of the largest interval that it is far from (and that lies wholly inside its
// wing cut), once, instead of at each grid point; what is near a leaf, or has its cut
// edge inside it, is summed point by point.  Lines are sorted, so all of these sets
// are index ranges and every in-cut (line, point) pair belongs to exactly one.
//
//   far_sum_kernel    node sums of the leaves and of the intervals above
//   down_kernel       node sums -> polynomials, from the larger intervals into the leaves
//   leaf_kernel       per leaf: its near lines at its points plus its polynomial; writes sigma
// and for the adjoint, where sum_j lambda_j f(nu_j) = sum_m Lambda_m f(node_m) for every
// polynomial f of the degree kept:
//   up_kernel         lambda -> the intervals' node weights Lambda
//   far_adjoint_kernel, leaf_adjoint_kernel
//
// The far condition (far_radius).  The centre lies at least kappa half-widths from the
// interval's middle (less where the smallest Lorentz width already keeps the poles
// away), and |z| >= Z0 at every point of the interval.  Measured over a in 1e-4 .. 100
// and half-widths of 0.01 .. 300 Doppler units against wofz, the interpolation error is
// below 1.6e-8 of the profile with 12 nodes, kappa = 3.3, Z0 = 6 (FP32; 1.9e-8 with 10
// and kappa = 4.5) and below 2e-16 with 18 nodes, kappa = 5, Z0 >= 8 (FP64, where the
// forms need |z| >= 10): under the rounding of the evaluations.  At one accuracy more
// nodes allow a smaller kappa: the far evaluations go as nodes x kappa, the near lines as
// kappa, but registers, polynomials and node weights as the nodes.  FP32, 100 layers of
// 220,000 lines forward + gradient: 34.7 ms with 10 nodes (kappa 4.5), 31.6 with 12,
// 32.1 with 14 (2.7), 31.6 with 16 (2.4); 3,060,000 lines x 4 layers 45.6, 45.2, 47.1,
// 46.4 ms; FP64, 60 layers of a retrieval 23.7 ms with 18 nodes, 22.9 with 20 (4.0) and
// 22.4 with 24 (3.1), but one layer 278, 285 and 290 us.
//
// What it saves: of the in-cut pairs of 220,000 lines on a 20,000-point grid about 1% are
// evaluated at a point and the rest at the nodes of an interval.  With every pair evaluated
// the 100-layer forward + gradient step on them took 224 ms, now 29.6; 4 layers of
// 3,060,000 lines on 100,000 points 564 and 44.3 ms; 20,000 lines on 20,000 points and 10
// layers forward 1.12 and 0.22 ms.
//
// Precision (XS_PREC_MIXED).  FP64: the strength exponent's argument, beta, line-centre
// offsets (then carried as float pairs), node sums, the intervals' polynomials and a leaf
// polynomial's constant term.  FP32 pairs: the strength's exponential and its products (to
// 1e-10, rounded once), running sums (TwoSum).  FP32: widths, stimulated emission, dlnS/dT, Voigt
// values, the leaf polynomials' other coefficients, the adjoint's lambda and, summed as pairs, the
// node weights.
// Measured against XS_PREC_FP64 over lists of 1,000 to 200,000 lines and 1e-6 to 1e3 bar, the
// relative rms error of sigma is 5.7e-8 to 1.13e-7 (5.8e-8 to 7e-6 when every pair was evaluated
// at its point), that of g_T with weights of mixed sign 1e-9 to 2.2e-8 of what weights of one
// sign give (1.6e-9 to 3.5e-7).  With the exponential, dlnS/dT or the leaf polynomials in
// FP64 instead none of these changes.  XS_PREC_FP64 does the same with double precision
// throughout.
#include <algorithm>
#include <type_traits>

#include "xs_device.cuh"
#include "xs_internal.h"

namespace xsd {

constexpr int LEAF = 32;       // grid points of a leaf: one per lane
constexpr int TOP_LOG = 6;     // the largest intervals have 64 leaves;
constexpr int TOP = 1 << TOP_LOG; // an interval has 2 or 4 below it (Tree::shift 1 or 2)
constexpr int LEVELS = TOP_LOG + 1; // most levels
// Neighbouring intervals of one block share most lines.  Two warps end a block sooner than
// four, whose registers wait for the longest list: 20,000 lines x 10 layers 217 against
// 222 us, 100 layers with the gradient 31.6 against 32.1 ms (eight warps: 6% above four).
constexpr int FAR_WARPS = 2;

// most warps of a leaf kernel's block (choose_leaf_blocks)
template <class R> struct LeafWarps { static constexpr int v = 4; };
template <> struct LeafWarps<double> { static constexpr int v = 8; };

// nodes and far condition per precision
template <class R> struct Far;
template <> struct Far<float> {
    static constexpr int n = 12;
    static constexpr double kappa = 3.3, Z0 = 6.0;
};
template <> struct Far<double> {
    static constexpr int n = 18;
    static constexpr double kappa = 5.0, Z0 = 10.0;
};

template <class R> static __device__ const ChebTable<Far<R>::n> CHEB = make_cheb<Far<R>::n>();
template <int n> __device__ __forceinline__ double cheb(int k, int m)
{
    if constexpr (n == Far<float>::n) return CHEB<float>.T[k][m];
    else return CHEB<double>.T[k][m];
}
struct ChebTableF {
    float T[Far<float>::n][Far<float>::n];
};
constexpr ChebTableF make_cheb_f()
{
    constexpr int n = Far<float>::n;
    ChebTableF r{};
    const ChebTable<n> c = make_cheb<n>();
    for (int k = 0; k < n; ++k)
        for (int m = 0; m < n; ++m) r.T[k][m] = (float)c.T[k][m];
    return r;
}
__device__ const ChebTableF CHEB_F = make_cheb_f();
// in the type of the path
__device__ __forceinline__ float cheb_r(float, int k, int m) { return CHEB_F.T[k][m]; }
__device__ __forceinline__ double cheb_r(double, int k, int m) { return CHEB<double>.T[k][m]; }
// the nodes as literals for unrolled loops
template <int n> struct NodeTable {
    float t[n];
};
template <int n>
constexpr NodeTable<n> make_nodes()
{
    NodeTable<n> r{};
    const ChebTable<n> c = make_cheb<n>();
    for (int m = 0; m < n; ++m) r.t[m] = (float)c.T[1][m];
    return r;
}

// Middle, half-width and its reciprocal (0 in an interval of one point).
struct Geo {
    double mid, h, inv;
};

// Intervals of the grid, all levels, leaves first.
struct Tree {
    const Geo* geo;
    const int2* cov;    // lines [x, y) that cover the interval with their cut
    const int2* win;    // lines [x, y) with an in-cut point in it (leaves only)
    const int2* pq;     // per layer: lines [x, y) too near for the far form
    int cnt[LEVELS], off[LEVELS], total;
    int shift, top;     // log2 of the intervals below one; the top level: TOP_LOG / shift
    int on;             // 0: no intervals (small workspaces): every line is near
};

// Line arrays of one layer.
template <class R>
struct Lines {
    using R4 = typename vec4<R>::type;
    const double* nu_hat;
    const float2* nuf; // centre - nu[0] as hi + lo floats (FP32)
    const int2* jr;
    const R4 *r1, *r2;
    const R* r3;
    const R* clo;
};

// Work of the far kernels: blocks of FAR_WARPS neighbouring intervals of a level and
// one part of their lists, largest intervals (longest lists) first.
struct FarWork {
    int parts[LEVELS], block0[LEVELS]; // block0: first block of the level
    size_t out0[LEVELS];               // first node-sum row of the level (in rows of n)
    int slot0[LEVELS], slots;          // first adjoint slot of the level, slots a layer
    size_t rows;                       // node-sum rows of all levels
};

// One species of a launch: its lists, workspace arrays and plan.  The line sums of a
// model's species are independent of one another and run in the same launches
// (blockIdx.z), which halves the launches of a two-species step and fills the chip with
// the blocks of both.
template <class R>
struct Species {
    using R4 = typename vec4<R>::type;
    Lines<R> ln;
    const double *inv_nu, *ln_S0, *elower, *gamma_ref, *n_temp;
    double mass, qexp;
    int64_t nl;
    Tree tree;
    FarWork fw;
    int setup_blocks, param_blocks, far_blocks;
    // per-call arrays (the same memory as the const pointers above)
    int2* jr;
    float2* nuf;
    double* w_inv_nu;
    float* agg;
    R4 *rec1, *rec2;
    R *rec3, *clo;
    Geo* geo;
    int2 *cov, *win, *pq;
    double *sums, *coef, *near; // forward: node sums, leaf polynomials, slices' sums
    R* wts;              // adjoint: node weights,
    double *slots, *leaf, *gbl; // and the partials of the far, the leaf and the reduction kernel
    void* sigma;
    const double* g_sigma;
    double *g_T, *g_b;
};
template <class R>
struct Batch {
    Species<R> s[XS_MAX_SPECIES];
    int n;
};

// ------------------------------------------------------------------ setup

// lo if upper == 0: first grid index with nu_j - c >= -W; else the last with nu_j - c <= W
// (double precision, boundary included).  Both are non-decreasing along a sorted line list.
__device__ __forceinline__ int cut_index(const double* nu, int64_t N, double c, double W, int upper)
{
    int64_t lo = 0, hi = N;
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        const double d = nu[m] - c;
        if (upper ? d > W : d >= -W) hi = m; else lo = m + 1;
    }
    return (int)(upper ? lo - 1 : lo);
}

// first line l whose cut has grid point v at or below its upper end (upper != 0:
// nu_v - c <= W) or strictly below its lower end (upper == 0: nu_v - c < -W)
__device__ __forceinline__ int first_line(const double* nu_hat, int64_t nl, double v, double W, int upper)
{
    int64_t lo = 0, hi = nl;
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        const double d = v - nu_hat[m];
        if (upper ? !(d > W) : !(d >= -W)) hi = m; else lo = m + 1;
    }
    return (int)lo;
}

// One thread per search: cut ranges of the lines (two each) and their centres
// relative to the first grid point as float pairs, the intervals' line ranges (four
// each) and geometry, and the start values of the per-layer minima.
template <class R>
__global__ void setup_kernel(const __grid_constant__ Batch<R> batch, const double* __restrict__ nu, int64_t N, double W,
                             int n_agg)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    const double* __restrict__ nu_hat = sp.ln.nu_hat;
    const int64_t nl = sp.nl;
    const Tree& tr = sp.tree;
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 2 * nl) {
        const int64_t l = t >> 1;
        const int upper = (int)(t & 1);
        const double c = nu_hat[l];
        ((int*)sp.jr)[t] = cut_index(nu, N, c, W, upper);
        if (!upper) sp.w_inv_nu[l] = 1.0 / c;
        if (sp.nuf && upper) {
            const double o = c - nu[0];
            const float h = (float)o;
            sp.nuf[l] = make_float2(h, (float)(o - (double)h));
        }
        return;
    }
    t -= 2 * nl;
    if (t < n_agg) {
        sp.agg[t] = __int_as_float(0x7f800000); // +inf: minima
        return;
    }
    t -= n_agg;
    if (!tr.on || t >= 4 * (int64_t)tr.total) return;
    const int which = (int)(t & 3), q = (int)(t >> 2);
    int k = tr.top;
    while (k > 0 && q < tr.off[k]) --k;
    const int points = LEAF << (tr.shift * k);
    const int64_t j0 = (int64_t)(q - tr.off[k]) * points;
    const int64_t j1 = min64(N, j0 + points) - 1;
    const double v0 = nu[j0], v1 = nu[j1];
    if (which == 0) {
        const double h = 0.5 * (v1 - v0);
        sp.geo[q] = {0.5 * (v0 + v1), h, h > 0.0 ? 1.0 / h : 0.0};
        sp.cov[q].x = first_line(nu_hat, nl, v1, W, 1); // covers v1 from its lower side on
    } else if (which == 1) {
        sp.cov[q].y = first_line(nu_hat, nl, v0, W, 0); // first that no longer reaches v0
    } else if (k == 0) {
        if (which == 2)
            sp.win[q].x = first_line(nu_hat, nl, v0, W, 1);
        else
            sp.win[q].y = first_line(nu_hat, nl, v1, W, 0);
    }
}

__global__ void sorted_check_kernel(const double* __restrict__ nu_hat, int64_t nl, int* __restrict__ bad)
{
    int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l + 1 < nl && !(nu_hat[l] <= nu_hat[l + 1])) atomicOr(bad, 1);
}

__global__ void grid_check_kernel(const double* __restrict__ nu, int64_t N, int* __restrict__ bad)
{
    int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j + 1 < N && !(nu[j] < nu[j + 1])) atomicOr(bad, 1);
}

// ------------------------------------------------------------------ line parameters

// e^{-(k h)^2}, k = 1.., for the two series steps (h = 0.7f and h = 0.5)
__device__ const float KC_E32[10] = {0.612626433f, 0.140858427f, 0.0121551799f, 0.00039366915f, 4.78511947e-06f,
                                     2.18295906e-08f, 3.73757449e-11f, 2.40173736e-14f, 5.79232066e-18f,
                                     5.24289428e-22f};
// K(a) = erfcx(a) - (2 a h/pi) sum_k e^{-(kh)^2} / ((kh)^2 + a^2), the per-line constant
// of the small-|z| series (see xs_device.cuh)
__device__ __forceinline__ float series_K(float a)
{
    const float h = Tier<float>::h;
    float s1 = 0.0f;
#pragma unroll
    for (int k = 1; k <= 10; ++k) {
        float kh = (float)k * h;
        s1 = fmaf(KC_E32[k - 1], rcp_fast(fmaf(kh, kh, a * a)), s1);
    }
    return erfcxf(a) - 2.0f * a * h * (float)(1.0 / PI) * s1;
}
__device__ __forceinline__ double series_K(double a)
{
    const double h = Tier<double>::h;
    double s1 = 0.0;
    for (int k = 1; k <= 13; ++k) {
        double kh = k * h;
        s1 += KC_E64[k - 1] / (kh * kh + a * a);
    }
    return erfcx(a) - 2.0 * a * h / PI * s1;
}

// Layer constants of the line parameters.
struct LayerConst {
    double kE, kq, kc, kg, k2E, kqT; // exponent slopes, c nu_hat, pressure factor, dlnS slopes
    double lnTr, T, bk, bT, Patm; // ln(T/296), T, beta cL/nu_hat, 1/T - 1/296, P/atm
};

__device__ __forceinline__ LayerConst layer_const(double Tn, double Pn, double mass, double qexp, double sb)
{
    LayerConst k;
    const double lnTr = log(Tn / Tref), iT = 1.0 / Tn;
    k.bT = iT - 1.0 / Tref;
    k.kE = c2 * k.bT;
    k.Patm = Pn / bar_per_atm;
    k.kq = qexp * lnTr;
    k.bk = sqrt(kB * Tn / (mass * amu));
    k.kc = cL / (SQRT2 * k.bk);
    k.kg = sb * k.Patm;
    k.k2E = c2 * iT * iT;
    k.kqT = qexp * iT;
    k.lnTr = lnTr;
    k.T = Tn;
    return k;
}

// 2^(i/64) as hi + lo floats
struct Exp2Table {
    float hi[64], lo[64];
};
constexpr double LN2 = 0.69314718055994530942;
constexpr Exp2Table make_exp2_table()
{
    Exp2Table t{};
    for (int i = 0; i < 64; ++i) {
        const double x = i * LN2 / 64;
        double s = 1.0;
        for (int k = 20; k >= 1; --k) s = 1.0 + s * x / k;
        t.hi[i] = (float)s;
        t.lo[i] = (float)(s - (double)t.hi[i]);
    }
    return t;
}
__device__ const Exp2Table EXP2 = make_exp2_table();

// e^v = 2^e (hi + lo), 1 <= hi < 2, to about 1e-10, table-driven (Tang 1989): the argument
// is reduced in FP64 (three operations), the rest is FP32.
__device__ __forceinline__ void exp_pair(double v, const float* tab, int* e, float* hi, float* lo)
{
    const int top = __double2hiint(v) & 0x7fffffff;
    if (top >= 0x40900000 && top <= 0x7ff00000 && v == v) v = v < 0.0 ? -1000.0 : 1000.0; // beyond FP32 either way
    const double magic = 6755399441055744.0; // 1.5 2^52: rounds to an integer
    const double t = fma(v, 64.0 / LN2, magic);
    const int k = __double2loint(t);
    const float r = (float)fma(t - magic, -LN2 / 64, v);
    const float h = tab[k & 63];
    *e = k >> 6;
    *hi = h;
    *lo = fmaf(h, fmaf(r * r, fmaf(r, 1.0f / 6.0f, 0.5f), r), tab[64 + (k & 63)]);
}

// Per (layer, line), rounded once to R:
//   rec1 = {G = gamma^2, Al = s gamma/pi, F1 = 1.5 B Al, F2 = -2 G B Al}   (B = 2 beta^2)
//   rec2 = {c = 1/(sqrt2 beta), a = gamma c, Av = s c / sqrt(pi), Kc = K(a)}
//   clo  = c - (R)c,  rec3 = {dlnS/dT, -n/T} (adjoint only)
// s = S(T) * scale.  The argument of the Boltzmann factor of S (Eq. Slog) and c are formed in
// FP64 in both paths; in the FP32 path the factor, c and their products are carried as hi + lo
// floats and what only needs ~1e-7 (stimulated emission, the width's temperature power, K(a))
// is FP32.  Per layer: agg[4n .. 4n+2] = min c, min a, min gamma.
//
// Bound by FP64 operations (2 lanes a clock and SM): what depends on the layer alone is
// formed once a block, 1/nu_hat once a call, and the exponential and the products of the
// FP32 path run in FP32: about 20 FP64 operations and conversions a line instead of about
// 200 (220,000 lines x 100 layers: 6.9 ms before).
template <class R>
__global__ void __launch_bounds__(256) line_params_kernel(const __grid_constant__ Batch<R> batch,
                                                          const double* __restrict__ T,
                                                          const double* __restrict__ P_bar, int layer0, double sb,
                                                          bool want_rec3)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    if ((int)blockIdx.x >= sp.param_blocks) return;
    const double* __restrict__ nu_hat = sp.ln.nu_hat;
    const double* __restrict__ inv_nu = sp.inv_nu;
    const double* __restrict__ ln_S0 = sp.ln_S0;
    const double* __restrict__ elower = sp.elower;
    const double* __restrict__ gamma_ref = sp.gamma_ref;
    const double* __restrict__ n_temp = sp.n_temp;
    const int64_t nl = sp.nl;
    const double mass = sp.mass, qexp = sp.qexp;
    auto* __restrict__ rec1 = sp.rec1;
    auto* __restrict__ rec2 = sp.rec2;
    R* __restrict__ clo = sp.clo;
    R* __restrict__ rec3 = want_rec3 ? sp.rec3 : nullptr;
    float* __restrict__ agg = sp.agg;
    constexpr bool FAST = std::is_same<R, float>::value;
    __shared__ LayerConst lc;
    __shared__ float tab[128];
    const int n = blockIdx.y;
    if (threadIdx.x == 0) lc = layer_const(T[layer0 + n], P_bar[layer0 + n], mass, qexp, sb);
    if (FAST && threadIdx.x >= 128) {
        const int i = threadIdx.x - 128;
        tab[i] = i < 64 ? EXP2.hi[i] : EXP2.lo[i - 64];
    }
    __syncthreads();
    const LayerConst k = lc;
    const float lnTr = (float)k.lnTr, Tf = (float)k.T;
    float cmin = __int_as_float(0x7f800000), amin = cmin, gmin = cmin;
    for (int64_t l = (int64_t)blockIdx.x * 256 + threadIdx.x; l < nl; l += (int64_t)sp.param_blocks * 256) {
        const double nuh = nu_hat[l], E = elower[l];
        const double c = FAST ? k.kc * inv_nu[l] : 1.0 / (SQRT2 * (k.bk * nuh / cL));
        const R cr = (R)c, c_lo = (R)(c - (double)cr); // the part of c the rounded value misses
        R gam, Al, Av;
        float u = 0.0f;
        if constexpr (FAST) {
            const float cu = (float)(c2 * nuh);
            u = cu / Tf;
            const float stim = expm1f(-u) / expm1f(-cu / (float)Tref);
            gam = (float)(k.kg * gamma_ref[l]) * expf(-(float)n_temp[l] * lnTr);
            int e;
            float hi, lo;
            exp_pair(fma(-E, k.kE, ln_S0[l]) - k.kq, tab, &e, &hi, &lo);
            // s = 2^e (hi + lo) stim 2^80, products in FP32 with the low part carried
            const float s = hi * stim, sl = fmaf(hi, stim, -s) + lo * stim;
            const float g = gam * (float)(1.0 / PI), ci = cr * (float)INV_SQRTPI;
            constexpr float gl0 = (float)(1.0 / PI - (double)(float)(1.0 / PI));
            constexpr float cl0 = (float)(INV_SQRTPI - (double)(float)INV_SQRTPI);
            const float gl = fmaf(gam, (float)(1.0 / PI), -g) + gam * gl0;
            const float cl = fmaf(cr, (float)INV_SQRTPI, -ci) + fmaf(cr, cl0, (float)INV_SQRTPI * c_lo); // all of c
            Al = ldexpf(fmaf(s, g, fmaf(s, gl, sl * g)), e + MIXED_SCALE_LOG2);
            Av = ldexpf(fmaf(s, ci, fmaf(s, cl, sl * ci)), e + MIXED_SCALE_LOG2);
        } else {
            // the checking path keeps the plain expressions, operation by operation
            const double s = exp(ln_S0[l] - c2 * E * k.bT - k.kq) * (expm1(-c2 * nuh / k.T) / expm1(-c2 * nuh / Tref));
            gam = sb * gamma_ref[l] * exp(-n_temp[l] * k.lnTr) * k.Patm;
            Al = s * gam / PI;
            Av = s * c * INV_SQRTPI;
        }
        const R a = gam * cr;
        const R B = R(1) / (cr * cr);
        const R G = gam * gam;
        const R Kc = (a * a < (R)Tier<R>::z2_series) ? series_K(a) : R(0);
        const size_t idx = (size_t)n * nl + l;
        typename vec4<R>::type v1, v2;
        v1.x = G;
        v1.y = Al;
        v1.z = R(1.5) * B * Al;
        v1.w = R(-2) * G * B * Al;
        v2.x = cr;
        v2.y = a;
        v2.z = Av;
        v2.w = Kc;
        rec1[idx] = v1;
        rec2[idx] = v2;
        if (FAST) clo[idx] = c_lo;
        if (rec3) {
            if constexpr (FAST) {
                const float aS = (float)fma(k.k2E, E, -k.kqT) - (u / Tf) / expm1f(u);
                ((float2*)rec3)[idx] = make_float2(aS, -(float)n_temp[l] / Tf);
            } else {
                const double ud = c2 * nuh / k.T;
                rec3[2 * idx] = (c2 * E / (k.T * k.T) - qexp / k.T) - (ud / k.T) / expm1(ud);
                rec3[2 * idx + 1] = -n_temp[l] / k.T;
            }
        }
        cmin = fminf(cmin, (float)cr * (1.0f - 1e-6f));
        amin = fminf(amin, (float)a * (1.0f - 1e-6f));
        gmin = fminf(gmin, (float)gam * (1.0f - 1e-6f));
    }
    // warp min then one atomic per warp (positive floats order like their bits)
    for (int o = 16; o > 0; o >>= 1) {
        cmin = fminf(cmin, __shfl_xor_sync(0xffffffffu, cmin, o));
        amin = fminf(amin, __shfl_xor_sync(0xffffffffu, amin, o));
        gmin = fminf(gmin, __shfl_xor_sync(0xffffffffu, gmin, o));
    }
    if ((threadIdx.x & 31) == 0 && cmin < __int_as_float(0x7f800000)) {
        atomicMin((int*)&agg[4 * (layer0 + n)], __float_as_int(cmin));
        atomicMin((int*)&agg[4 * (layer0 + n) + 1], __float_as_int(amin));
        atomicMin((int*)&agg[4 * (layer0 + n) + 2], __float_as_int(gmin));
    }
}

// ------------------------------------------------------------------ far sets

// Distance of a centre from the middle of an interval (half-width h) from which the
// far form holds for every line of a layer with smallest c, a and gamma.
template <class R>
__device__ __forceinline__ double far_radius(double h, double cmin, double amin, double gmin)
{
    const double kh = Far<R>::kappa * h, g = fmax(gmin, 0.0), a = fmax(amin, 0.0), Z0 = Far<R>::Z0;
    const double rk = kh > g ? sqrt(kh * kh - g * g) : 0.0;
    const double rz = a < Z0 ? h + sqrt(Z0 * Z0 - a * a) / cmin : 0.0;
    return fmax(rk, rz);
}

// pq[layer][interval]: lines with |centre - middle| below the far radius
template <class R>
__global__ void near_range_kernel(const __grid_constant__ Batch<R> batch, int layer0)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    const double* __restrict__ nu_hat = sp.ln.nu_hat;
    const int64_t nl = sp.nl;
    const Tree& tr = sp.tree;
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 2 * (int64_t)tr.total) return;
    const int q = (int)(t >> 1), n = blockIdx.y;
    const bool upper = t & 1;
    const Geo g = tr.geo[q];
    const float* ag = sp.agg + 4 * (layer0 + n);
    const double r = far_radius<R>(g.h, ag[0], ag[1], ag[2]);
    const double v = upper ? g.mid + r : g.mid - r;
    int64_t lo = 0, hi = nl; // first line with centre >= v (upper) or > v
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        if (upper ? nu_hat[m] >= v : nu_hat[m] > v) hi = m; else lo = m + 1;
    }
    ((int*)sp.pq)[2 * (size_t)tr.total * n + t] = (int)lo;
}

// Far lines of an interval: [a, p) and [q, b); its parent's, [A, P) and [Q, B), are
// inside them (a side on which the parent has none: A = P = a or Q = B = b).
struct FarSet {
    int a, p, q, b;
    int A, P, Q, B;
    __device__ __forceinline__ bool in_order(int64_t nl) const
    {
        return 0 <= a && a <= A && A <= P && P <= p && p <= q && q <= Q && Q <= B && B <= b && b <= nl;
    }
};

__device__ __forceinline__ int clampi(int v, int lo, int hi) { return min(max(v, lo), hi); }

// The set of interval i of a level, from the top interval above it downwards: near
// lines are kept out of the parent's far ones.
template <int shift>
__device__ __forceinline__ FarSet far_set(const Tree& tr, int level, int i, int nloc)
{
    FarSet f{};
    bool left = false, right = false; // the interval above has far lines on that side
    for (int k = TOP_LOG / shift; k >= level; --k) {
        const int at = tr.off[k] + (i >> (shift * (k - level)));
        if (!XS_CHECK(at >= 0 && at < tr.total)) return FarSet{};
        const int2 c = tr.cov[at], s = tr.pq[(size_t)tr.total * nloc + at];
        const int a = c.x, b = max(c.x, c.y);
        f.A = left ? f.a : a;
        f.P = left ? f.p : a;
        f.Q = right ? f.q : b;
        f.B = right ? f.b : b;
        f.p = clampi(s.x, f.P, f.Q);
        f.q = clampi(s.y, f.p, f.Q);
        f.a = a;
        f.b = b;
        left = f.p > f.a;
        right = f.b > f.q;
    }
    return f;
}

// both steps unrolled: the loads of a loop of unknown length wait for one another
__device__ __forceinline__ FarSet far_set(const Tree& tr, int level, int i, int nloc)
{
    return tr.shift == 2 ? far_set<2>(tr, level, i, nloc) : far_set<1>(tr, level, i, nloc);
}

// The lines of an interval that are not its parent's, as one numbering 0 .. total - 1.
struct FarList {
    int s0, s1, s2, s3, c1, c2, c3, total;
    __device__ __forceinline__ explicit FarList(const FarSet& f)
    {
        s0 = f.a;
        c1 = f.A - f.a;
        s1 = f.P - c1;
        c2 = c1 + (f.p - f.P);
        s2 = f.q - c2;
        c3 = c2 + (f.Q - f.q);
        s3 = f.B - c3;
        total = c3 + (f.b - f.B);
    }
    __device__ __forceinline__ int line(int t) const { return t + (t < c1 ? s0 : t < c2 ? s1 : t < c3 ? s2 : s3); }
};

// ------------------------------------------------------------------ packed helpers

__device__ __forceinline__ float2 dup(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 lo2(const float4& v) { return make_float2(v.x, v.y); }
__device__ __forceinline__ float2 hi2(const float4& v) { return make_float2(v.z, v.w); }
// both reciprocals from one: 1/D1 = D2/(D1 D2), 1/D2 = D1/(D1 D2) (about 1.5 ulp); trades
// a second MUFU op (16 a clock and SM) for FP32 multiplies (128 a clock and SM)
__device__ __forceinline__ float2 rcp2_shared(float2 v)
{
    const float r = rcp_fast(v.x * v.y);
    return __fmul2_rn(make_float2(v.y, v.x), make_float2(r, r));
}
// (hi, lo) += v, TwoSum
__device__ __forceinline__ void two_sum2(float2& hi, float2& lo, float2 v)
{
    const float2 s = __fadd2_rn(hi, v);
    const float2 mhi = make_float2(-hi.x, -hi.y);
    const float2 bb = __fadd2_rn(s, mhi);
    const float2 nb = make_float2(-bb.x, -bb.y);
    const float2 t = __fadd2_rn(s, nb); // s - bb
    const float2 e1 = __fadd2_rn(hi, make_float2(-t.x, -t.y));
    lo = __fadd2_rn(lo, __fadd2_rn(e1, __fadd2_rn(v, nb)));
    hi = s;
}
__device__ __forceinline__ void two_sum(float& hi, float& lo, float v)
{
    const float s = hi + v, bb = s - hi;
    lo += (hi - (s - bb)) + (v - bb);
    hi = s;
}

// A sum carried as hi + lo floats, and its addition (TwoSum): eight FP32 operations where
// an FP64 addition takes the FP64 pipe for 16 clocks.
struct Pair {
    float hi, lo;
};
__device__ __forceinline__ Pair add(const Pair& a, const Pair& b)
{
    const float s = a.hi + b.hi, bb = s - a.hi;
    return {s, (a.lo + b.lo) + ((a.hi - (s - bb)) + (b.hi - bb))};
}
__device__ __forceinline__ float add(float a, float b) { return a + b; }
__device__ __forceinline__ double add(double a, double b) { return a + b; }
__device__ __forceinline__ Pair shfl_xor(const Pair& v, int o)
{
    return {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)};
}
__device__ __forceinline__ float shfl_xor(float v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double shfl_xor(double v, int o) { return __shfl_xor_sync(0xffffffffu, v, o); }
__device__ __forceinline__ double to_double(const Pair& v) { return (double)v.hi + (double)v.lo; }

// Sums v[0 .. n-1] over the warp, each sum ending in one lane: halving exchanges, so
// about n adds a lane instead of 5 n.  Returns the lane's sum; idx its index or -1.
template <int n, int o, class V>
__device__ __forceinline__ V reduce_scatter_step(V (&v)[n], int base, int cnt, int& idx)
{
    constexpr int h = (n + 1) / 2;
    const bool up = (threadIdx.x & o) != 0;
    V w[h];
    if constexpr (n == 1) {
        w[0] = add(v[0], shfl_xor(v[0], o));
    } else {
#pragma unroll
        for (int i = 0; i < h; ++i) {
            const V a = v[i], b = (i + h < n) ? v[i + h] : V{};
            w[i] = add(up ? b : a, shfl_xor(up ? a : b, o));
        }
        base += up ? h : 0;
        cnt = up ? max(cnt - h, 0) : min(cnt, h);
    }
    if constexpr (o == 1) {
        idx = cnt > 0 ? base : -1;
        return w[0];
    } else {
        return reduce_scatter_step<h, o / 2, V>(w, base, cnt, idx);
    }
}
template <int n, class V>
__device__ __forceinline__ V warp_reduce_scatter(V (&v)[n], int& idx)
{
    return reduce_scatter_step<n, 16, V>(v, 0, n, idx);
}
template <class V>
__device__ __forceinline__ V warp_sum(V v)
{
    for (int o = 16; o > 0; o >>= 1) v = add(v, shfl_xor(v, o));
    return v;
}

// ------------------------------------------------------------------ far lines, FP32
//
// The profile in rho = 1/(dnu^2 + gamma^2), from the asymptotic series of Eq. asywofz
// (B = 2 beta^2, G = gamma^2, Al = s gamma/pi):
//   K = 1: Av H = rho (k0 + rho (k1 + rho F2)),  k0 = Al, k1 = 1.5 B Al, F2 = -2 G B Al
//   K = 2: rho (k0 + rho (k1 + rho (k2 + rho (k3 + rho k4)))),
//          k2 = Al (3.75 B^2 - 2 G B), k3 = -15 G B^2 Al, k4 = 12 G^2 B^2 Al
// K = 1 where |z| >= 100 (the K = 2 terms are below 4e-8 there), K = 2 from |z| = 16.5
// (the first dropped term is 15/(8 |z|^6), below 1e-7), the K = 6 polynomial in
// 1/|z|^2 (asy_coeffs) from |z| = 6.  A warp takes the cheapest form that all of its
// 32 lines allow, but for lines with a >= WIDE_A among others that need the polynomial: its
// powers of a leave the FP32 range at a of a few hundred, and a wing form holds for such a
// line everywhere.
constexpr float WING1_Z2 = 1.0e4f, WING2_Z2 = 272.25f;

__device__ __forceinline__ void wing2_consts(const float4& p1, float c, float* k2, float* k3, float* k4)
{
    const float B = rcp_fast(c * c);
    *k2 = fmaf(2.5f * B, p1.z, p1.w);
    *k3 = 7.5f * B * p1.w;
    *k4 = -6.0f * p1.x * B * p1.w;
}

// u sum_{n<13} C'_n v^n for two points, v = ASY_S u
__device__ __forceinline__ float2 horner13_2(const float (&C)[ASY_N], float2 u)
{
    const float2 v = __fmul2_rn(u, dup(ASY_S));
    float2 p = dup(C[ASY_N - 1]);
#pragma unroll
    for (int n = ASY_N - 2; n >= 0; --n) p = __ffma2_rn(p, v, dup(C[n]));
    return __fmul2_rn(p, u);
}

// An interval as the warps see it.
struct Span {
    double mid, h;
    float rh, rl; // mid - nu[0] as hi + lo floats
    __device__ __forceinline__ Span(const Geo& g, double nu0) : mid(g.mid), h(g.h)
    {
        const double o = mid - nu0;
        rh = (float)o;
        rl = (float)(o - (double)rh);
    }
};

constexpr int FAR_FOLD = 16; // lines of a lane between two foldings of its FP32 partial sums

// Sums over the lines t0 .. t1 - 1 of a list of Av H at the nodes: returns the sum at node
// idx (-1: none in this lane).  Lanes hold lines, 32 at a time, the nodes are in registers:
// a line is read once for all nodes, with no staging.
__device__ __forceinline__ double far_sum(const Lines<float>& ln, const FarList& fl, int t0, int t1, const Span& sp,
                                          float cmin, int& idx)
{
    constexpr int H = Far<float>::n / 2;
    constexpr NodeTable<Far<float>::n> nt = make_nodes<Far<float>::n>();
    const int lane = threadIdx.x & 31;
    const float h = (float)sp.h, c2min = cmin * cmin;
    float2 o2[H], acc[H], hi[H], lo[H];
#pragma unroll
    for (int p = 0; p < H; ++p) {
        o2[p] = make_float2(h * nt.t[2 * p], h * nt.t[2 * p + 1]);
        acc[p] = hi[p] = lo[p] = dup(0.0f);
    }
    int l = 0;
    float2 nf = make_float2(0.f, 0.f);
    float4 p1 = make_float4(1.f, 0.f, 0.f, 0.f);
    if (t0 < t1) {
        l = fl.line(min(t0 + lane, t1 - 1));
        nf = ln.nuf[l];
        p1 = ln.r1[l];
    }
    int fold = FAR_FOLD;
    for (int t = t0; t < t1; t += 32) {
        const bool live = t + lane < t1;
        const float nb = (sp.rh - nf.x) + (sp.rl - nf.y); // middle - centre
        const float G = p1.x;
        const float4 q1 = live ? p1 : make_float4(G, 0.f, 0.f, 0.f);
        const int lc = l;
        if (t + 32 < t1) { // next 32 lines in flight
            l = fl.line(min(t + 32 + lane, t1 - 1));
            nf = ln.nuf[l];
            p1 = ln.r1[l];
        }
        const float dist = fmaxf(fabsf(nb) - h, 0.0f);
        const float D0 = fmaf(dist, dist, G), z2 = D0 * c2min;
        const float2 nb2 = dup(nb), G2 = dup(G), k0 = dup(q1.y), k1 = dup(q1.z);
        if (__all_sync(0xffffffffu, z2 >= WING1_Z2)) {
            // the F2 term is 2 a^2/|z|^4 = 2 G/(D z2) of the leading one
            if (__all_sync(0xffffffffu, 2.0f * G <= 2.0e-8f * z2 * D0)) {
#pragma unroll
                for (int p = 0; p < H; ++p) {
                    const float2 d = __fadd2_rn(o2[p], nb2);
                    const float2 rho = rcp2_shared(__ffma2_rn(d, d, G2));
                    acc[p] = __ffma2_rn(rho, __ffma2_rn(rho, k1, k0), acc[p]);
                }
            } else {
                const float2 f2 = dup(q1.w);
#pragma unroll
                for (int p = 0; p < H; ++p) {
                    const float2 d = __fadd2_rn(o2[p], nb2);
                    const float2 rho = rcp2_shared(__ffma2_rn(d, d, G2));
                    acc[p] = __ffma2_rn(rho, __ffma2_rn(__ffma2_rn(f2, rho, k1), rho, k0), acc[p]);
                }
            }
        } else {
            const float4 p2 = ln.r2[lc];
            if (__all_sync(0xffffffffu, z2 >= WING2_Z2) || p2.y >= WIDE_A) {
                float a2, a3, a4;
                wing2_consts(q1, p2.x, &a2, &a3, &a4);
                const float2 k2 = dup(a2), k3 = dup(a3), k4 = dup(a4);
#pragma unroll
                for (int p = 0; p < H; ++p) {
                    const float2 d = __fadd2_rn(o2[p], nb2);
                    const float2 rho = rcp2_shared(__ffma2_rn(d, d, G2));
                    const float2 u = __ffma2_rn(
                        __ffma2_rn(__ffma2_rn(__ffma2_rn(k4, rho, k3), rho, k2), rho, k1), rho, k0);
                    acc[p] = __ffma2_rn(rho, u, acc[p]);
                }
            } else {
                float C[ASY_N];
                asy_coeffs(p2.y, live ? p2.z : 0.0f, C);
                const float2 c2 = dup(p2.x), aa = dup(p2.y * p2.y);
#pragma unroll
                for (int p = 0; p < H; ++p) {
                    const float2 x = __fmul2_rn(__fadd2_rn(o2[p], nb2), c2);
                    acc[p] = __fadd2_rn(acc[p], horner13_2(C, rcp2_shared(__ffma2_rn(x, x, aa))));
                }
            }
        }
        if (--fold == 0) {
            fold = FAR_FOLD;
#pragma unroll
            for (int p = 0; p < H; ++p) {
                two_sum2(hi[p], lo[p], acc[p]);
                acc[p] = dup(0.0f);
            }
        }
    }
    Pair v[2 * H];
#pragma unroll
    for (int p = 0; p < H; ++p) {
        two_sum2(hi[p], lo[p], acc[p]);
        v[2 * p] = {hi[p].x, lo[p].x};
        v[2 * p + 1] = {hi[p].y, lo[p].y};
    }
    return to_double(warp_reduce_scatter(v, idx));
}

// Adjoint: per evaluation
//   f_T = (dlnS/dT) V0 + (1/(2T)) D_beta + (-n/T) D_gamma   and   f_b = D_gamma
// with V0 = Av H, D_beta = beta d sigma/d beta = -Av (H + x H_x + a H_a),
// D_gamma = gamma d sigma/d gamma = Av a H_a.  In the wing forms
//   V0      = Al rho + F1 rho^2 + F2 rho^3,
//   D_beta  = 2 F1 rho^2 + 2 F2 rho^3,
//   D_gamma = Al rho + (F1 - 2 G Al) rho^2 + 6 F2 rho^3 - 6 G F2 rho^4,
// and for K = 2 in addition, with Q = B^2 Al,
//   V0      += Q (3.75 rho^3 - 15 G rho^4 + 12 G^2 rho^5),
//   D_beta  += Q (15 rho^3 - 60 G rho^4 + 48 G^2 rho^5),
//   D_gamma += Q (3.75 rho^3 - 67.5 G rho^4 + 180 G^2 rho^5 - 120 G^3 rho^6).
// A lane first sums Lambda_m v_m^k over the nodes and then applies its line's coefficients
// once.  v = rho for two moments; for more, v = rho D0 with D0 = 1/rho at the line's nearest
// point: it lies in 0.2 .. 1, so the powers stay in range whatever the units, where rho goes as
// 1/nu^2, its sixth power beyond FP32 below 10 cm^-1.  With b = B/D0 = 1/|z|^2 and g = G/D0 <= 1 there, the forms above are
//   V0      = (Al/D0) (v + 1.5 b v^2 - 2 g b v^3 + b^2 (3.75 v^3 - 15 g v^4 + 12 g^2 v^5))
// and so on.

template <int K>
__device__ __forceinline__ void rho_moments(const float2 (&o2)[Far<float>::n / 2], const float2 (&w2)[Far<float>::n / 2],
                                            float nb, float G, float D0, float (&r)[K])
{
    float2 s[K];
#pragma unroll
    for (int k = 0; k < K; ++k) s[k] = dup(0.0f);
    const float2 nb2 = dup(nb), G2 = dup(G), s0 = dup(D0);
#pragma unroll
    for (int p = 0; p < Far<float>::n / 2; ++p) {
        const float2 d = __fadd2_rn(o2[p], nb2);
        float2 v = rcp2_shared(__ffma2_rn(d, d, G2));
        if (K > 2) v = __fmul2_rn(v, s0);
        float2 t = __fmul2_rn(w2[p], v);
#pragma unroll
        for (int k = 0; k < K; ++k) {
            s[k] = __fadd2_rn(s[k], t);
            if (k + 1 < K) t = __fmul2_rn(t, v);
        }
    }
#pragma unroll
    for (int k = 0; k < K; ++k) r[k] = s[k].x + s[k].y;
}

// (sT, sB) = sum over the lines of sum_m Lambda_m (f_T, f_b)(node m), in every lane
__device__ __forceinline__ void far_adjoint_sum(const Lines<float>& ln, const FarList& fl, int t0, int t1,
                                                const Span& sp, float cmin, const float* lam, float hT, double& sT,
                                                double& sB)
{
    constexpr int H = Far<float>::n / 2;
    constexpr NodeTable<Far<float>::n> nt = make_nodes<Far<float>::n>();
    const int lane = threadIdx.x & 31;
    const float h = (float)sp.h, c2min = cmin * cmin;
    float2 o2[H], w2[H];
#pragma unroll
    for (int p = 0; p < H; ++p) {
        o2[p] = make_float2(h * nt.t[2 * p], h * nt.t[2 * p + 1]);
        w2[p] = make_float2(lam[2 * p], lam[2 * p + 1]);
    }
    float Th = 0.f, Tl = 0.f, Bh = 0.f, Bl = 0.f;
    int l = 0;
    float2 nf = make_float2(0.f, 0.f), p3 = nf;
    float4 p1 = make_float4(1.f, 0.f, 0.f, 0.f);
    if (t0 < t1) {
        l = fl.line(min(t0 + lane, t1 - 1));
        nf = ln.nuf[l];
        p1 = ln.r1[l];
        p3 = ((const float2*)ln.r3)[l];
    }
    for (int t = t0; t < t1; t += 32) {
        const bool live = t + lane < t1;
        const float nb = (sp.rh - nf.x) + (sp.rl - nf.y);
        const float G = p1.x, aS = p3.x, nn = p3.y;
        const float Al = live ? p1.y : 0.f, F1 = live ? p1.z : 0.f, F2 = live ? p1.w : 0.f;
        const int lc = l;
        if (t + 32 < t1) {
            l = fl.line(min(t + 32 + lane, t1 - 1));
            nf = ln.nuf[l];
            p1 = ln.r1[l];
            p3 = ((const float2*)ln.r3)[l];
        }
        const float dist = fmaxf(fabsf(nb) - h, 0.0f);
        const float D0 = fmaf(dist, dist, G), z2 = D0 * c2min;
        float V0, Db, Dg;
        if (__all_sync(0xffffffffu, z2 >= WING1_Z2)) {
            // the F2 terms are up to 12 a^2/|z|^4 of f_b's leading one
            if (__all_sync(0xffffffffu, 12.0f * G <= 2.0e-8f * z2 * D0)) {
                float r[2]; // of rho itself: its square stays in range
                rho_moments<2>(o2, w2, nb, G, D0, r);
                V0 = fmaf(F1, r[1], Al * r[0]);
                Db = 2.0f * F1 * r[1];
                Dg = fmaf(F1 - 2.0f * G * Al, r[1], Al * r[0]);
            } else {
                float r[4];
                rho_moments<4>(o2, w2, nb, G, D0, r);
                const float iD = rcp_fast(D0), A0 = Al * iD, g = G * iD;
                const float b1 = F1 * iD * iD, b2 = F2 * iD * iD * iD, u2 = b1 - 2.0f * g * A0;
                V0 = fmaf(b2, r[2], fmaf(b1, r[1], A0 * r[0]));
                Db = 2.0f * fmaf(b2, r[2], b1 * r[1]);
                Dg = fmaf(-6.0f * g * b2, r[3], fmaf(6.0f * b2, r[2], fmaf(u2, r[1], A0 * r[0])));
            }
        } else {
            const float4 p2 = ln.r2[lc];
            if (__all_sync(0xffffffffu, z2 >= WING2_Z2) || p2.y >= WIDE_A) {
                float r[6];
                rho_moments<6>(o2, w2, nb, G, D0, r);
                const float iD = rcp_fast(D0), A0 = Al * iD, g = G * iD;
                const float b = rcp_fast(D0 * (p2.x * p2.x)), g4 = g * r[3], g5 = g * g * r[4], g6 = g * g * g * r[5];
                const float q0 = fmaf(1.5f, r[1], -2.0f * g * r[2]), q = fmaf(3.75f, r[2], fmaf(-15.0f, g4, 12.0f * g5));
                V0 = A0 * fmaf(b, fmaf(b, q, q0), r[0]);
                Db = A0 * b * fmaf(4.0f * b, q, 2.0f * q0);
                Dg = A0 * fmaf(b, fmaf(b, 3.75f * r[2] - 67.5f * g4 + 180.0f * g5 - 120.0f * g6,
                                       1.5f * r[1] - 12.0f * g * r[2] + 12.0f * g * g4),
                               fmaf(-2.0f * g, r[1], r[0]));
            } else {
                // moments of u v^n, u = 1/|z|^2, v = ASY_S u, against the K = 6 coefficients
                float2 s[ASY_N + 1];
#pragma unroll
                for (int k = 0; k <= ASY_N; ++k) s[k] = dup(0.0f);
                const float2 c2 = dup(p2.x), aa = dup(p2.y * p2.y), nb2 = dup(nb);
#pragma unroll
                for (int p = 0; p < H; ++p) {
                    const float2 x = __fmul2_rn(__fadd2_rn(o2[p], nb2), c2);
                    const float2 u = rcp2_shared(__ffma2_rn(x, x, aa));
                    const float2 v = __fmul2_rn(u, dup(ASY_S));
                    float2 q = __fmul2_rn(w2[p], u);
#pragma unroll
                    for (int k = 0; k <= ASY_N; ++k) {
                        s[k] = __fadd2_rn(s[k], q);
                        if (k < ASY_N) q = __fmul2_rn(q, v);
                    }
                }
                float F[ASY_N + 1], Gc[ASY_N + 1];
                asy_coeffs_adj(p2.y, live ? p2.z : 0.0f, aS, hT, nn, F, Gc);
                float ft = 0.0f, fb = 0.0f;
#pragma unroll
                for (int k = 0; k <= ASY_N; ++k) {
                    const float r = s[k].x + s[k].y;
                    ft = fmaf(F[k], r, ft);
                    fb = fmaf(Gc[k], r, fb);
                }
                two_sum(Th, Tl, ft);
                two_sum(Bh, Bl, fb);
                continue;
            }
        }
        two_sum(Th, Tl, aS * V0 + hT * Db + nn * Dg);
        two_sum(Bh, Bl, Dg);
    }
    sT = to_double(warp_sum(Pair{Th, Tl}));
    sB = to_double(warp_sum(Pair{Bh, Bl}));
}

// ------------------------------------------------------------------ far lines, FP64

// The wing polynomials in u = 1/|z|^2 (asy64_coeffs) with the fewest terms that all 32
// lines of a warp allow: about 20 operations a line and node at |z| >= 150 (the generic
// tiers with their divisions took 60 and more).  Each class ends where its first dropped
// term times 2K + 3 (the derivative's) is 2e-16 or less.  With K = 4 and 7 beside 3, 5 and
// 12 a retrieval step of 60 layers and 3,500 lines takes 20.8 ms instead of 21.8 and one layer 270
// us instead of 274; the errors against 64 bits are the same.
template <class F>
__device__ __forceinline__ void by_terms64(double z2, F f)
{
    if (__all_sync(0xffffffffu, z2 >= Tier<double>::z2_far)) f(std::integral_constant<int, 3>{});
    else if (__all_sync(0xffffffffu, z2 >= Tier<double>::z2_k4)) f(std::integral_constant<int, 4>{});
    else if (__all_sync(0xffffffffu, z2 >= Tier<double>::z2_mid)) f(std::integral_constant<int, 5>{});
    else if (__all_sync(0xffffffffu, z2 >= Tier<double>::z2_k7)) f(std::integral_constant<int, 7>{});
    else f(std::integral_constant<int, ASY64_K>{});
}

template <int K>
__device__ __forceinline__ void far_nodes64(double nb, double h, const double4_32a& p2, double amp,
                                            double (&v)[Far<double>::n])
{
    double C[2 * K + 1];
    asy64_coeffs<K>(p2.y, amp, C);
    const double a2 = p2.y * p2.y;
#pragma unroll
    for (int m = 0; m < Far<double>::n; ++m) {
        const double x = fma(h, cheb<Far<double>::n>(1, m), nb) * p2.x;
        const double u = rcp64(fma(x, x, a2));
        double p = C[2 * K];
#pragma unroll
        for (int n = 2 * K - 1; n >= 0; --n) p = fma(p, u, C[n]);
        v[m] = fma(p, u, v[m]);
    }
}

// |z|^2 of a line's nearest point of an interval
__device__ __forceinline__ double nearest_z2(double nb, double h, const double4_32a& p2)
{
    const double x = fmax(fabs(nb) - h, 0.0) * p2.x;
    return fma(x, x, p2.y * p2.y);
}

__device__ __forceinline__ double far_sum(const Lines<double>& ln, const FarList& fl, int t0, int t1, const Span& sp,
                                          float, int& idx)
{
    constexpr int n = Far<double>::n;
    const int lane = threadIdx.x & 31;
    double v[n];
#pragma unroll
    for (int m = 0; m < n; ++m) v[m] = 0.0;
    for (int t = t0; t < t1; t += 32) {
        const int l = fl.line(min(t + lane, t1 - 1));
        const double nb = sp.mid - ln.nu_hat[l];
        const double4_32a p2 = ln.r2[l];
        const double amp = t + lane < t1 ? p2.z : 0.0, z2 = nearest_z2(nb, sp.h, p2);
        by_terms64(z2, [&](auto K) { far_nodes64<decltype(K)::value>(nb, sp.h, p2, amp, v); });
    }
    return warp_reduce_scatter(v, idx);
}

// f_T and f_b from a line's V0, D_beta and D_gamma sums
__device__ __forceinline__ void add_adjoint(double V0, double Db, double Dg, double aS, double hT, double nn, double& sT,
                                            double& sB)
{
    sT += fma(aS, V0, fma(hT, Db, nn * Dg));
    sB += Dg;
}

template <int K>
__device__ __forceinline__ void far_adjoint64(double nb, double h, const double4_32a& p2, double amp, const double* lam,
                                              double aS, double hT, double nn, double& sT, double& sB)
{
    double r[2 * K + 2];
#pragma unroll
    for (int k = 0; k < 2 * K + 2; ++k) r[k] = 0.0;
    const double a2 = p2.y * p2.y;
#pragma unroll 2
    for (int m = 0; m < Far<double>::n; ++m) {
        const double x = fma(h, cheb<Far<double>::n>(1, m), nb) * p2.x;
        const double u = rcp64(fma(x, x, a2));
        double q = lam[m] * u;
#pragma unroll
        for (int k = 0; k < 2 * K + 2; ++k) {
            r[k] += q;
            q *= u;
        }
    }
    double V0, Db, Dg;
    asy64_adjoint<K>(p2.y, amp, r, &V0, &Db, &Dg);
    add_adjoint(V0, Db, Dg, aS, hT, nn, sT, sB);
}

__device__ __forceinline__ void far_adjoint_sum(const Lines<double>& ln, const FarList& fl, int t0, int t1,
                                                const Span& sp, float, const double* lam, double hT, double& sT,
                                                double& sB)
{
    const int lane = threadIdx.x & 31;
    sT = sB = 0.0;
    for (int t = t0; t < t1; t += 32) {
        const int l = fl.line(min(t + lane, t1 - 1));
        const double nb = sp.mid - ln.nu_hat[l];
        const double4_32a p2 = ln.r2[l];
        const double aS = ln.r3[2 * (size_t)l], nn = ln.r3[2 * (size_t)l + 1];
        const double amp = t + lane < t1 ? p2.z : 0.0, z2 = nearest_z2(nb, sp.h, p2);
        by_terms64(z2, [&](auto K) { far_adjoint64<decltype(K)::value>(nb, sp.h, p2, amp, lam, aS, hT, nn, sT, sB); });
    }
    sT = warp_sum(sT);
    sB = warp_sum(sB);
}

// ------------------------------------------------------------------ far kernels

__device__ __forceinline__ bool far_task(const Tree& tr, const FarWork& fw, int* level, int* i, int* part)
{
    int k = 0;
    while (k < tr.top && (int)blockIdx.x < fw.block0[k]) ++k;
    const int r = blockIdx.x - fw.block0[k];
    *level = k;
    *part = r % fw.parts[k];
    *i = (r / fw.parts[k]) * FAR_WARPS + (threadIdx.x >> 5);
    return *i < tr.cnt[k];
}

// this part's share of a list, in whole chunks of 32
__device__ __forceinline__ void part_range(int total, int part, int parts, int* t0, int* t1)
{
    const int64_t chunks = ((int64_t)total + 31) / 32, per = (chunks + parts - 1) / parts;
    *t0 = (int)min64(total, 32 * per * part);
    *t1 = (int)min64(total, 32 * per * (part + 1));
}

template <class R>
__device__ __forceinline__ Lines<R> layer_lines(Lines<R> ln, int64_t nl, int nloc)
{
    const size_t lay = (size_t)nloc * nl;
    ln.r1 += lay;
    ln.r2 += lay;
    ln.r3 += 2 * lay;
    if (ln.clo) ln.clo += lay;
    return ln;
}

// Blocks on an SM that the far adjoint's registers have to leave room for (102 and 128 a
// thread): unbounded the FP32 one takes 123 and is 17% slower (16 warps an SM, not 20).
template <class R> struct FarBlocks { static constexpr int v = 10; };
template <> struct FarBlocks<double> { static constexpr int v = 8; };

template <class R>
__global__ void __launch_bounds__(32 * FAR_WARPS) far_sum_kernel(const __grid_constant__ Batch<R> batch,
                                                                 const double* __restrict__ nu, int layer0)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    if ((int)blockIdx.x >= sp.far_blocks) return;
    const Tree& tr = sp.tree;
    const FarWork& fw = sp.fw;
    const int64_t nl = sp.nl;
    constexpr int n = Far<R>::n;
    int k, i, part;
    if (!far_task(tr, fw, &k, &i, &part)) return;
    const int nloc = blockIdx.y;
    const Lines<R> ln = layer_lines(sp.ln, nl, nloc);
    const FarSet fs = far_set(tr, k, i, nloc);
    const FarList fl(fs);
    int t0, t1;
    part_range(fl.total, part, fw.parts[k], &t0, &t1);
    if (!XS_CHECK(fs.in_order(nl))) t0 = t1 = 0;
    int idx;
    const double s = far_sum(ln, fl, t0, t1, Span(tr.geo[tr.off[k] + i], nu[0]), sp.agg[4 * (layer0 + nloc)],
                             idx);
    const size_t row = fw.out0[k] + ((size_t)part * gridDim.y + nloc) * tr.cnt[k] + i;
    if (idx >= 0 && XS_CHECK(idx < n && row < fw.rows)) sp.sums[row * n + idx] = s;
}

template <class R>
__global__ void __launch_bounds__(32 * FAR_WARPS, FarBlocks<R>::v)
    far_adjoint_kernel(const __grid_constant__ Batch<R> batch, const double* __restrict__ nu, int layer0,
                       const double* __restrict__ T)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    if ((int)blockIdx.x >= sp.far_blocks) return;
    const Tree& tr = sp.tree;
    const FarWork& fw = sp.fw;
    const int64_t nl = sp.nl;
    constexpr int n = Far<R>::n;
    int k, i, part;
    if (!far_task(tr, fw, &k, &i, &part)) return;
    const int nloc = blockIdx.y, layer = layer0 + nloc;
    const Lines<R> ln = layer_lines(sp.ln, nl, nloc);
    const FarSet fs = far_set(tr, k, i, nloc);
    const FarList fl(fs);
    int t0, t1;
    part_range(fl.total, part, fw.parts[k], &t0, &t1);
    if (!XS_CHECK(fs.in_order(nl))) t0 = t1 = 0;
    double sT, sB;
    far_adjoint_sum(ln, fl, t0, t1, Span(tr.geo[tr.off[k] + i], nu[0]), sp.agg[4 * layer],
                    sp.wts + ((size_t)nloc * tr.total + tr.off[k] + i) * n,
                    (R)(0.5 / T[layer]), sT, sB);
    if ((threadIdx.x & 31) == 0) {
        const size_t o = (size_t)nloc * fw.slots + fw.slot0[k] + (size_t)part * tr.cnt[k] + i;
        if (XS_CHECK(o < (size_t)gridDim.y * fw.slots)) {
            sp.slots[2 * o] = sT;
            sp.slots[2 * o + 1] = sB;
        }
    }
}

// x of a position in an interval, -1 .. 1
__device__ __forceinline__ double in_span(double v, const Geo& g) { return (v - g.mid) * g.inv; }

// the same of a child's node t, from the distance of the middles, which is exact: the
// position itself rounds to an ulp of nu, 1e-12 of a narrow interval, and cost FP64 sums
// up to 3e-13 of relative error (1e-14 so)
__device__ __forceinline__ double node_in_span(const Geo& child, double t, const Geo& g)
{
    return fma(child.h, t, child.mid - g.mid) * g.inv;
}

// coefficient k of the polynomial through the node values v
template <int n>
__device__ __forceinline__ double cheb_coeff(const double* v, int k)
{
    double s = 0.0;
#pragma unroll
    for (int m = 0; m < n; ++m) s = fma(v[m], cheb<n>(k, m), s);
    return s * (k ? 2.0 / n : 1.0 / n);
}

// sum_k c_k T_k(x) (Clenshaw)
template <int n, class R>
__device__ __forceinline__ R clenshaw(const R* c, R x)
{
    R b1 = R(0), b2 = R(0);
    const R x2 = x + x;
#pragma unroll
    for (int k = n - 1; k >= 1; --k) {
        const R b = x2 * b1 + (c[k] - b2);
        b2 = b1;
        b1 = b;
    }
    return x * b1 + (c[0] - b2);
}

// A leaf's polynomial: n doubles, or in the FP32 path the constant term, which dominates,
// in FP64 and the others in FP32, in half the space.
template <class R>
struct LeafPoly {
    static constexpr int n = Far<R>::n, stride = n;
    __device__ static void store(double* coef, size_t leaf, int k, double c) { coef[leaf * stride + k] = c; }
    __device__ static double eval(const double* coef, size_t leaf, double x)
    {
        return clenshaw<n, double>(coef + leaf * stride, x);
    }
};
template <>
struct LeafPoly<float> {
    static constexpr int n = Far<float>::n, stride = 1 + n / 2;
    __device__ static void store(double* coef, size_t leaf, int k, double c)
    {
        double* p = coef + leaf * stride;
        if (k == 0) p[0] = c;
        else ((float*)(p + 1))[k] = (float)c;
    }
    __device__ static double eval(const double* coef, size_t leaf, double x)
    {
        const double* p = coef + leaf * stride;
        float c[n];
        c[0] = 0.0f;
#pragma unroll
        for (int k = 1; k < n; ++k) c[k] = ((const float*)(p + 1))[k];
        return p[0] + (double)clenshaw<n, float>(c, (float)x);
    }
};

// Polynomials of the leaves: the node sums of each level plus the polynomial of the
// interval above, from the top interval down.  A block takes 2^root_log leaves and repeats
// the chain of intervals above them: root_log = 6 (64 leaves, nothing repeated) where that
// makes enough blocks to fill the chip, smaller subtrees otherwise.
template <class R> struct DownRows { static constexpr int v = 64; }; // intervals of a level that a block takes at a time
template <> struct DownRows<double> { static constexpr int v = 32; };
template <class R>
__global__ void __launch_bounds__(DownRows<R>::v * Far<R>::n) down_kernel(const __grid_constant__ Batch<R> batch, int Lc,
                                                                     int root_log)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    const Tree& tr = sp.tree;
    const FarWork& fw = sp.fw;
    constexpr int n = Far<R>::n;
    __shared__ double v[DownRows<R>::v][n], c[2][TOP / 2][n];
    const int m = threadIdx.x % n, row = threadIdx.x / n, rows = blockDim.x / n;
    const int nloc = blockIdx.y;
    for (int k = tr.top; k >= 0; --k) {
        const int below = root_log - tr.shift * k;
        const int many = 1 << max(below, 0); // intervals of this level
        const int first = below <= 0 ? blockIdx.x >> -below : blockIdx.x * many;
        for (int q0 = 0; q0 < many; q0 += rows) {
            const int q = q0 + row, i = first + q;
            const bool mine = q < many && i < tr.cnt[k] && XS_CHECK(i >= 0 && row < DownRows<R>::v && (k == 0 || q < TOP / 2));
            if (mine) {
                double s = 0.0;
                for (int p = 0; p < fw.parts[k]; ++p) {
                    const size_t at = fw.out0[k] + ((size_t)p * Lc + nloc) * tr.cnt[k] + i;
                    if (XS_CHECK(at < fw.rows)) s += sp.sums[at * n + m];
                }
                if (k < tr.top) {
                    const Geo g = tr.geo[tr.off[k] + i], gp = tr.geo[tr.off[k + 1] + (i >> tr.shift)];
                    s += clenshaw<n, double>(c[(k + 1) & 1][q >> tr.shift], node_in_span(g, cheb<n>(1, m), gp));
                }
                v[row][m] = s;
            }
            __syncthreads();
            if (mine) {
                const double ck = cheb_coeff<n>(v[row], m);
                if (k > 0)
                    c[k & 1][q][m] = ck;
                else
                    LeafPoly<R>::store(sp.coef, (size_t)nloc * tr.cnt[0] + i, m, ck);
            }
            __syncthreads();
        }
    }
}

// A weight's products and sums on the way up: FP64, or float pairs in the FP32 path.  In plain
// FP32 the roundings of the levels add up to three times that of lambda itself: g_b of weights
// of mixed sign at 4 to 100 cm^-1 is off by 3.2e-9 to 3.5e-9 of what weights of one sign give,
// 0.7e-9 to 1.9e-9 with pairs (1.1e-9 to 3.1e-9 with every line evaluated at every point).  One
// layer's adjoint takes 80 us in plain FP32, 84 with pairs, 119 with FP64; 220,000 lines x 20
// layers 3.71, 3.72 and 3.82 ms.
template <class R> struct UpSum { using type = double; };
template <> struct UpSum<float> { using type = Pair; };
__device__ __forceinline__ Pair times(const Pair& w, float t)
{
    const float p = w.hi * t;
    return {p, fmaf(w.lo, t, fmaf(w.hi, t, -p))};
}
__device__ __forceinline__ double times(double w, double t) { return w * t; }
__device__ __forceinline__ Pair up_weight(double v, float) { return {(float)v, 0.0f}; }
__device__ __forceinline__ double up_weight(double v, double) { return v; }
__device__ __forceinline__ float rounded(const Pair& v) { return v.hi + v.lo; }
__device__ __forceinline__ double rounded(double v) { return v; }

// moments sum w T_k(x) of a weight at x, added to s
template <int n>
__device__ __forceinline__ void add_moments(double w, double x, double (&s)[n])
{
    double a = w, b = w * x;
    const double x2 = x + x;
    s[0] += a;
    s[1] += b;
#pragma unroll
    for (int k = 2; k < n; ++k) {
        const double t = x2 * b - a;
        s[k] += t;
        a = b;
        b = t;
    }
}
template <int n>
__device__ __forceinline__ void add_moments(const Pair& w, float x, Pair (&s)[n])
{
    float a = 1.0f, b = x;
    const float x2 = x + x;
    s[0] = add(s[0], w);
#pragma unroll
    for (int k = 1; k < n; ++k) {
        s[k] = add(s[k], times(w, b));
        const float t = fmaf(x2, b, -a);
        a = b;
        b = t;
    }
}

// node weight m from the moments M: sum_k (1 or 2)/n M_k T_k(t_m)
template <int n>
__device__ __forceinline__ double node_weight(const double* M, int m)
{
    double s = 0.5 * M[0];
#pragma unroll
    for (int k = 1; k < n; ++k) s += M[k] * cheb_r(0.0, k, m);
    return s * (2.0 / n);
}
template <int n>
__device__ __forceinline__ Pair node_weight(const Pair* M, int m)
{
    Pair s = {0.5f * M[0].hi, 0.5f * M[0].lo};
#pragma unroll
    for (int k = 1; k < n; ++k) s = add(s, times(M[k], cheb_r(0.0f, k, m)));
    constexpr float c = (float)(2.0 / n), cl = (float)(2.0 / n - (double)c);
    Pair r = times(s, c);
    r.lo = fmaf(s.hi, cl, r.lo);
    return r;
}

// Node weights of all intervals: per layer and top interval, one warp per leaf takes its
// points, then the larger intervals take the nodes of those below (whose weights
// reproduce every polynomial of the degree kept).  In the FP32 path lambda is rounded once and
// the sums are float pairs (UpSum); the weights are stored in FP32.  weights[layer][interval][n].
constexpr int UP_WARPS = 16;
template <class R>
__global__ void __launch_bounds__(32 * UP_WARPS) up_kernel(const __grid_constant__ Batch<R> batch,
                                                           const double* __restrict__ nu, int64_t N, int layer0,
                                                           double lam_scale)
{
    using A = typename UpSum<R>::type;
    const Species<R>& spc = batch.s[blockIdx.z];
    const Tree& tr = spc.tree;
    constexpr int n = Far<R>::n;
    __shared__ A M[UP_WARPS][n], w[2][TOP][n];
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int nloc = blockIdx.y, top = blockIdx.x;
    const double* g = spc.g_sigma + (size_t)(layer0 + nloc) * N;
    for (int k = 0; k <= tr.top; ++k) {
        const int many = 1 << (tr.shift * (tr.top - k)), below = 1 << tr.shift;
        for (int q = row; q < many; q += UP_WARPS) {
            const int i = top * many + q;
            if (i >= tr.cnt[k] || !XS_CHECK(q < TOP)) break;
            const Geo sp = tr.geo[tr.off[k] + i];
            A s[n];
#pragma unroll
            for (int m = 0; m < n; ++m) s[m] = A{};
            if (k == 0) {
                const int64_t j = (int64_t)i * LEAF + lane;
                if (j < N) add_moments<n>(up_weight(g[j] * lam_scale, R(0)), (R)in_span(nu[j], sp), s);
            } else {
#pragma unroll 1
                for (int r = lane; r < below * n; r += 32) {
                    const int ch = below * i + r / n, m = r % n; // child interval and its node
                    if (ch >= tr.cnt[k - 1]) break;
                    const Geo gc = tr.geo[tr.off[k - 1] + ch];
                    add_moments<n>(w[(k - 1) & 1][below * q + r / n][m], (R)node_in_span(gc, cheb<n>(1, m), sp), s);
                }
            }
            __syncwarp();
            int idx;
            const A v = warp_reduce_scatter(s, idx);
            if (idx >= 0 && XS_CHECK(idx < n)) M[row][idx] = v;
            __syncwarp();
            if (lane < n) {
                const A x = node_weight<n>(M[row], lane);
                w[k & 1][q][lane] = x;
                spc.wts[((size_t)nloc * tr.total + tr.off[k] + i) * n + lane] = rounded(x);
            }
            __syncwarp();
        }
        __syncthreads();
    }
}

// u sum_{n<13} C'_n v^n, v = ASY_S u, by Horner from four float4 of coefficients
__device__ __forceinline__ float horner13(const float4* h, float u)
{
    const float v = ASY_S * u;
    const float4 h0 = h[0], h1 = h[1], h2 = h[2], h3 = h[3];
    float p = h3.x;
    p = fmaf(p, v, h2.w);
    p = fmaf(p, v, h2.z);
    p = fmaf(p, v, h2.y);
    p = fmaf(p, v, h2.x);
    p = fmaf(p, v, h1.w);
    p = fmaf(p, v, h1.z);
    p = fmaf(p, v, h1.y);
    p = fmaf(p, v, h1.x);
    p = fmaf(p, v, h0.w);
    p = fmaf(p, v, h0.z);
    p = fmaf(p, v, h0.y);
    p = fmaf(p, v, h0.x);
    return p * u;
}
// u sum_{n<14} F_n v^n
__device__ __forceinline__ float horner14(const float4* h, float u)
{
    const float v = ASY_S * u;
    const float4 h0 = h[0], h1 = h[1], h2 = h[2], h3 = h[3];
    float p = h3.y;
    p = fmaf(p, v, h3.x);
    p = fmaf(p, v, h2.w);
    p = fmaf(p, v, h2.z);
    p = fmaf(p, v, h2.y);
    p = fmaf(p, v, h2.x);
    p = fmaf(p, v, h1.w);
    p = fmaf(p, v, h1.z);
    p = fmaf(p, v, h1.y);
    p = fmaf(p, v, h1.x);
    p = fmaf(p, v, h0.w);
    p = fmaf(p, v, h0.z);
    p = fmaf(p, v, h0.y);
    p = fmaf(p, v, h0.x);
    return p * u;
}

__device__ __forceinline__ void store16(float4* dst, const float* v, int n)
{
#pragma unroll
    for (int q = 0; q < 4; ++q)
        dst[q] = make_float4(4 * q < n ? v[4 * q] : 0.0f, 4 * q + 1 < n ? v[4 * q + 1] : 0.0f,
                             4 * q + 2 < n ? v[4 * q + 2] : 0.0f, 4 * q + 3 < n ? v[4 * q + 3] : 0.0f);
}

// ------------------------------------------------------------------ leaves

// Near-line tiles of a leaf's warp: 32 lines staged for its 32 points, offsets to the
// leaf's middle as hi + lo floats (their sum keeps the relative accuracy of a small
// distance in a wide leaf).
struct NearTile {
    float4 nb[32]; // middle of the leaf - centre (hi, lo), the part of c that r2.x misses, 1/a
    float4 r2[32]; // c, a, Av, Kc
    int2 jr[32];
    float4 hc[32][4];      // Av C'_0 .. Av C'_12 of the wing polynomial (6 <= |z|), or the wing form's constants
    float sd[32][SER_TAB]; // series table (|z| < 6, lines with a < 6)
};
struct NearAdjTile {
    float4 nb[32];
    float4 r2[32];
    int2 jr[32];
    float aS[32], nn[32];
    float4 hf[32][4], hg[32][4]; // f_T and f_b wing polynomials (6 <= |z|)
    float sd[32][SER_TAB];
};
// FP64: 16 lines at a time.
constexpr int NEAR64 = 16;
struct NearTile64 {
    double cen[NEAR64];
    double4_32a r2[NEAR64]; // c, a, Av, Kc
    double ia[NEAR64];      // 1/a
    int2 jr[NEAR64];
    double C[NEAR64][2 * ASY64_K + 1];
    double sd[NEAR64][SER64_TAB];
};
struct NearAdjTile64 {
    double pos[LEAF], lam[LEAF]; // the leaf's points
    double cen[NEAR64];
    double4_32a r2[NEAR64];
    double ia[NEAR64], aS[NEAR64], nn[NEAR64];
    int2 jr[NEAR64];
    double sd[NEAR64][SER64_TAB];
};

// |z|^2 from which the near lines take the wing polynomial in u = 1/|z|^2;
// below it the series.
constexpr float NEAR_POLY_Z2 = 36.0f;

__device__ __forceinline__ bool in_range(int j, int2 r) { return j >= r.x && j <= r.y; }

// zero for the lines of a group of four that do not reach point j
__device__ __forceinline__ void mask4(const int2* jr, int j, float2& a, float2& b)
{
    a.x = in_range(j, jr[0]) ? a.x : 0.0f;
    a.y = in_range(j, jr[1]) ? a.y : 0.0f;
    b.x = in_range(j, jr[2]) ? b.x : 0.0f;
    b.y = in_range(j, jr[3]) ? b.y : 0.0f;
}

// A warp's leaf: its points and its near lines as up to five ranges (the first and last masked
// per point, the others inside every line's cut).  `split` neighbouring warps of `slices`
// blocks share a leaf and take its chunks of lines in turn.
constexpr int RANGES = 5;
// |z|^2 from which short forms hold: without far sets the lines nearer than it are a range
// of their own, so that few chunks mix them with others.  A window of fewer lines than
// SPLIT_LINES stays one masked range: each range ends in a chunk that is not full (128 lines on
// 50,000 points x 100 layers 567 us split, 627 not; 64 lines 622 and 480).
constexpr int SPLIT_LINES = 96;

// first index of v[0], v[stride], .. that holds at least x
template <class V>
__device__ __forceinline__ int first_index(const V* v, int stride, int64_t n, V x)
{
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        if (v[stride * m] >= x) hi = m; else lo = m + 1;
    }
    return (int)lo;
}
// the centres, FP32: relative to the first grid point (no digits are needed here)
__device__ __forceinline__ const float* near_keys(const Lines<float>& ln) { return (const float*)ln.nuf; }
__device__ __forceinline__ const double* near_keys(const Lines<double>& ln) { return ln.nu_hat; }
__device__ __forceinline__ int near_stride(const Lines<float>&) { return 2; }
__device__ __forceinline__ int near_stride(const Lines<double>&) { return 1; }
__device__ __forceinline__ float near_key(const Lines<float>&, double mid, double nu0, float r) { return (float)(mid - nu0) + r; }
__device__ __forceinline__ double near_key(const Lines<double>&, double mid, double, float r) { return mid + r; }
template <class R> struct ShortForm { static constexpr double z2 = WING2_Z2; };
template <> struct ShortForm<double> { static constexpr double z2 = Tier<double>::z2_k7; };
template <class R>
struct Leaf {
    int64_t jb, jl;
    int lane, i, sub, slice;
    bool any, live; // the leaf has points; the lane has one
    int s[RANGES], e[RANGES];
    Geo g;

    __device__ void init(const Tree& tr, const Lines<R>& ln, const float* agg, int64_t nl, const double* nu, int64_t N,
                         int nloc, int split, int slices)
    {
        const int w = threadIdx.x >> 5;
        lane = threadIdx.x & 31;
        int block = blockIdx.x;
        slice = 0;
        if (slices > 1) {
            block /= slices;
            slice = blockIdx.x - block * slices;
        }
        i = (block * (int)(blockDim.x >> 5) + w) / split;
        sub = slice * split + w % split;
        jb = (int64_t)i * LEAF;
        jl = min64(N - 1, jb + LEAF - 1);
        any = jb < N;
        g = {0.0, 0.0, 0.0};
        live = any && jb + lane <= jl;
#pragma unroll
        for (int k = 0; k < RANGES; ++k) s[k] = e[k] = 0;
        if (!any) return;
        if (tr.on) {
            g = tr.geo[i];
            const FarSet fs = far_set(tr, 0, i, nloc);
            const int2 w = tr.win[i];
            s[0] = w.x;
            e[0] = fs.a;
            s[2] = fs.p;
            e[2] = fs.q;
            s[4] = fs.b;
            e[4] = w.y;
        } else {
            // no far sets: the lines that cover the leaf, around the near ones, and on each
            // side those cut inside it.  A lane a search, in whole numbers (an FP64 operation
            // of a warp takes the SM's FP64 pipe for 16 clocks).
            const double v0 = nu[jb], v1 = nu[jl];
            g = {0.5 * (v0 + v1), 0.5 * (v1 - v0), 0.0};
            const int upper = lane == 0 || lane == 3; // jr.y >= jb, jr.x > jl, jr.x > jb, jr.y >= jl
            const int f = first_index((const int*)ln.jr + upper, 2, nl, (int)(lane & 1 ? jl : jb) + !upper);
            s[0] = __shfl_sync(0xffffffffu, f, 0);
            e[4] = __shfl_sync(0xffffffffu, f, 1);
            if (e[4] - s[0] < SPLIT_LINES) {
                e[0] = s[4] = e[4];
            } else {
                const float a2 = agg[1] * agg[1], z2 = ShortForm<R>::z2;
                const float r = a2 < z2 ? (float)g.h + sqrtf(z2 - a2) * rcp_fast(agg[0]) : 0.0f;
                const R v = near_key(ln, g.mid, nu[0], lane & 1 ? r : -r);
                const int n = first_index(near_keys(ln), near_stride(ln), nl, v);
                e[0] = s[1] = __shfl_sync(0xffffffffu, f, 3);
                e[3] = s[4] = max(e[0], __shfl_sync(0xffffffffu, f, 2));
                e[1] = s[2] = clampi(__shfl_sync(0xffffffffu, n, 0), s[1], e[3]);
                e[2] = s[3] = clampi(__shfl_sync(0xffffffffu, n, 1), s[2], e[3]);
            }
        }
#pragma unroll
        for (int k = 0; k < RANGES; ++k)
            if (!XS_CHECK(s[k] >= 0 && e[k] <= nl)) e[k] = s[k];
    }
};

// sum of v over the warps that share a leaf, valid in the first of them (fixed order)
template <int warps>
__device__ __forceinline__ double split_sum(double v, int split)
{
    __shared__ double part[warps][LEAF];
    if (split == 1) return v;
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    part[w][lane] = v;
    __syncthreads();
    double s = 0.0;
    if (w % split == 0)
        for (int q = 0; q < split; ++q) s += part[w + q][lane];
    return s;
}

// sigma of one leaf: FP32
__global__ void __launch_bounds__(32 * LeafWarps<float>::v) leaf_kernel_f32(const __grid_constant__ Batch<float> batch,
                                                                           const double* __restrict__ nu, int64_t N,
                                                                           int layer0, double unscale,
                                                                           int split, int slices, int stride)
{
    const Species<float>& sp = batch.s[blockIdx.z];
    const Tree& tr = sp.tree;
    const int64_t nl = sp.nl;
    float* __restrict__ sigma = (float*)sp.sigma;
    __shared__ NearTile tiles[LeafWarps<float>::v];
    NearTile& tl = tiles[threadIdx.x >> 5];
    const int nloc = blockIdx.y, layer = layer0 + nloc;
    Leaf<float> lf;
    lf.init(tr, sp.ln, sp.agg + 4 * layer, nl, nu, N, nloc, split, slices);
    const Lines<float> ln = layer_lines(sp.ln, nl, nloc);
    const int lane = lf.lane;
    const int64_t j = min64(lf.jb + lane, N - 1);
    const double nuj = nu[j];
    const Span span(lf.g, nu[0]);
    const float rh = span.rh, rl = span.rl;
    const double oj = nuj - lf.g.mid;
    const float ohi = (float)oj, olo = (float)(oj - (double)ohi), h = (float)lf.g.h;
    float shi = 0.0f, slo = 0.0f;
#pragma unroll 1
    for (int k = 0; k < RANGES; k += tr.on ? 2 : 1) { // without 1 and 3 where there are far sets
        const bool masked = k == 0 || k == RANGES - 1;
        const int ce = lf.e[k];
        for (int t0 = lf.s[k] + 32 * lf.sub; t0 < ce; t0 += stride) {
            const int l = t0 + lane;
            const bool have = l < ce;
            __syncwarp();
            float nb = 0.0f, nbl = 0.0f, z2 = 1e30f;
            float4 p2 = make_float4(1.f, 1.f, 0.f, 0.f);
            if (have) {
                const float2 nf = ln.nuf[l];
                nb = rh - nf.x; // (nb, nbl) = middle - centre, TwoSum of the high parts
                const float bb = nb - rh;
                nbl = ((rh - (nb - bb)) - (nf.x + bb)) + (rl - nf.y);
                p2 = ln.r2[l];
                const float x = fmaxf(fabsf(nb) - h, 0.0f) * p2.x;
                z2 = fmaf(x, x, p2.y * p2.y);
                if (masked) tl.jr[lane] = ln.jr[l];
            }
            const int cnt = min(32, ce - t0);
            float acc = 0.0f;
            if (__all_sync(0xffffffffu, z2 >= WING2_Z2)) {
                // no point closer than |z| = 16.5 to any of the lines: wing forms, a field of
                // the 32 lines a row, so that one load fills two packed pairs of lines (some 7
                // instructions a line and warp, 14 a line at a time)
                const bool k1only = __all_sync(0xffffffffu, z2 >= WING1_Z2);
                float* const f = (float*)tl.hc;
                const float4 p1 = have ? ln.r1[l] : make_float4(1.f, 0.f, 0.f, 0.f);
                f[lane] = nb;
                f[32 + lane] = nbl;
                f[64 + lane] = p1.x;
                f[96 + lane] = p1.y;
                f[128 + lane] = p1.z;
                if (k1only) {
                    f[160 + lane] = p1.w;
                } else {
                    float a2, a3, a4;
                    wing2_consts(p1, p2.x, &a2, &a3, &a4);
                    f[160 + lane] = a2;
                    f[192 + lane] = a3;
                    f[224 + lane] = a4;
                }
                __syncwarp();
                const float4* const r = (const float4*)f;
                float2 a01 = dup(0.0f), a23 = a01;
                for (int q = 0; q < (cnt + 3) / 4; ++q) {
                    const float4 b = r[q], bl = r[8 + q], G = r[16 + q], k0 = r[24 + q], k1 = r[32 + q], k2 = r[40 + q];
                    const float2 d0 = __fadd2_rn(__fadd2_rn(dup(ohi), lo2(b)), __fadd2_rn(dup(olo), lo2(bl)));
                    const float2 d1 = __fadd2_rn(__fadd2_rn(dup(ohi), hi2(b)), __fadd2_rn(dup(olo), hi2(bl)));
                    float2 r0 = rcp2_shared(__ffma2_rn(d0, d0, lo2(G))), r1 = rcp2_shared(__ffma2_rn(d1, d1, hi2(G)));
                    float2 u0 = lo2(k2), u1 = hi2(k2);
                    if (!k1only) {
                        const float4 k3 = r[48 + q], k4 = r[56 + q];
                        u0 = __ffma2_rn(__ffma2_rn(lo2(k4), r0, lo2(k3)), r0, u0);
                        u1 = __ffma2_rn(__ffma2_rn(hi2(k4), r1, hi2(k3)), r1, u1);
                    }
                    u0 = __ffma2_rn(__ffma2_rn(u0, r0, lo2(k1)), r0, lo2(k0));
                    u1 = __ffma2_rn(__ffma2_rn(u1, r1, hi2(k1)), r1, hi2(k0));
                    if (masked) mask4(tl.jr + 4 * q, (int)j, r0, r1);
                    a01 = __ffma2_rn(r0, u0, a01);
                    a23 = __ffma2_rn(r1, u1, a23);
                }
                acc = (a01.x + a01.y) + (a23.x + a23.y);
            } else {
                if (have) {
                    tl.nb[lane] = make_float4(nb, nbl, ln.clo[l], p2.y > 0.0f ? rcp_fast(p2.y) : 0.0f);
                    tl.r2[lane] = p2;
                    const bool wide = p2.y >= WIDE_A; // summed below
                    float C[ASY_N];
                    asy_coeffs(wide ? 0.0f : p2.y, wide ? 0.0f : p2.z, C);
                    store16(tl.hc[lane], C, ASY_N);
                    if (p2.y * p2.y < NEAR_POLY_Z2) series_table(p2.y, tl.sd[lane]);
                }
                unsigned wide = __ballot_sync(0xffffffffu, have && p2.y >= WIDE_A);
                __syncwarp();
                // the staged lines in ascending order (warp-uniform loop)
                for (int q = 0; q < cnt; ++q) {
                    const bool in = lf.live && (!masked || in_range((int)j, tl.jr[q]));
                    // x to FP32 accuracy suffices for the polynomial (a rational
                    // function of x); the series takes the exact pair
                    const float4 c4 = tl.r2[q];
                    const float4 b = tl.nb[q];
                    const float dh = ohi + b.x, dl = olo + b.y;
                    const float xq = c4.x * (dh + dl);
                    const float zz = fmaf(xq, xq, c4.y * c4.y);
                    if (!__any_sync(0xffffffffu, in && zz < NEAR_POLY_Z2)) {
                        // no lane in the series zone: the polynomial, branch-free
                        const float hv = horner13(tl.hc[q], rcp_fast(zz));
                        acc += in ? hv : 0.0f;
                    } else if (in) {
                        // the series also serves the lanes just outside its zone
                        if (!(fabsf(xq) <= SER_X)) {
                            acc += horner13(tl.hc[q], rcp_fast(zz));
                        } else {
                            float x, xl;
                            scaled_pair(dh, dl, c4.x, b.z, &x, &xl);
                            acc = fmaf(c4.z, w_series_re(x, xl, c4.y, b.w, c4.w, tl.sd[q]), acc);
                        }
                    }
                }
                if (wide) {
                    __syncwarp();
                    if (have) tl.hc[lane][0] = ln.r1[l];
                    __syncwarp();
                    for (; wide; wide &= wide - 1) {
                        const int q = __ffs(wide) - 1;
                        const float4 u = tl.hc[q][0], b = tl.nb[q];
                        const float d = (ohi + b.x) + (olo + b.y);
                        const bool in = !masked || in_range((int)j, tl.jr[q]);
                        const float rho = rcp_fast(fmaf(d, d, u.x));
                        acc = fmaf(in ? rho : 0.0f, fmaf(fmaf(u.w, rho, u.z), rho, u.y), acc);
                    }
                }
            }
            two_sum(shi, slo, acc); // the chunk's FP32 partial into the compensated sum
        }
    }
    if (!tr.on && split * slices == 1) { // nothing to add; the scale is a power of two
        if (lf.live) sigma[(size_t)layer * N + j] = (shi + slo) * (float)unscale;
        return;
    }
    const double near = split_sum<LeafWarps<float>::v>((double)shi + (double)slo, split);
    if (!lf.live || lf.sub % split) return;
    if (slices > 1) {
        if (XS_CHECK(lf.slice < slices && j < N)) sp.near[((size_t)lf.slice * gridDim.y + nloc) * N + j] = near;
        return;
    }
    // the far lines' part
    const double far =
        tr.on && XS_CHECK(lf.i < tr.cnt[0]) ? LeafPoly<float>::eval(sp.coef, (size_t)nloc * tr.cnt[0] + lf.i, in_span(nuj, lf.g)) : 0.0;
    sigma[(size_t)layer * N + j] = (float)((far + near) * unscale);
}

template <int K>
__device__ __forceinline__ void stage_poly64(double a, double amp, double* dst)
{
    double C[2 * K + 1];
    asy64_coeffs<K>(a, amp, C);
#pragma unroll
    for (int n = 0; n < 2 * K + 1; ++n) dst[n] = C[n];
}
template <int K>
__device__ __forceinline__ double poly64(const double* C, double z2)
{
    const double u = rcp64(z2);
    double p = C[2 * K];
#pragma unroll
    for (int n = 2 * K - 1; n >= 0; --n) p = fma(p, u, C[n]);
    return p * u;
}

// sum over the staged lines at one point, wing polynomials of one length
template <int K>
__device__ __forceinline__ double near_poly64(const NearTile64& tl, int cnt, double nuj, int j, bool masked)
{
    double acc = 0.0;
    for (int q = 0; q < cnt; ++q) {
        const double4_32a p2 = tl.r2[q];
        const double x = (nuj - tl.cen[q]) * p2.x;
        const double v = poly64<K>(tl.C[q], fma(x, x, p2.y * p2.y));
        acc += (!masked || in_range(j, tl.jr[q])) ? v : 0.0;
    }
    return acc;
}

// sigma of one leaf: FP64.  Bound by FP64 operations: a chunk of 16 lines takes the
// shortest wing polynomial that all of them allow, and the series only its own lanes.
// (2,000 lines, 4,096 points, one layer: this kernel 3.1 ms with the generic tiers and one
// exponential a term of the series.)
__global__ void __launch_bounds__(32 * LeafWarps<double>::v) leaf_kernel_f64(const __grid_constant__ Batch<double> batch,
                                                                           const double* __restrict__ nu, int64_t N,
                                                                           int layer0, double unscale,
                                                                           int split, int slices, int stride)
{
    const Species<double>& sp = batch.s[blockIdx.z];
    const Tree& tr = sp.tree;
    const int64_t nl = sp.nl;
    double* __restrict__ sigma = (double*)sp.sigma;
    extern __shared__ __align__(32) unsigned char smem64[];
    NearTile64& tl = ((NearTile64*)smem64)[threadIdx.x >> 5];
    const int nloc = blockIdx.y, layer = layer0 + nloc;
    Leaf<double> lf;
    lf.init(tr, sp.ln, sp.agg + 4 * layer, nl, nu, N, nloc, split, slices);
    const Lines<double> ln = layer_lines(sp.ln, nl, nloc);
    const int lane = lf.lane;
    const int64_t j = min64(lf.jb + lane, N - 1);
    const double nuj = nu[j];
    double acc = 0.0;
#pragma unroll 1
    for (int k = 0; k < RANGES; k += tr.on ? 2 : 1) { // without 1 and 3 where there are far sets
        const bool masked = k == 0 || k == RANGES - 1;
        const int ce = lf.e[k];
        for (int t0 = lf.s[k] + NEAR64 * lf.sub; t0 < ce; t0 += stride) {
            const int l = t0 + lane;
            const bool have = lane < NEAR64 && l < ce;
            __syncwarp();
            double z2 = 1e300;
            double4_32a p2{};
            if (have) {
                const double c = ln.nu_hat[l];
                p2 = ln.r2[l];
                z2 = nearest_z2(lf.g.mid - c, lf.g.h, p2);
                tl.cen[lane] = c;
                tl.r2[lane] = p2;
                if (masked) tl.jr[lane] = ln.jr[l];
            }
            const int cnt = min(NEAR64, ce - t0);
            if (__all_sync(0xffffffffu, z2 >= Tier<double>::z2_k7)) {
                by_terms64(z2, [&](auto Kc) {
                    constexpr int K = decltype(Kc)::value;
                    if constexpr (K < ASY64_K) {
                        if (have) stage_poly64<K>(p2.y, p2.z, tl.C[lane]);
                        __syncwarp();
                        acc += near_poly64<K>(tl, cnt, nuj, (int)j, masked);
                    }
                });
            } else {
                if (have) stage_poly64<ASY64_K>(p2.y, p2.z, tl.C[lane]);
                if (have && z2 < Tier<double>::z2_stage) {
                    tl.ia[lane] = p2.y > 0.0 ? 1.0 / p2.y : 0.0;
                    series_table64(p2.y, tl.sd[lane]);
                }
                __syncwarp();
                for (int q = 0; q < cnt; ++q) {
                    const bool in = lf.live && (!masked || in_range((int)j, tl.jr[q]));
                    const double4_32a c4 = tl.r2[q];
                    const double x = fabs(nuj - tl.cen[q]) * c4.x, zz = fma(x, x, c4.y * c4.y);
                    if (in) {
                        if (zz < Tier<double>::z2_series)
                            acc = fma(c4.z, w_series_re(x, c4.y, tl.ia[q], c4.w, tl.sd[q]), acc);
                        else
                            acc += poly64<ASY64_K>(tl.C[q], zz);
                    }
                }
            }
        }
    }
    acc = split_sum<LeafWarps<double>::v>(acc, split);
    if (!lf.live || lf.sub % split) return;
    if (slices > 1) {
        if (XS_CHECK(lf.slice < slices && j < N)) sp.near[((size_t)lf.slice * gridDim.y + nloc) * N + j] = acc;
        return;
    }
    if (tr.on && XS_CHECK(lf.i < tr.cnt[0])) acc += LeafPoly<double>::eval(sp.coef, (size_t)nloc * tr.cnt[0] + lf.i, in_span(nuj, lf.g));
    sigma[(size_t)layer * N + j] = acc * unscale;
}

// sigma from the slices' sums over the near lines (in order) and the far lines' polynomials
template <class R>
__global__ void __launch_bounds__(256) slices_kernel(const __grid_constant__ Batch<R> batch, const double* __restrict__ nu,
                                                     int64_t N, int layer0, double unscale, int slices)
{
    const Species<R>& sp = batch.s[blockIdx.z];
    const int nloc = blockIdx.y;
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= N) return;
    double s = 0.0;
    for (int k = 0; k < slices; ++k) s += sp.near[((size_t)k * gridDim.y + nloc) * N + j];
    if (sp.tree.on) {
        const int i = (int)(j / LEAF);
        s += LeafPoly<R>::eval(sp.coef, (size_t)nloc * sp.tree.cnt[0] + i, in_span(nu[j], sp.tree.geo[i]));
    }
    ((R*)sp.sigma)[(size_t)(layer0 + nloc) * N + j] = (R)(s * unscale);
}

// a block's sums of the leaves' (f_T, f_b) to part[layer of the chunk][block], fixed order
template <int warps>
__device__ __forceinline__ void block_pair(double sT, double sB, double* part)
{
    __shared__ double red[2][warps];
    for (int o = 16; o > 0; o >>= 1) {
        sT += __shfl_xor_sync(0xffffffffu, sT, o);
        sB += __shfl_xor_sync(0xffffffffu, sB, o);
    }
    if ((threadIdx.x & 31) == 0) {
        red[0][threadIdx.x >> 5] = sT;
        red[1][threadIdx.x >> 5] = sB;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        for (int i = 0; i < (int)(blockDim.x >> 5); ++i) {
            a += red[0][i];
            b += red[1][i];
        }
        part[0] = a;
        part[1] = b;
    }
}

// A line's K = 1 wing forms of f_T and f_b as polynomials in rho (see far_adjoint_sum):
// hf = {G, f_T's first three coefficients}, {its last, f_b's first two}, hg = {f_b's last two}
__device__ __forceinline__ void stage_wing1_adj(const float4& p1, float aS, float nn, float hT, float4* hf, float4* hg)
{
    const float G = p1.x, Al = p1.y, F1 = p1.z, F2 = p1.w;
    const float U2 = F1 - 2.0f * G * Al, U4 = -6.0f * G * F2;
    hf[0] = make_float4(G, Al * (aS + nn), aS * F1 + hT * 2.0f * F1 + nn * U2, (aS + 2.0f * hT + 6.0f * nn) * F2);
    hf[1] = make_float4(nn * U4, Al, U2, 0.0f);
    hg[0] = make_float4(6.0f * F2, U4, 0.0f, 0.0f);
}
__device__ __forceinline__ void add_wing1_adj(const float4* hf, const float4* hg, float d, bool in, float& aT, float& aB)
{
    const float4 t = hf[0], u = hf[1], v = hg[0];
    const float rho = rcp_fast(fmaf(d, d, t.x)), r = in ? rho : 0.0f;
    aT = fmaf(r, fmaf(fmaf(fmaf(u.x, rho, t.w), rho, t.z), rho, t.y), aT);
    aB = fmaf(r, fmaf(fmaf(fmaf(v.y, rho, v.x), rho, u.z), rho, u.y), aB);
}

__global__ void __launch_bounds__(32 * LeafWarps<float>::v) leaf_adjoint_f32(const __grid_constant__ Batch<float> batch,
                                                                            const double* __restrict__ nu, int64_t N,
                                                                            int layer0,
                                                                            const double* __restrict__ T,
                                                                            double lam_scale, int split, int slices,
                                                                            int stride)
{
    const Species<float>& sp = batch.s[blockIdx.z];
    const Tree& tr = sp.tree;
    const int64_t nl = sp.nl;
    const double* __restrict__ g_sigma = sp.g_sigma;
    __shared__ NearAdjTile tiles[LeafWarps<float>::v];
    NearAdjTile& tl = tiles[threadIdx.x >> 5];
    const int nloc = blockIdx.y, layer = layer0 + nloc;
    double sT = 0.0, sB = 0.0;
    Leaf<float> lf;
    lf.init(tr, sp.ln, sp.agg + 4 * layer, nl, nu, N, nloc, split, slices);
    if (lf.any) {
        const Lines<float> ln = layer_lines(sp.ln, nl, nloc);
        const int lane = lf.lane;
        const int64_t j = min64(lf.jb + lane, N - 1);
        const double nuj = nu[j];
        const double lamd = lf.live ? g_sigma[(size_t)layer * N + j] * lam_scale : 0.0;
        const float hT = (float)(0.5 / T[layer]);
        const float lam = (float)lamd;
        float Th = 0.f, Tl = 0.f, Bh = 0.f, Bl = 0.f; // the chunks' sums as hi + lo floats
        const Span span(lf.g, nu[0]);
        const float rh = span.rh, rl = span.rl;
        const double oj = nuj - lf.g.mid;
        const float ohi = (float)oj, olo = (float)(oj - (double)ohi), h = (float)lf.g.h;
#pragma unroll 1
        for (int k = 0; k < RANGES; k += tr.on ? 2 : 1) { // without 1 and 3 where there are far sets
            const bool masked = k == 0 || k == RANGES - 1;
            const int ce = lf.e[k];
            for (int t0 = lf.s[k] + 32 * lf.sub; t0 < ce; t0 += stride) {
                const int l = t0 + lane;
                const bool have = l < ce;
                __syncwarp();
                float nb = 0.0f, nbl = 0.0f, z2 = 1e30f;
                float4 p2 = make_float4(1.f, 1.f, 0.f, 0.f);
                float2 p3 = make_float2(0.f, 0.f);
                if (have) {
                    const float2 nf = ln.nuf[l];
                    nb = rh - nf.x; // (nb, nbl) = middle - centre, TwoSum of the high parts
                    const float bb = nb - rh;
                    nbl = ((rh - (nb - bb)) - (nf.x + bb)) + (rl - nf.y);
                    p2 = ln.r2[l];
                    p3 = ((const float2*)ln.r3)[l];
                    const float x = fmaxf(fabsf(nb) - h, 0.0f) * p2.x;
                    z2 = fmaf(x, x, p2.y * p2.y);
                    if (masked) tl.jr[lane] = ln.jr[l];
                }
                const int cnt = min(32, ce - t0);
                float aT = 0.0f, aB = 0.0f;
                if (__all_sync(0xffffffffu, z2 >= WING2_Z2)) {
                    // wing forms, f_T and f_b as polynomials in rho (K = 1 from |z| = 100), rows of
                    // fields as in the forward kernel
                    const bool k1only = __all_sync(0xffffffffu, z2 >= WING1_Z2);
                    float* const f = (float*)tl.hf;
                    const float4 p1 = have ? ln.r1[l] : make_float4(1.f, 0.f, 0.f, 0.f);
                    const float G = p1.x, Al = p1.y, F1 = p1.z, F2 = p1.w, aS = p3.x, nn = p3.y;
                    const float U2 = F1 - 2.0f * G * Al;
                    float U3 = 6.0f * F2, U4 = -6.0f * G * F2;
                    float T3 = (aS + 2.0f * hT + 6.0f * nn) * F2, T4 = nn * U4;
                    if (!k1only) {
                        const float cc = p2.x * p2.x, Q = Al * rcp_fast(cc * cc);
                        const float GQ = G * Q, G2Q = G * GQ;
                        T3 = fmaf(Q, 3.75f * aS + 15.0f * hT + 3.75f * nn, T3);
                        T4 = fmaf(-GQ, 15.0f * aS + 60.0f * hT + 67.5f * nn, T4);
                        U3 = fmaf(3.75f, Q, U3);
                        U4 = fmaf(-67.5f, GQ, U4);
                        f[352 + lane] = G2Q * (12.0f * aS + 48.0f * hT + 180.0f * nn);
                        f[384 + lane] = -120.0f * G * G2Q * nn;
                        f[416 + lane] = 180.0f * G2Q;
                        f[448 + lane] = -120.0f * G * G2Q;
                    }
                    f[lane] = nb;
                    f[32 + lane] = nbl;
                    f[64 + lane] = G;
                    f[96 + lane] = Al * (aS + nn);
                    f[128 + lane] = aS * F1 + hT * 2.0f * F1 + nn * U2;
                    f[160 + lane] = T3;
                    f[192 + lane] = T4;
                    f[224 + lane] = Al;
                    f[256 + lane] = U2;
                    f[288 + lane] = U3;
                    f[320 + lane] = U4;
                    __syncwarp();
                    const float4* const r = (const float4*)f;
                    float2 t01 = dup(0.0f), t23 = t01, b01 = t01, b23 = t01;
                    for (int q = 0; q < (cnt + 3) / 4; ++q) {
                        const float4 b = r[q], bl = r[8 + q], g = r[16 + q];
                        const float2 d0 = __fadd2_rn(__fadd2_rn(dup(ohi), lo2(b)), __fadd2_rn(dup(olo), lo2(bl)));
                        const float2 d1 = __fadd2_rn(__fadd2_rn(dup(ohi), hi2(b)), __fadd2_rn(dup(olo), hi2(bl)));
                        float2 r0 = rcp2_shared(__ffma2_rn(d0, d0, lo2(g))), r1 = rcp2_shared(__ffma2_rn(d1, d1, hi2(g)));
                        const float4 t4 = r[48 + q], u4 = r[80 + q];
                        float2 pt0 = lo2(t4), pt1 = hi2(t4), pu0 = lo2(u4), pu1 = hi2(u4);
                        if (!k1only) {
                            const float4 t5 = r[88 + q], t6 = r[96 + q], u5 = r[104 + q], u6 = r[112 + q];
                            pt0 = __ffma2_rn(__ffma2_rn(lo2(t6), r0, lo2(t5)), r0, pt0);
                            pt1 = __ffma2_rn(__ffma2_rn(hi2(t6), r1, hi2(t5)), r1, pt1);
                            pu0 = __ffma2_rn(__ffma2_rn(lo2(u6), r0, lo2(u5)), r0, pu0);
                            pu1 = __ffma2_rn(__ffma2_rn(hi2(u6), r1, hi2(u5)), r1, pu1);
                        }
#pragma unroll
                        for (int k = 2; k >= 0; --k) { // the three lower coefficients of each
                            const float4 t = r[24 + 8 * k + q], u = r[56 + 8 * k + q];
                            pt0 = __ffma2_rn(pt0, r0, lo2(t));
                            pt1 = __ffma2_rn(pt1, r1, hi2(t));
                            pu0 = __ffma2_rn(pu0, r0, lo2(u));
                            pu1 = __ffma2_rn(pu1, r1, hi2(u));
                        }
                        if (masked) mask4(tl.jr + 4 * q, (int)j, r0, r1);
                        t01 = __ffma2_rn(r0, pt0, t01);
                        t23 = __ffma2_rn(r1, pt1, t23);
                        b01 = __ffma2_rn(r0, pu0, b01);
                        b23 = __ffma2_rn(r1, pu1, b23);
                    }
                    aT = (t01.x + t01.y) + (t23.x + t23.y);
                    aB = (b01.x + b01.y) + (b23.x + b23.y);
                } else {
                    if (have) {
                        tl.nb[lane] = make_float4(nb, nbl, ln.clo[l], p2.y > 0.0f ? rcp_fast(p2.y) : 0.0f);
                        tl.r2[lane] = p2;
                        tl.aS[lane] = p3.x;
                        tl.nn[lane] = p3.y;
                        const bool wide = p2.y >= WIDE_A; // summed below
                        float F[ASY_N + 1], G[ASY_N + 1];
                        asy_coeffs_adj(wide ? 0.0f : p2.y, wide ? 0.0f : p2.z, p3.x, hT, p3.y, F, G);
                        store16(tl.hf[lane], F, ASY_N + 1);
                        store16(tl.hg[lane], G, ASY_N + 1);
                        if (p2.y * p2.y < NEAR_POLY_Z2) series_table(p2.y, tl.sd[lane]);
                    }
                    unsigned wide = __ballot_sync(0xffffffffu, have && p2.y >= WIDE_A);
                    __syncwarp();
                    for (int q = 0; q < cnt; ++q) {
                        const bool in = lf.live && (!masked || in_range((int)j, tl.jr[q]));
                        // x to FP32 accuracy suffices for the polynomial (a rational
                        // function of x); the series takes the exact pair
                        const float4 c4 = tl.r2[q];
                        const float4 b = tl.nb[q];
                        const float dh = ohi + b.x, dl = olo + b.y;
                        const float xq = c4.x * (dh + dl);
                        const float zz = fmaf(xq, xq, c4.y * c4.y);
                        if (!__any_sync(0xffffffffu, in && zz < NEAR_POLY_Z2)) {
                            // no lane in the series zone: the polynomials, branch-free
                            const float u = rcp_fast(zz);
                            const float ft = horner14(tl.hf[q], u), fb = horner14(tl.hg[q], u);
                            aT += in ? ft : 0.0f;
                            aB += in ? fb : 0.0f;
                        } else if (in) {
                            // the series also serves the lanes just outside its zone
                            if (!(fabsf(xq) <= SER_X)) {
                                const float u = rcp_fast(zz);
                                aT += horner14(tl.hf[q], u);
                                aB += horner14(tl.hg[q], u);
                            } else {
                                float x, xl;
                                scaled_pair(dh, dl, c4.x, b.z, &x, &xl);
                                float wr, dr, di; // H_x = dr, H_a = -di
                                w_series_deriv(x, xl, c4.y, b.w, c4.w, tl.sd[q], &wr, &dr, &di);
                                const float V0 = c4.z * wr;
                                const float V2 = -c4.z * c4.y * di;
                                const float Db = -(V0 + c4.z * x * dr + V2);
                                aT += tl.aS[q] * V0 + hT * Db + tl.nn[q] * V2;
                                aB += V2;
                            }
                        }
                    }
                    if (wide) {
                        __syncwarp();
                        if (have) stage_wing1_adj(ln.r1[l], p3.x, p3.y, hT, tl.hf[lane], tl.hg[lane]);
                        __syncwarp();
                        for (; wide; wide &= wide - 1) {
                            const int q = __ffs(wide) - 1;
                            const float4 b = tl.nb[q];
                            const float d = (ohi + b.x) + (olo + b.y);
                            add_wing1_adj(tl.hf[q], tl.hg[q], d, !masked || in_range((int)j, tl.jr[q]), aT, aB);
                        }
                    }
                }
                two_sum(Th, Tl, lam * aT);
                two_sum(Bh, Bl, lam * aB);
            }
        }
        sT = (double)Th + (double)Tl;
        sB = (double)Bh + (double)Bl;
    }
    block_pair<LeafWarps<float>::v>(sT, sB, sp.leaf + 2 * ((size_t)nloc * gridDim.x + blockIdx.x));
}

// Moments over half of the leaf's points (the lane's half) of lambda u^(n+1) for the lane's
// line, where the point is inside the cut and at |z| >= 10, and the line's terms.
template <int K>
__device__ __forceinline__ void near_adjoint64(const NearAdjTile64& tl, int q, int half, double amp, bool masked, int jb,
                                               double hT, double& sT, double& sB)
{
    double r[2 * K + 2];
#pragma unroll
    for (int k = 0; k < 2 * K + 2; ++k) r[k] = 0.0;
    const double4_32a p2 = tl.r2[q];
    const double c = tl.cen[q], a2 = p2.y * p2.y;
    const int2 jr = tl.jr[q];
    for (int i = half * (LEAF / 2); i < (half + 1) * (LEAF / 2); ++i) {
        const double x = (tl.pos[i] - c) * p2.x, zz = fma(x, x, a2);
        const bool in = (!masked || in_range(jb + i, jr)) && zz >= Tier<double>::z2_series;
        const double u = rcp64(in ? zz : 1.0);
        double s = in ? tl.lam[i] * u : 0.0;
#pragma unroll
        for (int k = 0; k < 2 * K + 2; ++k) {
            r[k] += s;
            s *= u;
        }
    }
    double V0, Db, Dg;
    asy64_adjoint<K>(p2.y, amp, r, &V0, &Db, &Dg);
    add_adjoint(V0, Db, Dg, tl.aS[q], hT, tl.nn[q], sT, sB);
}

// FP64 adjoint of a leaf: the wing polynomials with a line (and half of the points) a
// lane, so that a line's coefficients are applied once to its moments; the series with a
// point a lane.
__global__ void __launch_bounds__(32 * LeafWarps<double>::v) leaf_adjoint_f64(const __grid_constant__ Batch<double> batch,
                                                                            const double* __restrict__ nu, int64_t N,
                                                                            int layer0,
                                                                            const double* __restrict__ T,
                                                                            double lam_scale, int split, int slices,
                                                                            int stride)
{
    const Species<double>& sp = batch.s[blockIdx.z];
    const Tree& tr = sp.tree;
    const int64_t nl = sp.nl;
    const double* __restrict__ g_sigma = sp.g_sigma;
    extern __shared__ __align__(32) unsigned char smem64[];
    NearAdjTile64& tl = ((NearAdjTile64*)smem64)[threadIdx.x >> 5];
    const int nloc = blockIdx.y, layer = layer0 + nloc;
    double sT = 0.0, sB = 0.0;
    Leaf<double> lf;
    lf.init(tr, sp.ln, sp.agg + 4 * layer, nl, nu, N, nloc, split, slices);
    if (lf.any) {
        const Lines<double> ln = layer_lines(sp.ln, nl, nloc);
        const int lane = lf.lane;
        const int64_t j = min64(lf.jb + lane, N - 1);
        const double nuj = nu[j];
        const double lam = lf.live ? g_sigma[(size_t)layer * N + j] * lam_scale : 0.0;
        const double hT = 0.5 / T[layer];
        tl.pos[lane] = nuj;
        tl.lam[lane] = lam;
#pragma unroll 1
        for (int k = 0; k < RANGES; k += tr.on ? 2 : 1) { // without 1 and 3 where there are far sets
            const bool masked = k == 0 || k == RANGES - 1;
            const int ce = lf.e[k];
            for (int t0 = lf.s[k] + NEAR64 * lf.sub; t0 < ce; t0 += stride) {
                const int l = t0 + lane;
                const bool have = lane < NEAR64 && l < ce;
                const int cnt = min(NEAR64, ce - t0);
                __syncwarp();
                double z2 = 1e300;
                if (have) {
                    const double c = ln.nu_hat[l];
                    const double4_32a p2 = ln.r2[l];
                    z2 = nearest_z2(lf.g.mid - c, lf.g.h, p2);
                    tl.cen[lane] = c;
                    tl.r2[lane] = p2;
                    tl.aS[lane] = ln.r3[2 * (size_t)l];
                    tl.nn[lane] = ln.r3[2 * (size_t)l + 1];
                    if (masked) tl.jr[lane] = ln.jr[l];
                    if (z2 < Tier<double>::z2_stage) {
                        tl.ia[lane] = p2.y > 0.0 ? 1.0 / p2.y : 0.0;
                        series_table64(p2.y, tl.sd[lane]);
                    }
                }
                unsigned near = __ballot_sync(0xffffffffu, z2 < Tier<double>::z2_stage); // lines with series points
                __syncwarp();
                const int q = min(lane % NEAR64, cnt - 1), half = lane / NEAR64;
                const double amp = lane % NEAR64 < cnt ? tl.r2[q].z : 0.0;
                by_terms64(z2, [&](auto K) {
                    near_adjoint64<decltype(K)::value>(tl, q, half, amp, masked, (int)lf.jb, hT, sT, sB);
                });
                while (near) {
                    const int i = __ffs(near) - 1;
                    near &= near - 1;
                    const double4_32a c4 = tl.r2[i];
                    const double x = fabs(nuj - tl.cen[i]) * c4.x, zz = fma(x, x, c4.y * c4.y);
                    if (lf.live && zz < Tier<double>::z2_series && (!masked || in_range((int)j, tl.jr[i]))) {
                        double wr, dr, di; // H_x = dr, H_a = -di
                        w_series_deriv(x, c4.y, tl.ia[i], c4.w, tl.sd[i], &wr, &dr, &di);
                        const double V0 = c4.z * wr, V2 = -c4.z * c4.y * di;
                        const double Db = -(V0 + c4.z * x * dr + V2);
                        sT = fma(lam, fma(tl.aS[i], V0, fma(hT, Db, tl.nn[i] * V2)), sT);
                        sB = fma(lam, V2, sB);
                    }
                }
            }
        }
    }
    block_pair<LeafWarps<double>::v>(sT, sB, sp.leaf + 2 * ((size_t)nloc * gridDim.x + blockIdx.x));
}

// g_T[n] = sum over the leaf blocks' and the far kernel's partials of layer n (one
// block per layer of the chunk, fixed order); gbl[n] the same for the broadening term.
template <class R>
__global__ void __launch_bounds__(256) adjoint_reduce_kernel(const __grid_constant__ Batch<R> batch, int layer0,
                                                             int leaf_blocks)
{
    __shared__ double red[2][256];
    const Species<R>& sp = batch.s[blockIdx.z];
    const int n = blockIdx.x, slots = sp.tree.on ? sp.fw.slots : 0;
    const double* __restrict__ leaf = sp.leaf + 2 * (size_t)n * leaf_blocks;
    const double* __restrict__ far = sp.slots + 2 * (size_t)n * slots;
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < leaf_blocks; i += blockDim.x) {
        a += leaf[2 * (size_t)i];
        b += leaf[2 * (size_t)i + 1];
    }
    for (int i = threadIdx.x; i < slots; i += blockDim.x) {
        a += far[2 * (size_t)i];
        b += far[2 * (size_t)i + 1];
    }
    red[0][threadIdx.x] = a;
    red[1][threadIdx.x] = b;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        sp.g_T[layer0 + n] = red[0][0];
        sp.gbl[layer0 + n] = red[1][0];
    }
}

// g_b = sum over layers of gbl / s_b per species (one warp, fixed order); g_T_sum += the
// species' g_T where given
template <class R>
__global__ void broad_sum_kernel(const __grid_constant__ Batch<R> batch, int L, double inv_sb,
                                 double* __restrict__ g_T_sum)
{
    for (int m = 0; m < batch.n; ++m) {
        const Species<R>& sp = batch.s[m];
        double s = 0.0;
        for (int n = threadIdx.x; n < L; n += 32) {
            s += sp.gbl[n];
            if (g_T_sum) g_T_sum[n] += sp.g_T[n];
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (threadIdx.x == 0) sp.g_b[0] = s * inv_sb;
    }
}

} // namespace xsd

// ====================================================================== host side

using namespace xsd;

namespace {

size_t align256(size_t v) { return (v + 255) & ~(size_t)255; }

// Lists shorter than this are summed point by point.  With the intervals a call pays three
// more launches, and polynomials and node weights per layer whatever the list's length.  FP32,
// us without and with them, forward and adjoint: 255 lines on 4,096 points x 20 layers 43 and
// 64, 60 and 78; on 50,000 x 100 698 and 787, 1084 and 852 (128 lines 502 and 764, 810 and
// 823).  FP64 pairs cost ten times more: 64 lines on 4,096 points 185 and 118, 339 and 270; x 20
// layers 312 and 246, 635 and 614; 32 lines 117 and 102, 210 and 246.
template <class R> struct ShortList { static constexpr int64_t v = 256; };
template <> struct ShortList<double> { static constexpr int64_t v = 64; };
int64_t tree_min_lines(int prec) { return prec == XS_PREC_MIXED ? ShortList<float>::v : ShortList<double>::v; }

// Density of lines from which an interval has two intervals below it instead of four, in
// half lines a grid point.  A level's list holds the lines between its far radius and that
// of the interval above, so halving makes seven levels of a third of the list each instead
// of four: 2/3 of the far evaluations for 1.5 times the polynomials, node weights and
// reductions.  FP32, 20,000 points x 20 layers, us with quarters and halves: at one line a
// point forward 362 and 371, adjoint 498 and 487; at two 615 and 606, 883 and 840; at
// eight 2016 and 1893, 3126 and 2888.  FP64, 4,096 points x 20 layers, a line every two
// points 2039 and 1877, 3920 and 3606 (one layer 279 and 286, 483 and 493), one a point
// 3807 and 3464, 7249 and 6517.  With the choice at run time calls that keep the quarters
// are up to 1% slower than with four fixed levels (one FP64 layer 268 -> 275 us).
template <class R> struct DenseLines { static constexpr int64_t v = 4; };
template <> struct DenseLines<double> { static constexpr int64_t v = 1; };

struct XsPlan {
    int prec, Lc, nchunks, leaf_blocks, leaf_warps, leaf_split, slices; // leaf_blocks: of all slices
    Tree tree; // counts and offsets; pointers set at run time
    FarWork fw;
    int far_blocks;
    size_t off_jr, off_nuf, off_inv, off_agg, off_rec1, off_rec2, off_rec3, off_clo, off_geo, off_cov, off_win, off_pq,
        off_fwd, off_coef, off_near, off_wts, off_slots, off_leaf, off_gbl, total;
};

// What of the intervals a plan holds: COMPACT has four intervals below each one and splits
// their lists in as many parts as cost about a byte a line, the least space with which far
// lines go to the nodes.
enum Intervals { LEAVES_ONLY, COMPACT, FULL };

// Parts of the far lists: enough warps to fill the GPU several times over, each with a
// list long enough to pay for its reduction (FP64 evaluations cost about ten times
// more).  A level's list is estimated from its share of the grid: the lines between
// its own far radius and its parent's, about 16 interval lengths.
void split_far(XsPlan* p, int64_t nl, int64_t N, int Lc, bool mixed, bool compact)
{
    const int64_t warps = mixed ? 10000 : 8000, min_lines = mixed ? 1024 : 64;
    int block = 0;
    size_t row = 0;
    p->fw.slots = 0;
    const Tree& tr = p->tree;
    const double lengths = tr.shift == 2 ? 16.0 : 8.0;
    for (int k = tr.top; k >= 0; --k) {
        const double share = std::min(1.0, lengths * (double)(LEAF << (tr.shift * k)) / (double)N);
        const int64_t est = (k == tr.top) ? nl : (int64_t)(share * (double)nl);
        const int64_t want = (warps + (int64_t)Lc * p->tree.cnt[k] - 1) / ((int64_t)Lc * p->tree.cnt[k]);
        int64_t parts = std::max<int64_t>(1, std::min(want, est / min_lines));
        if (compact) parts = std::min(parts, std::max<int64_t>(1, nl / (512 * (int64_t)p->tree.cnt[k])));
        p->fw.parts[k] = (int)parts;
        p->fw.block0[k] = block;
        p->fw.out0[k] = row;
        p->fw.slot0[k] = p->fw.slots;
        block += (int)parts * ((p->tree.cnt[k] + FAR_WARPS - 1) / FAR_WARPS);
        row += (size_t)parts * Lc * p->tree.cnt[k];
        p->fw.slots += (int)parts * p->tree.cnt[k];
    }
    p->far_blocks = block;
    p->fw.rows = row;
}

// Blocks of the leaf kernels.  With enough leaves, a warp each and full blocks; fewer
// leaves than fill the chip share each leaf's lines between up to a block's warps and use
// smaller blocks, so that the work reaches more SMs (one layer of 4,096 points has 128
// leaves: in FP64, 16 blocks of 8 leaves took 616 us, 128 blocks with 8 warps on a leaf
// 125 us; FP32, 32 blocks of 4 leaves 22 us, 128 blocks of one 14 us).
void choose_leaf_blocks(XsPlan* p, int64_t nl, int64_t N, int Lc, bool mixed, Intervals how)
{
    const int most = mixed ? LeafWarps<float>::v : LeafWarps<double>::v;
    const int64_t leaves = (N + LEAF - 1) / LEAF, all = leaves * Lc;
    const int64_t want = mixed ? xsi::SMS * 16 : xsi::SMS * 8; // warps
    const bool small = how == LEAVES_ONLY; // the smallest workspaces hold one partial per full block
    int split = 1;
    while (!small && split < most && all * split < want) split *= 2;
    int warps = most;
    while (!small && warps > split && all * split / warps < 2 * xsi::SMS) warps /= 2;
    p->leaf_split = split;
    p->leaf_warps = warps;
    const int per = warps / split;
    // and of long lists between blocks as well: 1,000,000 lines at 64 points 60 cm^-1 apart, one
    // layer, 25.1 -> 1.3 ms (its two leaves ran on two SMs), 60,000 on 2,000 points 235 -> 147 us;
    // FP64, 6,000 on 500 1312 -> 507 us
    const int64_t lines = mixed ? 8192 : 512; // of the whole list for each slice
    p->slices = how == FULL ? (int)std::max<int64_t>(1, std::min<int64_t>({64, want / (all * split), nl / lines})) : 1;
    p->leaf_blocks = (int)((leaves + per - 1) / per) * p->slices;
}

XsPlan plan_xs(int64_t nl, int64_t N, int32_t L, int prec, int Lc, Intervals how)
{
    const bool tree = how != LEAVES_ONLY;
    XsPlan p{};
    p.prec = prec;
    p.Lc = Lc;
    const bool mixed = (prec == XS_PREC_MIXED);
    const size_t rs = mixed ? sizeof(float) : sizeof(double);
    const int n = mixed ? Far<float>::n : Far<double>::n;
    const size_t n1 = (size_t)std::max<int64_t>(nl, 1);
    size_t off = 0;
    auto take = [&](size_t bytes) {
        size_t o = off;
        off += align256(bytes);
        return o;
    };
    choose_leaf_blocks(&p, nl, N, Lc, mixed, how);
    p.off_jr = take(sizeof(int2) * n1);
    p.off_nuf = take(mixed ? sizeof(float2) * n1 : 0);
    p.off_inv = take(sizeof(double) * n1);
    p.off_agg = take(sizeof(float) * 4 * (size_t)L);
    p.off_rec1 = take(4 * rs * n1 * Lc);
    p.off_rec2 = take(4 * rs * n1 * Lc);
    p.off_rec3 = take(2 * rs * n1 * Lc);
    p.off_clo = take(mixed ? rs * n1 * Lc : 0);
    p.off_gbl = take(sizeof(double) * (size_t)L);
    p.tree.on = tree ? 1 : 0;
    if (tree) {
        p.tree.shift = how == FULL && 2 * nl >= (mixed ? DenseLines<float>::v : DenseLines<double>::v) * N ? 1 : 2;
        p.tree.top = TOP_LOG / p.tree.shift;
        for (int k = 0; k <= p.tree.top; ++k) {
            const int64_t pts = (int64_t)LEAF << (p.tree.shift * k);
            p.tree.cnt[k] = (int)((N + pts - 1) / pts);
            p.tree.off[k] = p.tree.total;
            p.tree.total += p.tree.cnt[k];
        }
        split_far(&p, nl, N, Lc, mixed, how == COMPACT);
        p.off_geo = take(sizeof(Geo) * (size_t)p.tree.total);
        p.off_cov = take(sizeof(int2) * (size_t)p.tree.total);
        p.off_win = take(sizeof(int2) * (size_t)p.tree.cnt[0]);
        p.off_pq = take(sizeof(int2) * (size_t)p.tree.total * Lc);
    }
    // the forward's node sums and polynomials; the adjoint's weights and partials reuse the space
    const size_t base = off;
    if (tree) {
        p.off_fwd = take(sizeof(double) * n * p.fw.rows);
        p.off_coef = take(sizeof(double) * (mixed ? LeafPoly<float>::stride : LeafPoly<double>::stride) * (size_t)Lc *
                          p.tree.cnt[0]);
    }
    p.off_near = take(p.slices > 1 ? sizeof(double) * p.slices * (size_t)Lc * (size_t)N : 0);
    const size_t fwd_end = off;
    off = base;
    if (tree) {
        p.off_wts = take(rs * n * (size_t)Lc * p.tree.total);
        p.off_slots = take(sizeof(double) * 2 * (size_t)Lc * p.fw.slots);
    }
    p.off_leaf = take(sizeof(double) * 2 * (size_t)Lc * p.leaf_blocks);
    p.total = std::max(off, fwd_end);
    p.nchunks = (L + Lc - 1) / Lc;
    return p;
}

} // namespace

size_t xs_workspace_bytes(int64_t n_lines, int64_t N, int32_t L, int prec)
{
    if (n_lines < 0 || N <= 0 || L <= 0) return 0;
    return plan_xs(n_lines, N, L, prec, L, n_lines >= tree_min_lines(prec) ? FULL : LEAVES_ONLY).total;
}

// Lists of this length and more ask for the intervals in the smallest workspace too: without
// them 20,000 lines on 20,000 points and 10 layers take 7.6 ms instead of 1.0, 220,000 and 4
// layers 32.7 ms instead of 1.1.  They cost 8 to 13 bytes a grid point beside the lines' 68 to
// 96 each; shorter lists would grow by more than they gain.
constexpr int64_t COMPACT_MIN_LINES = 2048;

size_t xs_workspace_min_bytes(int64_t n_lines, int64_t N, int32_t L, int prec)
{
    if (n_lines < 0 || N <= 0 || L <= 0) return 0;
    return plan_xs(n_lines, N, L, prec, 1, n_lines >= COMPACT_MIN_LINES ? COMPACT : LEAVES_ONLY).total;
}

namespace xsi {

size_t xs_least_bytes(int64_t n_lines, int64_t N, int32_t L, int prec)
{
    return plan_xs(n_lines, N, L, prec, 1, LEAVES_ONLY).total;
}

// The largest chunk of layers whose plan fits, with the intervals if any such fits.
static int pick_plan(int64_t nl, int64_t N, int32_t L, int prec, size_t ws_bytes, XsPlan* out)
{
    for (int how = nl >= tree_min_lines(prec) ? FULL : LEAVES_ONLY; how >= LEAVES_ONLY; --how)
        for (int Lc = L;; Lc = (Lc + 1) / 2) {
            XsPlan p = plan_xs(nl, N, L, prec, Lc, (Intervals)how);
            if (p.total <= ws_bytes) {
                *out = p;
                return XS_OK;
            }
            if (Lc == 1) break;
        }
    return XS_EINVAL;
}

static unsigned blocks_of(int64_t n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// A species' arrays in its workspace.
template <class R>
static Species<R> make_species(const xs_lines* ln, const XsPlan& p, char* ws, int32_t L)
{
    constexpr bool FAST = std::is_same<R, float>::value;
    using R4 = typename vec4<R>::type;
    const int64_t nl = ln->n;
    Species<R> s{};
    s.ln_S0 = ln->ln_S0;
    s.elower = ln->elower;
    s.gamma_ref = ln->gamma_ref;
    s.n_temp = ln->n_temp;
    s.mass = ln->mass_amu;
    s.qexp = ln->q_exponent;
    s.nl = nl;
    s.fw = p.fw;
    s.setup_blocks = (int)blocks_of(2 * nl + 4 * (int64_t)L + 4 * (int64_t)p.tree.total, 256);
    // four lines a thread where that leaves enough blocks: the layer's constants are formed per block
    s.param_blocks = (int)(nl >= 65536 ? blocks_of(nl, 1024) : blocks_of(nl, 256));
    s.far_blocks = p.far_blocks;
    s.jr = (int2*)(ws + p.off_jr);
    s.nuf = FAST ? (float2*)(ws + p.off_nuf) : nullptr;
    s.w_inv_nu = (double*)(ws + p.off_inv);
    s.agg = (float*)(ws + p.off_agg);
    s.rec1 = (R4*)(ws + p.off_rec1);
    s.rec2 = (R4*)(ws + p.off_rec2);
    s.rec3 = (R*)(ws + p.off_rec3);
    s.clo = FAST ? (R*)(ws + p.off_clo) : nullptr;
    s.geo = (Geo*)(ws + p.off_geo);
    s.cov = (int2*)(ws + p.off_cov);
    s.win = (int2*)(ws + p.off_win);
    s.pq = (int2*)(ws + p.off_pq);
    s.sums = (double*)(ws + p.off_fwd);
    s.coef = (double*)(ws + p.off_coef);
    s.near = (double*)(ws + p.off_near);
    s.wts = (R*)(ws + p.off_wts);
    s.slots = (double*)(ws + p.off_slots);
    s.leaf = (double*)(ws + p.off_leaf);
    s.gbl = (double*)(ws + p.off_gbl);
    s.inv_nu = s.w_inv_nu;
    s.tree = p.tree;
    s.tree.geo = s.geo;
    s.tree.cov = s.cov;
    s.tree.win = s.win;
    s.tree.pq = s.pq;
    s.ln = Lines<R>{ln->nu_hat, s.nuf, s.jr, s.rec1, s.rec2, s.rec3, s.clo};
    return s;
}

// The line sums (or their adjoints) of a batch of species with plans of the same shape
// (same chunks of layers, same use of the intervals, same slices); p: the first one's.
template <class R>
static int run_batch(const Batch<R>& b, const XsPlan& p, const double* nu, int64_t N, const double* T, const double* P,
                     int32_t L, double sb, double W, bool adjoint, cudaStream_t st, int flags, double* g_T_sum)
{
    // flags: XS_RUN_KEEP_ADJ  (forward) also write the adjoint's per-line records
    //        XS_RUN_REUSE     (adjoint) the records and ranges of an immediately preceding
    //                         forward with the same inputs and workspace are still valid
    constexpr bool FAST = std::is_same<R, float>::value;
    const bool reuse = adjoint && (flags & XS_RUN_REUSE) && p.nchunks == 1;
    const bool want_rec3 = adjoint || (flags & XS_RUN_KEEP_ADJ);
    const double unscale = FAST ? MIXED_UNSCALE : 1.0;
    const unsigned nz = (unsigned)b.n;
    const Tree& tr = p.tree;
    int setup_blocks = 0, param_blocks = 0, far_blocks = 0, intervals = 0;
    for (int m = 0; m < b.n; ++m) {
        intervals = std::max(intervals, b.s[m].tree.total);
        setup_blocks = std::max(setup_blocks, b.s[m].setup_blocks);
        param_blocks = std::max(param_blocks, b.s[m].param_blocks);
        far_blocks = std::max(far_blocks, b.s[m].far_blocks);
    }
    if constexpr (!FAST) {
        // beyond 48 KB of shared memory a block has to ask (cheap; per device)
        if (cudaFuncSetAttribute(leaf_kernel_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(LeafWarps<double>::v * sizeof(NearTile64))) != cudaSuccess ||
            cudaFuncSetAttribute(leaf_adjoint_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)(LeafWarps<double>::v * sizeof(NearAdjTile64))) != cudaSuccess)
            return XS_ECUDA;
    }
    if (!reuse) {
        setup_kernel<R><<<dim3((unsigned)setup_blocks, 1, nz), 256, 0, st>>>(b, nu, N, W, 4 * L);
        count_launch();
    }
    for (int c = 0; c < p.nchunks; ++c) {
        const int l0 = c * p.Lc;
        const int lc = std::min(p.Lc, L - l0);
        if (!reuse) {
            line_params_kernel<R>
                <<<dim3((unsigned)param_blocks, (unsigned)lc, nz), 256, 0, st>>>(b, T, P, l0, sb, want_rec3);
            count_launch();
            if (tr.on) {
                near_range_kernel<R>
                    <<<dim3(blocks_of(2 * (int64_t)intervals, 256), (unsigned)lc, nz), 256, 0, st>>>(b, l0);
                count_launch();
            }
        }
        const dim3 lgrid((unsigned)p.leaf_blocks, (unsigned)lc, nz);
        const dim3 fgrid((unsigned)far_blocks, (unsigned)lc, nz);
        const int lthreads = 32 * p.leaf_warps;
        const int stride = (FAST ? 32 : NEAR64) * p.leaf_split * p.slices; // lines from a warp's chunk to its next
        prof_begin(adjoint ? 1 : 0, st);
        if (!adjoint) {
            if (tr.on) {
                far_sum_kernel<R><<<fgrid, 32 * FAR_WARPS, 0, st>>>(b, nu, l0);
                int root = TOP_LOG; // log2 of the leaves of a block
                auto subtrees = [&] { return blocks_of(tr.cnt[0], 1 << root); };
                while (root > 2 && (int64_t)subtrees() * lc * b.n < 2 * SMS) root -= 2;
                const int rows = std::min(DownRows<R>::v, 1 << root);
                down_kernel<R><<<dim3(subtrees(), (unsigned)lc, nz), rows * Far<R>::n, 0, st>>>(b, lc, root);
                count_launch(2);
            }
            if constexpr (FAST)
                leaf_kernel_f32<<<lgrid, lthreads, 0, st>>>(b, nu, N, l0, unscale, p.leaf_split, p.slices, stride);
            else
                leaf_kernel_f64<<<lgrid, lthreads, p.leaf_warps * sizeof(NearTile64), st>>>(b, nu, N, l0, unscale,
                                                                                           p.leaf_split, p.slices, stride);
        } else {
            if (tr.on) {
                up_kernel<R><<<dim3(blocks_of(tr.cnt[0], TOP), (unsigned)lc, nz), 32 * UP_WARPS, 0, st>>>(b, nu, N, l0,
                                                                                                         unscale);
                far_adjoint_kernel<R><<<fgrid, 32 * FAR_WARPS, 0, st>>>(b, nu, l0, T);
                count_launch(2);
            }
            if constexpr (FAST)
                leaf_adjoint_f32<<<lgrid, lthreads, 0, st>>>(b, nu, N, l0, T, unscale, p.leaf_split, p.slices, stride);
            else
                leaf_adjoint_f64<<<lgrid, lthreads, p.leaf_warps * sizeof(NearAdjTile64), st>>>(b, nu, N, l0, T,
                                                                                              unscale, p.leaf_split, p.slices, stride);
        }
        if (!adjoint && p.slices > 1) {
            slices_kernel<R><<<dim3(blocks_of(N, 256), (unsigned)lc, nz), 256, 0, st>>>(b, nu, N, l0, unscale, p.slices);
            count_launch();
        }
        prof_end(adjoint ? 1 : 0, st);
        count_launch();
        if (adjoint) { // the next chunk of layers takes the partials' space
            adjoint_reduce_kernel<R><<<dim3((unsigned)lc, 1, nz), 256, 0, st>>>(b, l0, p.leaf_blocks);
            count_launch();
        }
    }
    if (adjoint) {
        broad_sum_kernel<R><<<1, 32, 0, st>>>(b, L, 1.0 / sb, g_T_sum);
        count_launch();
    }
    return (cudaGetLastError() == cudaSuccess) ? XS_OK : XS_ECUDA;
}

// Species with lines and plans of one shape run together, the others by themselves, in order.
template <class R>
static int run_species(int n, const XsJob* job, const XsPlan* plan, const double* nu, int64_t N, const double* T,
                       const double* P, int32_t L, double sb, double W, bool adjoint, cudaStream_t st, int flags,
                       double* g_T_sum)
{
    int m = 0;
    while (m < n) {
        if (job[m].lines->n == 0) {
            if (adjoint) {
                if (cudaMemsetAsync(job[m].g_T, 0, sizeof(double) * L, st) != cudaSuccess) return XS_ECUDA;
                if (cudaMemsetAsync(job[m].g_b, 0, sizeof(double), st) != cudaSuccess) return XS_ECUDA;
            } else if (cudaMemsetAsync(job[m].sigma, 0, sizeof(R) * (size_t)L * N, st) != cudaSuccess) {
                return XS_ECUDA;
            }
            ++m;
            continue;
        }
        const int first = m;
        Batch<R> b{};
        while (m < n && job[m].lines->n > 0 && plan[m].tree.on == plan[first].tree.on && plan[m].Lc == plan[first].Lc &&
               plan[m].slices == plan[first].slices) {
            Species<R>& s = b.s[b.n++];
            s = make_species<R>(job[m].lines, plan[m], (char*)job[m].ws, L);
            s.sigma = job[m].sigma;
            s.g_sigma = job[m].g_sigma;
            s.g_T = job[m].g_T;
            s.g_b = job[m].g_b;
            ++m;
        }
        const int r = run_batch<R>(b, plan[first], nu, N, T, P, L, sb, W, adjoint, st, flags, g_T_sum);
        if (r != XS_OK) return r;
    }
    return XS_OK;
}

int xs_run(int n, const XsJob* job, const double* nu, int64_t N, const double* T, const double* P, int32_t L, double sb,
           double W, int prec, bool adjoint, cudaStream_t st, int flags, double* g_T_sum)
{
    XsPlan plan[XS_MAX_SPECIES];
    for (int m = 0; m < n; ++m)
        if (pick_plan(job[m].lines->n, N, L, prec, job[m].ws_bytes, &plan[m]) != XS_OK) return XS_EINVAL;
    if (prec == XS_PREC_FP64)
        return run_species<double>(n, job, plan, nu, N, T, P, L, sb, W, adjoint, st, flags, g_T_sum);
    return run_species<float>(n, job, plan, nu, N, T, P, L, sb, W, adjoint, st, flags, g_T_sum);
}

int check_sorted(const double* nu_hat, int64_t n, cudaStream_t st, int* flag_dev, bool grid)
{
    if (n < 2) return XS_OK;
    if (cudaMemsetAsync(flag_dev, 0, sizeof(int), st) != cudaSuccess) return XS_ECUDA;
    if (grid)
        grid_check_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(nu_hat, n, flag_dev);
    else
        sorted_check_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(nu_hat, n, flag_dev);
    count_launch();
    int h = 0;
    if (cudaMemcpyAsync(&h, flag_dev, sizeof(int), cudaMemcpyDeviceToHost, st) != cudaSuccess) return XS_ECUDA;
    if (cudaStreamSynchronize(st) != cudaSuccess) return XS_ECUDA;
    return h ? XS_EUNSORTED : XS_OK;
}

} // namespace xsi

XS_CHECK_ACCESSOR(linesum)
