// Astronomical and instrumental responses (Sec. 4): rigid rotation with
// quadratic limb darkening and a Gaussian instrumental profile with a radial
// velocity, as the normalised kernel sums of Eq. responsenu,
//   F(nu'_i) = sum_j k(c ln(nu'_i/nu_j) + RV) F0_j / sum_j k(c ln(nu'_i/nu_j)),
// and their adjoints (in the input spectrum and in vsini or RV).
//
// The pairs inside the kernel's support are found by binary search on the (increasing)
// grids.  The rotation kernel vanishes for |v| >= vsini; the Gaussian is summed over
// |v| <= 10 beta (the rest is below e^-50 of its peak).  Velocities in km/s, FP64
// throughout; FP64 runs at 2 lanes a clock and SM here, so what counts is the number of
// operations a pair.  A block takes neighbouring output points, whose supports overlap,
// and stages the input points, their reciprocals and values once; a pair's logarithm of
// a ratio near one is then a quotient from the reciprocal and a short polynomial instead of
// a division and a logarithm.  Several lanes share an output point.
#include <algorithm>
#include <cmath>

#include "xs_device.cuh"
#include "xs_internal.h"

namespace xsd {

constexpr double C_KMS = 299792.458;
constexpr int RESP_THREADS = 128;
constexpr int RESP_TILE = 512; // staged points
constexpr double GAUSS_SUPPORT = 10.0;

// The kernels in the scaled velocity x = v/scale: value and derivative in x.
//
// zeta(x) of Sec. 4.1 from its disk-integral definition, s = sqrt(1 - x^2):
//   zeta = (2s (1 - u1 - u2) + (pi/2)(u1 + 2u2) s^2 - (4/3) u2 s^3) / (pi (1 - u1/3 - u2/6)),
// scale = vsini; d zeta/d vsini = -x zeta'(x)/vsini.
struct RotKernel {
    static constexpr bool ROT = true;
    double scale, W;
    double c1, c2, c3; // zeta = s (c1 + s (c2 + s c3))
    template <bool D>
    __device__ __forceinline__ void eval(double x, double* k, double* dk) const
    {
        const double q = fmax(fma(-x, x, 1.0), 0.0);
        const double y = q > 0.0 ? rsqrt(q) : 0.0, s = q * y;
        *k = s * fma(s, fma(s, c3, c2), c1);
        if (D) *dk = -x * y * fma(s, fma(s, 3.0 * c3, 2.0 * c2), c1);
    }
};

// Gaussian IP of Sec. 4.2 (normalisation cancels in Eq. responsenu), scale = beta
struct GaussKernel {
    static constexpr bool ROT = false;
    double scale, W;
    template <bool D>
    __device__ __forceinline__ void eval(double x, double* k, double* dk) const
    {
        *k = exp(-0.5 * x * x);
        if (D) *dk = -x * *k;
    }
};

// What every pair needs of the kernel's scale and the velocity, and the ends of a support as
// factors of its point's wavenumber, formed on the host.
struct PairConst {
    double inv, rvs, cinv; // 1/scale, rv/scale, c/scale
    double lo, hi;
};

__device__ __forceinline__ int64_t lower_idx(const double* v, int64_t n, double x) // first i with v[i] >= x
{
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        if (v[m] >= x) hi = m; else lo = m + 1;
    }
    return lo;
}

// The points [b, e) of a grid v that meet each of a block's own points (G lanes each), and
// the block's range of them.  sparse: the own points lie so far apart that a tile of the range
// serves few of them; then each group reads its own support from memory (50 points observed
// of 1,000,000: 1092 us in tiles, whose groups wait for one another, 274 before them).
struct Support {
    int64_t b, e, first, last;
    bool sparse;
    template <int G>
    __device__ __forceinline__ void find(const double* v, int64_t n, double lo, double hi, bool live)
    {
        __shared__ long long r[3];
        // the first two lanes of a group search one end each
        const int g = threadIdx.x % G;
        long long f = 0;
        if (g < 2) f = live ? lower_idx(v, n, g ? hi : lo) : 0;
        b = __shfl_sync(0xffffffffu, f, 0, G);
        e = __shfl_sync(0xffffffffu, f, 1, G);
        if (!live) e = b;
        if (threadIdx.x == 0) {
            r[0] = n;
            r[1] = r[2] = 0;
        }
        __syncthreads();
        if (g == 0 && live && e > b) {
            atomicMin(&r[0], (long long)b);
            atomicMax(&r[1], (long long)e);
            atomicMax(&r[2], (long long)(e - b));
        }
        __syncthreads();
        first = r[0];
        last = r[1];
        sparse = last - first > RESP_TILE && last - first > 2 * r[2];
    }
};

template <int G>
__device__ __forceinline__ double group_sum(double v)
{
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, G);
    return v;
}

// ln(a/b), rb = 1/b: the quotient rounded as a division rounds it (Markstein 1990: one
// residual step from a product with the reciprocal), and as its distance from one is
// exact, the series of ln(1 + d) to d^6; the next term is below 2e-17 of ln for |d| < 2e-3.
// Supports that reach further (SMALL = false) take the logarithm.
constexpr double RESP_SMALL_KMS = 500.0;
template <bool SMALL>
__device__ __forceinline__ double log_ratio(double a, double b, double rb)
{
    const double q0 = a * rb;
    const double q = fma(fma(-q0, b, a), rb, q0);
    if (!SMALL) return log(q);
    const double d = q - 1.0;
    double p = fma(d, -1.0 / 6.0, 1.0 / 5.0);
    p = fma(d, p, -1.0 / 4.0);
    p = fma(d, p, 1.0 / 3.0);
    p = fma(d, p, -1.0 / 2.0);
    return fma(d * d, p, d);
}

// Forward (and, with D, the derivative of the output in the kernel's parameter: for the
// rotation d/d vsini of num/den, for the Gaussian d/d RV).  den[i] is written when
// den != nullptr.  G lanes an output point; RESP_THREADS/G points a block.
// (Rotation at 30 km/s on 20,000 points, 350 pairs a point, and a Gaussian of 2 km/s onto
// 3,001 points, both with gradients: 8.76 -> 1.65 ms; before, a division, a logarithm and
// two square roots or exponentials a pair, one thread an output point.)
template <class K, bool D, int G, bool SMALL>
__global__ void __launch_bounds__(RESP_THREADS) response_kernel(const double* __restrict__ F, const double* __restrict__ nu,
                                                                int64_t N, const double* __restrict__ nu_out,
                                                                int64_t No, K ker, PairConst kc,
                                                                double* __restrict__ out, double* __restrict__ den_out,
                                                                const double* __restrict__ g_out,
                                                                double* __restrict__ part)
{
    __shared__ double red[RESP_THREADS], pv[RESP_TILE], pr[RESP_TILE], pf[RESP_TILE];
    constexpr int OB = RESP_THREADS / G;
    const int t = threadIdx.x, g = t % G;
    const int64_t i0 = (int64_t)blockIdx.x * OB, i = i0 + t / G;
    const bool live = i < No;
    const double nui = nu_out[live ? i : i0];
    const double inv = kc.inv, rvs = kc.rvs, cinv = kc.cinv;
    Support sp{};
    sp.find<G>(nu, N, nui * kc.lo, nui * kc.hi, live);
    double num = 0.0, den = 0.0, dnum = 0.0, dden = 0.0;
    auto pair = [&](double v, double r, double Fj) {
        const double x = cinv * log_ratio<SMALL>(nui, v, r);
        double k, dk = 0.0;
        ker.template eval<D>(x + rvs, &k, &dk);
        num = fma(k, Fj, num);
        if (K::ROT) {
            // rv = 0: the numerator's kernel is the denominator's
            den += k;
            if (D) {
                dnum = fma(-(x + rvs) * dk, Fj, dnum);
                dden = fma(-(x + rvs), dk, dden);
            }
        } else {
            double k0, unused;
            ker.template eval<false>(x, &k0, &unused);
            den += k0;
            if (D) dnum = fma(dk, Fj, dnum);
        }
    };
    if (sp.sparse) {
        for (int64_t j = sp.b + g; j < sp.e; j += G) pair(nu[j], 1.0 / nu[j], F[j]);
        sp.last = sp.first;
    }
    for (int64_t t0 = sp.first; t0 < sp.last; t0 += RESP_TILE) {
        const int64_t t1 = min64(sp.last, t0 + RESP_TILE);
        __syncthreads();
        for (int64_t j = t0 + t; j < t1; j += RESP_THREADS) {
            const double v = nu[j];
            pv[j - t0] = v;
            pr[j - t0] = 1.0 / v;
            pf[j - t0] = F[j];
        }
        __syncthreads();
        const int jb = (int)(max(sp.b, t0) - t0), je = (int)(min64(sp.e, t1) - t0);
        for (int j = jb + g; j < je; j += G) pair(pv[j], pr[j], pf[j]);
    }
    num = group_sum<G>(num);
    den = group_sum<G>(den);
    if (D) {
        dnum = group_sum<G>(dnum) * inv;
        dden = group_sum<G>(dden) * inv;
    }
    double contrib = 0.0;
    if (live && g == 0) {
        const double o = num / den;
        if (out) out[i] = o;
        if (den_out) den_out[i] = den;
        if (D) contrib = g_out[i] * (dnum - o * dden) / den;
    }
    if (D) {
        red[t] = contrib;
        __syncthreads();
        for (int s = blockDim.x / 2; s > 0; s >>= 1) {
            if (t < s) red[t] += red[t + s];
            __syncthreads();
        }
        if (t == 0) part[blockIdx.x] = red[0];
    }
}

// g_F[j] = sum_i g_out[i] k(c ln(nu'_i/nu_j) + RV) / den[i]  (transpose of Eq. responsenu)
template <class K, int G, bool SMALL>
__global__ void __launch_bounds__(RESP_THREADS) response_transpose_kernel(
    const double* __restrict__ g_out, const double* __restrict__ den, const double* __restrict__ nu, int64_t N,
    const double* __restrict__ nu_out, int64_t No, K ker, PairConst kc, double* __restrict__ g_F)
{
    __shared__ double pv[RESP_TILE], pg[RESP_TILE];
    constexpr int OB = RESP_THREADS / G;
    const int t = threadIdx.x, g = t % G;
    const int64_t j0 = (int64_t)blockIdx.x * OB, j = j0 + t / G;
    const bool live = j < N;
    const double nuj = nu[live ? j : j0];
    Support sp{};
    sp.find<G>(nu_out, No, nuj * kc.lo, nuj * kc.hi, live);
    if (sp.first >= sp.last) { // sparse outputs leave most blocks without any
        if (live && g == 0) g_F[j] = 0.0;
        return;
    }
    const double rvs = kc.rvs, cinv = kc.cinv, rj = 1.0 / nuj;
    double s = 0.0;
    auto pair = [&](double v, double gd) {
        const double x = cinv * log_ratio<SMALL>(v, nuj, rj);
        double k, unused;
        ker.template eval<false>(x + rvs, &k, &unused);
        s = fma(gd, k, s);
    };
    if (sp.sparse) {
        for (int64_t i = sp.b + g; i < sp.e; i += G) pair(nu_out[i], g_out[i] / den[i]);
        sp.last = sp.first;
    }
    for (int64_t t0 = sp.first; t0 < sp.last; t0 += RESP_TILE) {
        const int64_t t1 = min64(sp.last, t0 + RESP_TILE);
        __syncthreads();
        for (int64_t i = t0 + t; i < t1; i += RESP_THREADS) {
            pv[i - t0] = nu_out[i];
            pg[i - t0] = g_out[i] / den[i];
        }
        __syncthreads();
        const int ib = (int)(max(sp.b, t0) - t0), ie = (int)(min64(sp.e, t1) - t0);
        for (int i = ib + g; i < ie; i += G) pair(pv[i], pg[i]);
    }
    s = group_sum<G>(s);
    if (live && g == 0) g_F[j] = s;
}

__global__ void sum_parts_kernel(const double* __restrict__ part, int64_t n, double* __restrict__ out)
{
    __shared__ double red[256];
    double a = 0.0;
    for (int64_t i = threadIdx.x; i < n; i += blockDim.x) a += part[i];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[0] = red[0];
}

} // namespace xsd

namespace {

using namespace xsd;

RotKernel rot_kernel(double vsini, double u1, double u2)
{
    RotKernel k;
    const double inv_norm = 1.0 / (PI * (1.0 - u1 / 3.0 - u2 / 6.0));
    k.scale = vsini;
    k.W = vsini;
    k.c1 = 2.0 * (1.0 - u1 - u2) * inv_norm;
    k.c2 = 0.5 * PI * (u1 + 2.0 * u2) * inv_norm;
    k.c3 = -(4.0 / 3.0) * u2 * inv_norm;
    return k;
}

GaussKernel gauss_kernel(double beta)
{
    GaussKernel k;
    k.scale = beta;
    k.W = GAUSS_SUPPORT * beta;
    return k;
}

// c ln(nu'_i/nu_j) in [v0, v1], as ends of nu_j (output points' supports) or, negated, of nu'_i
PairConst pair_const(double scale, double rv, double v0, double v1)
{
    const double inv = 1.0 / scale;
    return {inv, rv * inv, C_KMS * inv, std::exp(-v1 / C_KMS) * (1.0 - 1e-15), std::exp(-v0 / C_KMS) * (1.0 + 1e-15)};
}

// Lanes an output point: 4, so that a few thousand points already fill the GPU with
// blocks of 32; 16 for the shorter observed grids.
constexpr int64_t RESP_SHORT = 8192;
unsigned blocks(int64_t n)
{
    const int per = RESP_THREADS / (n < RESP_SHORT ? 16 : 4);
    return (unsigned)((n + per - 1) / per);
}

template <class K, bool D, int G>
void launch_response_g(const double* F, const double* nu, int64_t N, const double* nu_out, int64_t No, const K& k,
                       double rv, double* out, double* den, const double* g_out, double* part, cudaStream_t st)
{
    const PairConst kc = pair_const(k.scale, rv, std::fmin(-k.W - rv, -k.W), std::fmax(k.W - rv, k.W));
    if (k.W + fabs(rv) < RESP_SMALL_KMS)
        response_kernel<K, D, G, true>
            <<<blocks(No), RESP_THREADS, 0, st>>>(F, nu, N, nu_out, No, k, kc, out, den, g_out, part);
    else
        response_kernel<K, D, G, false>
            <<<blocks(No), RESP_THREADS, 0, st>>>(F, nu, N, nu_out, No, k, kc, out, den, g_out, part);
}

template <class K, bool D>
void launch_response(const double* F, const double* nu, int64_t N, const double* nu_out, int64_t No, const K& k,
                     double rv, double* out, double* den, const double* g_out, double* part, cudaStream_t st)
{
    if (No < RESP_SHORT)
        launch_response_g<K, D, 16>(F, nu, N, nu_out, No, k, rv, out, den, g_out, part, st);
    else
        launch_response_g<K, D, 4>(F, nu, N, nu_out, No, k, rv, out, den, g_out, part, st);
}

template <class K, int G>
void launch_transpose_g(const double* g_out, const double* den, const double* nu, int64_t N, const double* nu_out,
                        int64_t No, const K& k, double rv, double* g_F, cudaStream_t st)
{
    // c ln(nu'_i/nu_j) + rv in [-W, W]  <=>  nu'_i in [nu_j e^{(-W - rv)/c}, nu_j e^{(W - rv)/c}]
    const PairConst kc = pair_const(k.scale, rv, -k.W + rv, k.W + rv);
    if (k.W + fabs(rv) < RESP_SMALL_KMS)
        response_transpose_kernel<K, G, true>
            <<<blocks(N), RESP_THREADS, 0, st>>>(g_out, den, nu, N, nu_out, No, k, kc, g_F);
    else
        response_transpose_kernel<K, G, false>
            <<<blocks(N), RESP_THREADS, 0, st>>>(g_out, den, nu, N, nu_out, No, k, kc, g_F);
}

template <class K>
void launch_transpose(const double* g_out, const double* den, const double* nu, int64_t N, const double* nu_out,
                      int64_t No, const K& k, double rv, double* g_F, cudaStream_t st)
{
    if (N < RESP_SHORT)
        launch_transpose_g<K, 16>(g_out, den, nu, N, nu_out, No, k, rv, g_F, st);
    else
        launch_transpose_g<K, 4>(g_out, den, nu, N, nu_out, No, k, rv, g_F, st);
}

size_t al256(size_t b) { return (b + 255) / 256 * 256; }

bool grid_ok(const double* nu, int64_t N) { return nu != nullptr && N >= 1; }

int finish(int n_launch)
{
    xsi::count_launch(n_launch);
    return cudaGetLastError() == cudaSuccess ? XS_OK : XS_ECUDA;
}

} // namespace

extern "C" {

int response_rotation(const double* F0, const double* nu, int64_t N, double vsini, double u1, double u2, double* F1,
                      xs_stream stream)
{
    XS_NVTX("response_rotation");
    if (!F0 || !F1 || !grid_ok(nu, N) || !(vsini > 0.0) || !(1.0 - u1 / 3.0 - u2 / 6.0 > 0.0)) return XS_EINVAL;
    launch_response<RotKernel, false>(F0, nu, N, nu, N, rot_kernel(vsini, u1, u2), 0.0, F1, nullptr, nullptr, nullptr,
                                      (cudaStream_t)stream);
    return finish(1);
}

int response_ip_rv(const double* F1, const double* nu, int64_t N, const double* nu_out, int64_t N_out, double beta,
                   double rv, double* F, xs_stream stream)
{
    XS_NVTX("response_ip_rv");
    if (!F1 || !F || !grid_ok(nu, N) || !grid_ok(nu_out, N_out) || !(beta > 0.0) || !(fabs(rv) < C_KMS))
        return XS_EINVAL;
    launch_response<GaussKernel, false>(F1, nu, N, nu_out, N_out, gauss_kernel(beta), rv, F, nullptr, nullptr, nullptr,
                                        (cudaStream_t)stream);
    return finish(1);
}

size_t response_workspace_bytes(int64_t N_out)
{
    if (N_out <= 0) return 0;
    // a partial a block; grids of RESP_SHORT points and a little more have fewer blocks than
    // shorter ones, and a workspace that serves a grid serves every shorter one too
    const size_t parts = std::max(blocks(N_out), blocks(std::min(N_out, RESP_SHORT - 1)));
    return al256(sizeof(double) * (size_t)N_out) + al256(sizeof(double) * parts);
}

int response_rotation_adjoint(const double* g_F1, const double* F0, const double* nu, int64_t N, double vsini,
                              double u1, double u2, double* g_F0, double* g_vsini, void* workspace,
                              size_t workspace_bytes, xs_stream stream)
{
    XS_NVTX("response_rotation_adjoint");
    if (!g_F1 || !F0 || !g_F0 || !g_vsini || !workspace || !grid_ok(nu, N) || !(vsini > 0.0) ||
        !(1.0 - u1 / 3.0 - u2 / 6.0 > 0.0))
        return XS_EINVAL;
    if (workspace_bytes < response_workspace_bytes(N)) return XS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    double* den = (double*)workspace;
    double* part = (double*)((char*)workspace + al256(sizeof(double) * (size_t)N));
    const RotKernel k = rot_kernel(vsini, u1, u2);
    launch_response<RotKernel, true>(F0, nu, N, nu, N, k, 0.0, nullptr, den, g_F1, part, st);
    sum_parts_kernel<<<1, 256, 0, st>>>(part, blocks(N), g_vsini);
    launch_transpose(g_F1, den, nu, N, nu, N, k, 0.0, g_F0, st);
    return finish(3);
}

int response_ip_rv_adjoint(const double* g_F, const double* F1, const double* nu, int64_t N, const double* nu_out,
                           int64_t N_out, double beta, double rv, double* g_F1, double* g_rv, void* workspace,
                           size_t workspace_bytes, xs_stream stream)
{
    XS_NVTX("response_ip_rv_adjoint");
    if (!g_F || !F1 || !g_F1 || !g_rv || !workspace || !grid_ok(nu, N) || !grid_ok(nu_out, N_out) ||
        !(beta > 0.0) || !(fabs(rv) < C_KMS))
        return XS_EINVAL;
    if (workspace_bytes < response_workspace_bytes(N_out)) return XS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    double* den = (double*)workspace;
    double* part = (double*)((char*)workspace + al256(sizeof(double) * (size_t)N_out));
    const GaussKernel k = gauss_kernel(beta);
    launch_response<GaussKernel, true>(F1, nu, N, nu_out, N_out, k, rv, nullptr, den, g_F, part, st);
    sum_parts_kernel<<<1, 256, 0, st>>>(part, blocks(N_out), g_rv);
    launch_transpose(g_F, den, nu, N, nu_out, N_out, k, rv, g_F1, st);
    return finish(3);
}

} // extern "C"

XS_CHECK_ACCESSOR(resp)
