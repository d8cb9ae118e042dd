// MODIT (Sec. 2.1.2, Eq. MODIT): the cross-section of many lines through a
// lineshape distribution on the log grid and FFT convolution.
//
// Grid: nu_i = nu_min exp(i/R0), i = 0..N-1, R0 = (N-1)/ln(nu_max/nu_min), so the
// variable q = R0 ln(nu/nu_min) steps by 1.  For each layer:
//   1. per line, once, q_l = R0 ln(nu_hat/nu_min) and the layer-independent parts of S(T)
//      and ln gamma' (modit_prepass_kernel); per layer the min and max of ln gamma',
//      gamma' = R0 gamma/nu_hat (modit_range_kernel), and the layer's constants
//      (modit_layer_kernel);
//   2. the lineshape distribution S[k][j]: each line adds S(T) (Eq. Slog) to the
//      two q nodes around q_l and the two ln gamma' nodes around its width, with
//      linear weights (modit_lsd_kernel).  One thread per q node takes the lines
//      with floor(q_l) = j (binary search) and hands the upper node's share to its
//      neighbour through shared memory, so the sum has a fixed order (no atomics);
//   3. batched real FFTs of the n_gamma rows (cuFFT);
//   4. Y[f] = sum_k FT(S_k)[f] K_k[f], K_k = exp(-2 pi^2 beta'^2 f^2)
//      (exp(-2 pi gamma'_k |f|) - gamma'_k DFT(A)[f]), beta' = R0 beta/nu_hat (common
//      to all lines of a species at one T), A the sum of a unit Lorentzian's periodic
//      images (its first-order aliasing, removed here);
//   5. inverse FFT per layer, then sigma(nu_i) = sigma(q_i) R0/nu_i.
// The q axis is periodic with the caller's length n_fft (a power of two); node j
// lives at slot j mod n_fft, nodes -(n_fft-N)/2 .. (n_fft+N)/2 - 1 are gathered.
//
// FP64 runs at 2 lanes a clock and SM here and bounds every kernel of this file but the
// last ones: layer constants are formed once a layer, exponentials along the frequency
// axis are advanced by multiplication, and the adjoint of a composite call takes the
// distribution's transform from the forward instead of forming it again.  (220,000 lines,
// 100 layers, n_fft 65,536, FP64: forward + gradient step 125.5 -> 50.4 ms, the kernels of
// this file 73 -> 15 ms of it; the rest are the FFTs, 51 -> 34 ms.)
#include <cufft.h>

#include <map>
#include <mutex>
#include <tuple>
#include <type_traits>

#include "xs_device.cuh"
#include "xs_internal.h"

namespace xsd {

constexpr int MODIT_MAX_GAMMA = 32;
constexpr int MODIT_THREADS = 128;

template <class R> struct CplxOf;
template <> struct CplxOf<double> { using type = cufftDoubleComplex; };
template <> struct CplxOf<float> { using type = cufftComplex; };

// Constants of a layer; the first part from T and P alone, the second from the range of
// ln gamma' (modit_layer_kernel).
struct ModitLayer {
    double lnTr, kE, kq, lgP, T, uT; // ln(T/296), c2 (1/T - 1/296), q ln(T/296), ln(sb P/atm), T, c2/T
    double lg0, dlg, idlg;           // first gamma' node and node step (ln), its inverse (0 if there is one node)
    double gauss, bT;                // -2 pi^2 beta'^2, c2/T^2
    double n_lo, n_hi;               // temperature exponents of the extreme lines (adjoint)
    double g[MODIT_MAX_GAMMA];       // gamma' nodes
    unsigned long long range[2], ext[2];
};

// doubles in the order of unsigned integers
__device__ __forceinline__ unsigned long long ordered(double v)
{
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return b ^ ((b >> 63) ? ~0ull : 1ull << 63);
}
__device__ __forceinline__ double unordered(unsigned long long k)
{
    return __longlong_as_double((long long)(k ^ ((k >> 63) ? 1ull << 63 : ~0ull)));
}

__global__ void modit_layer_init_kernel(const double* __restrict__ T, const double* __restrict__ P, double sb,
                                        double qexp, int L, ModitLayer* __restrict__ lay)
{
    const int n = blockIdx.x * blockDim.x + threadIdx.x;
    if (n >= L) return;
    ModitLayer& y = lay[n];
    const double Tn = T[n], lnTr = log(Tn / Tref);
    y.lnTr = lnTr;
    y.kE = c2 * (1.0 / Tn - 1.0 / Tref);
    y.kq = qexp * lnTr;
    y.lgP = log(sb * P[n] / bar_per_atm);
    y.T = Tn;
    y.uT = c2 / Tn;
    y.bT = c2 / (Tn * Tn);
    y.range[0] = y.ext[0] = y.ext[1] = ~0ull;
    y.range[1] = 0ull;
}

// ln gamma' of a line without the layer's ln(sb P), the same operations everywhere
__device__ __forceinline__ double line_lg(double lgref, double n_temp, double lnTr) { return fma(-n_temp, lnTr, lgref); }

constexpr int MODIT_LINES = 4; // lines a thread of the (line, layer) kernels takes

// per layer min and max of ln gamma' (two operations a line)
__global__ void modit_range_kernel(const double* __restrict__ lgref, const double* __restrict__ n_temp, int64_t nl,
                                   ModitLayer* __restrict__ lay)
{
    ModitLayer& y = lay[blockIdx.y];
    const double lnTr = y.lnTr;
    double lo = __longlong_as_double(0x7ff0000000000000ll), hi = -lo;
    for (int r = 0; r < MODIT_LINES; ++r) {
        const int64_t l = ((int64_t)blockIdx.x * MODIT_LINES + r) * blockDim.x + threadIdx.x;
        if (l >= nl) break;
        const double g = line_lg(lgref[l], n_temp[l], lnTr);
        lo = fmin(lo, g);
        hi = fmax(hi, g);
    }
    __syncwarp();
    for (int o = 16; o > 0; o >>= 1) {
        lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
        hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
    }
    if ((threadIdx.x & 31) == 0 && lo <= hi) {
        atomicMin(&y.range[0], ordered(lo));
        atomicMax(&y.range[1], ordered(hi));
    }
}

// index of the line attaining the layer's smallest and largest gamma'
__global__ void modit_extreme_kernel(const double* __restrict__ lgref, const double* __restrict__ n_temp, int64_t nl,
                                     ModitLayer* __restrict__ lay)
{
    ModitLayer& y = lay[blockIdx.y];
    const double lnTr = y.lnTr;
    const unsigned long long r0 = y.range[0], r1 = y.range[1];
    for (int r = 0; r < MODIT_LINES; ++r) {
        const int64_t l = ((int64_t)blockIdx.x * MODIT_LINES + r) * blockDim.x + threadIdx.x;
        if (l >= nl) return;
        const unsigned long long g = ordered(line_lg(lgref[l], n_temp[l], lnTr));
        if (g == r0) atomicMin(&y.ext[0], (unsigned long long)l);
        if (g == r1) atomicMin(&y.ext[1], (unsigned long long)l);
    }
}

// the layer's gamma' nodes (thread k: node k) and, with n_temp, the extreme lines' exponents
__global__ void modit_layer_kernel(int ng, double mass, double R0, const double* __restrict__ n_temp, int64_t nl,
                                   ModitLayer* __restrict__ lay)
{
    ModitLayer& y = lay[blockIdx.x];
    const int k = threadIdx.x;
    const double lo = unordered(y.range[0]), hi = unordered(y.range[1]);
    const double dlg = (ng >= 2 && hi > lo) ? (hi - lo) / (double)(ng - 1) : 0.0;
    if (k < ng) y.g[k] = exp(lo + y.lgP + dlg * (double)k);
    if (k == 0) {
        y.lg0 = lo;
        y.dlg = dlg;
        y.idlg = dlg > 0.0 ? 1.0 / dlg : 0.0;
        const double bq = sqrt(kB * y.T / (mass * amu)) * R0 / cL; // beta' (q units)
        y.gauss = -2.0 * PI * PI * bq * bq;
        if (n_temp) {
            y.n_lo = n_temp[min(y.ext[0], (unsigned long long)(nl - 1))];
            y.n_hi = n_temp[min(y.ext[1], (unsigned long long)(nl - 1))];
        }
    }
}

// 1 - e^-u, u >= 0, given e = e^-u
__device__ __forceinline__ double one_minus(double u, double e) { return u < 0.5 ? -expm1(-u) : 1.0 - e; }

// Layer-independent per-line terms: q = R0 ln(nu_hat/nu_min), the inverse stimulated-
// emission denominator 1/(1 - e^(-c2 nu_hat/296)) and ln(R0 gamma_ref/nu_hat).
__global__ void modit_prepass_kernel(const double* __restrict__ nu_hat, const double* __restrict__ gamma_ref,
                                     int64_t nl, double nu_min, double R0, double* __restrict__ qv,
                                     double* __restrict__ sinv, double* __restrict__ lgref)
{
    const int64_t l = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (l >= nl) return;
    const double nuh = nu_hat[l];
    qv[l] = R0 * log(nuh / nu_min);
    sinv[l] = -1.0 / expm1(-c2 * nuh / Tref);
    lgref[l] = log(R0 * gamma_ref[l] / nuh);
}

__device__ __forceinline__ int64_t first_at_least(const double* v, int64_t n, double x) // first i with v[i] >= x
{
    int64_t lo = 0, hi = n;
    while (lo < hi) {
        const int64_t m = (lo + hi) >> 1;
        if (v[m] >= x) hi = m; else lo = m + 1;
    }
    return lo;
}

// One thread per (layer, slot); node j = slot, or slot - M for the left padding.
// Each thread takes the lines with floor(q_l) == j (found by binary search on
// the monotone q_l of the prepass), so every line is visited once: weight 1 - w
// goes to node j, w to node j + 1 through shared memory (the slot before the
// block's first comes from an extra halo thread).  Per line and layer: S(T)
// (Eq. Slog) from two exponentials, ln gamma' from the prepass by one FMA.
// Blocks of MODIT_THREADS threads write MODIT_THREADS - 1 slots.
template <class R>
__global__ void __launch_bounds__(MODIT_THREADS) modit_lsd_kernel(
    const double* __restrict__ nu_hat, const double* __restrict__ ln_S0, const double* __restrict__ elower,
    const double* __restrict__ n_temp, const double* __restrict__ qv, const double* __restrict__ sinv,
    const double* __restrict__ lgref, int64_t nl, double scale, int64_t N, int64_t M, int ng,
    const ModitLayer* __restrict__ lay, R* __restrict__ lsd)
{
    __shared__ double shR[MODIT_THREADS][MODIT_MAX_GAMMA + 1]; // odd rows: the lanes' rows on different banks
    const int t = threadIdx.x;
    const int n = blockIdx.y;
    const int64_t s_raw = (int64_t)blockIdx.x * (MODIT_THREADS - 1) + t - 1;
    const bool valid = s_raw < M;
    const int64_t s = (s_raw + M) % M; // the halo of block 0 is slot M - 1
    const int64_t j = (s < (M + N) / 2) ? s : s - M;
    int64_t b = 0, e = 0;
    if (valid && nl > 0 && (double)(j + 1) > qv[0] && (double)j <= qv[nl - 1]) { // a slot without lines searches nothing
        b = first_at_least(qv, nl, (double)j);
        e = first_at_least(qv, nl, (double)(j + 1));
    }
    // most slots of the padding are empty: such a block writes zeros
    if (!__syncthreads_or(e > b)) {
        if (t >= 1 && valid)
            for (int k = 0; k < ng; ++k) lsd[((size_t)n * ng + k) * M + s] = R(0);
        return;
    }
    double accL[MODIT_MAX_GAMMA];
    for (int k = 0; k < ng; ++k) {
        accL[k] = 0.0;
        shR[t][k] = 0.0;
    }
    const ModitLayer& y = lay[n];
    const double lnTr = y.lnTr, kE = y.kE, kq = y.kq, uT = y.uT, lg0 = y.lg0, idlg = y.idlg;
    for (int64_t l = b; l < e; ++l) {
        const double wq = qv[l] - (double)j;
        const double u = uT * nu_hat[l];
        const double S = exp_tab(fma(-elower[l], kE, ln_S0[l]) - kq) * (one_minus(u, exp_tab(-u)) * sinv[l]) * scale;
        int k0 = 0;
        double wk = 0.0;
        if (idlg > 0.0) {
            const double tt = (line_lg(lgref[l], n_temp[l], lnTr) - lg0) * idlg;
            k0 = min(max((int)floor(tt), 0), ng - 2);
            wk = tt - (double)k0;
        }
        const double vl = S * (1.0 - wq), vr = S * wq;
        accL[k0] += vl * (1.0 - wk);
        shR[t][k0] += vr * (1.0 - wk);
        if (idlg > 0.0) {
            accL[k0 + 1] += vl * wk;
            shR[t][k0 + 1] += vr * wk;
        }
    }
    __syncthreads();
    if (t >= 1 && valid)
        for (int k = 0; k < ng; ++k) lsd[((size_t)n * ng + k) * M + s] = (R)(accL[k] + shR[t - 1][k]);
}

// A(d) = sum over p != 0 of 1/(pi (d + pM)^2) on one period (index d mod M):
// (pi/M)^2/sin^2(pi d/M) - 1/d^2 over pi, near d = 0 from the Laurent series of csc^2.
template <class R>
__global__ void modit_images_kernel(int64_t M, R* __restrict__ A)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= M) return;
    const double d = (i < M / 2) ? (double)i : (double)(i - M);
    const double x = PI * d / (double)M;
    double v;
    if (fabs(x) < 0.3) {
        const double x2 = x * x;
        v = (PI / ((double)M * (double)M)) *
            (1.0 / 3 + x2 * (1.0 / 15 + x2 * (2.0 / 189 + x2 * (1.0 / 675 + x2 * (2.0 / 10395)))));
    } else {
        const double sx = sin(x);
        v = ((PI / M) * (PI / M) / (sx * sx) - 1.0 / (d * d)) / PI;
    }
    A[i] = (R)v;
}

// A thread's frequencies lie MODIT_STEP apart: e^(-2 pi gamma'_k f) is advanced from one to
// the next by a product.  Blocks of 64 threads: with 256, short transforms of a few layers had
// one to a few blocks, whose FP64 operations waited for one SM's pipe (FP32, 2,000 lines on
// 1,000 points, one layer 174 -> 131 us; 20,000 x 5 layers with the adjoint 552 -> 441).
constexpr int MODIT_STEP = 64;

// Y[n][m] = sum_k Z[n][k][m] K_k(m) for m = 0..M/2
template <class R, int F>
__global__ void __launch_bounds__(MODIT_STEP) modit_multiply_kernel(const typename CplxOf<R>::type* __restrict__ Z,
                                                                    const typename CplxOf<R>::type* __restrict__ Ahat,
                                                                    int64_t M, int ng,
                                                                    const ModitLayer* __restrict__ lay,
                                                                    typename CplxOf<R>::type* __restrict__ Y)
{
    const int n = blockIdx.y;
    const ModitLayer& y = lay[n];
    const int64_t H = M / 2 + 1, m0 = (int64_t)blockIdx.x * (MODIT_STEP * F) + threadIdx.x;
    const double f0 = (double)m0 / (double)M;
    double ah[F], yr[F], yi[F];
#pragma unroll
    for (int i = 0; i < F; ++i) {
        const int64_t m = m0 + MODIT_STEP * i;
        ah[i] = m < H ? (double)Ahat[m].x : 0.0;
        yr[i] = yi[i] = 0.0;
    }
    for (int k = 0; k < ng; ++k) {
        const double g = y.g[k], step = exp_tab(-2.0 * PI * g * ((double)MODIT_STEP / (double)M));
        double E = exp_tab(-2.0 * PI * g * f0);
#pragma unroll
        for (int i = 0; i < F; ++i) {
            const int64_t m = m0 + MODIT_STEP * i;
            if (m < H) {
                const double K = fma(-g, ah[i], E);
                const typename CplxOf<R>::type z = Z[((size_t)n * ng + k) * H + m];
                yr[i] = fma((double)z.x, K, yr[i]);
                yi[i] = fma((double)z.y, K, yi[i]);
            }
            E *= step;
        }
    }
#pragma unroll
    for (int i = 0; i < F; ++i) {
        const int64_t m = m0 + MODIT_STEP * i;
        if (m >= H) break;
        const double f = (double)m / (double)M, G = exp_tab(y.gauss * f * f);
        Y[(size_t)n * H + m].x = (R)(G * yr[i]);
        Y[(size_t)n * H + m].y = (R)(G * yi[i]);
    }
}

template <class R>
__global__ void modit_finish_kernel(const R* __restrict__ y, int64_t M, int64_t N, int L, double R0, double nu_min,
                                    double unscale, void* __restrict__ sigma)
{
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int n = blockIdx.y;
    if (i >= N) return;
    const double nu = nu_min * exp((double)i / R0);
    const double v = (double)y[(size_t)n * M + i] / (double)M * R0 / nu * unscale;
    if (std::is_same<R, float>::value) ((float*)sigma)[(size_t)n * N + i] = (float)v;
    else ((double*)sigma)[(size_t)n * N + i] = v;
}


// ------------------------------------------------------------------ adjoint
//
// With lambda = dF/dsigma [L][N] and mu_i = lambda_i R0 unscale/(M nu_i) (so that
// F = sum_i mu_i y_i, y the unnormalised inverse transform), per layer:
//   M^ = FFT(mu); the kernel term sum_m c_m Re(Z_k[m] conj(M^[m])) dK_k[m]/dtheta
//   (c_m = 1 at m = 0 and M/2, else 2); the correlations corr_k = IFFT(K_k M^),
//   so that dF/dLSD_k[j] = corr_k[j]; and per line the distribution term
//   S (dlnS/dT A + B dt/dT), A and B the weight-averaged correlations and their
//   difference across the two gamma' nodes, t the line's fractional gamma' node.
// s_b moves every ln gamma' and both grid ends alike, so it enters through the
// kernels only.

__device__ __forceinline__ double block_sum(double v, double* red)
{
    red[threadIdx.x] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    const double r = red[0];
    __syncthreads();
    return r;
}

template <class R>
__global__ void modit_mu_kernel(const double* __restrict__ g_sigma, int64_t N, int64_t M, double R0, double nu_min,
                                double fac, R* __restrict__ mu)
{
    const int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const int n = blockIdx.y;
    if (s >= M) return;
    double v = 0.0;
    if (s < N) v = g_sigma[(size_t)n * N + s] * R0 / (nu_min * exp((double)s / R0)) * fac;
    mu[(size_t)n * M + s] = (R)v;
}

// Kernel term (per layer, block partials) and X_k = K_k M^ for the correlations.  With
// e = E - g A^ and d = g (2 pi f E + A^): K = G e, dK/d ln gamma' = -G d, dK/dT|_G = -G' e;
// d ln gamma'_k/dT = -((1 - k w) n_lo + k w n_hi)/T, w = 1/(ng - 1).
template <class R, int F>
__global__ void __launch_bounds__(MODIT_STEP) modit_adj_kernel_term(
    const typename CplxOf<R>::type* __restrict__ Z, typename CplxOf<R>::type* __restrict__ X,
    const typename CplxOf<R>::type* __restrict__ Mh, const typename CplxOf<R>::type* __restrict__ Ahat, int64_t M,
    int ng, double sb, const ModitLayer* __restrict__ lay, double* __restrict__ partT, double* __restrict__ partB)
{
    __shared__ double red[MODIT_STEP];
    const int n = blockIdx.y;
    const ModitLayer& y = lay[n];
    const int64_t H = M / 2 + 1, m0 = (int64_t)blockIdx.x * (MODIT_STEP * F) + threadIdx.x;
    const double f0 = (double)m0 / (double)M, df = (double)MODIT_STEP / (double)M;
    double mr[F], mi[F], ah[F], G[F], sumE[F];
#pragma unroll
    for (int i = 0; i < F; ++i) {
        const int64_t m = m0 + MODIT_STEP * i;
        const bool in = m < H;
        const double f = (double)m / (double)M;
        ah[i] = in ? (double)Ahat[m].x : 0.0;
        mr[i] = in ? (double)Mh[(size_t)n * H + m].x : 0.0;
        mi[i] = in ? (double)Mh[(size_t)n * H + m].y : 0.0;
        G[i] = in ? exp_tab(y.gauss * f * f) : 0.0;
        sumE[i] = 0.0;
    }
    double s0 = 0.0, s1 = 0.0; // sums over k and f of c G d Re(Z conj M^), times 1 and k
    for (int k = 0; k < ng; ++k) {
        const double g = y.g[k], step = exp_tab(-2.0 * PI * g * df);
        double E = exp_tab(-2.0 * PI * g * f0), t = 0.0;
#pragma unroll
        for (int i = 0; i < F; ++i) {
            const int64_t m = m0 + MODIT_STEP * i;
            if (m < H) {
                const size_t zi = ((size_t)n * ng + k) * H + m;
                const typename CplxOf<R>::type z = Z[zi];
                const double Pk = fma((double)z.x, mr[i], (double)z.y * mi[i]);
                const double e = fma(-g, ah[i], E), K = G[i] * e;
                const double d = g * fma(2.0 * PI * fma((double)i, df, f0), E, ah[i]);
                const double c = (m == 0 || 2 * m == M) ? 1.0 : 2.0;
                sumE[i] = fma(Pk, e, sumE[i]);
                t = fma(c * G[i] * d, Pk, t);
                X[zi].x = (R)(K * mr[i]);
                X[zi].y = (R)(K * mi[i]);
            }
            E *= step;
        }
        s0 += t;
        s1 = fma((double)k, t, s1);
    }
    double gT = 0.0;
#pragma unroll
    for (int i = 0; i < F; ++i) {
        const int64_t m = m0 + MODIT_STEP * i;
        if (m >= H) break;
        const double f = fma((double)i, df, f0), c = (m == 0 || 2 * m == M) ? 1.0 : 2.0;
        gT = fma(c * G[i] * (y.gauss * f * f), sumE[i], gT); // dG/dT = G gauss f^2/T
    }
    const double w = ng >= 2 ? 1.0 / (double)(ng - 1) : 0.0;
    gT = (gT + s0 * y.n_lo + s1 * w * (y.n_hi - y.n_lo)) / y.T;
    const double sT = block_sum(gT, red), sB = block_sum(-s0 / sb, red);
    if (threadIdx.x == 0) {
        partT[(size_t)n * gridDim.x + blockIdx.x] = sT;
        partB[(size_t)n * gridDim.x + blockIdx.x] = sB;
    }
}

// distribution term per (line, layer), block partials; corr rows have M + 2 values
template <class R>
__global__ void __launch_bounds__(256) modit_adj_line_term(
    const double* __restrict__ nu_hat, const double* __restrict__ ln_S0, const double* __restrict__ elower,
    const double* __restrict__ n_temp, const double* __restrict__ qv, const double* __restrict__ sinv,
    const double* __restrict__ lgref, int64_t nl, double qexp, double scale, int64_t N, int64_t M, int ng,
    const ModitLayer* __restrict__ lay, const R* __restrict__ corr, double* __restrict__ part)
{
    __shared__ double red[256];
    const int n = blockIdx.y;
    const ModitLayer& y = lay[n];
    const double lnTr = y.lnTr, kE = y.kE, kq = y.kq, uT = y.uT, lg0 = y.lg0, dlg = y.dlg, idlg = y.idlg, bT = y.bT;
    const double iT = 1.0 / y.T, qT = qexp * iT;
    // node slopes: t = (lg - lg0)/dlg, dt/dT = (-n/T - dlg0 - t ddlg)/dlg
    const double dlg0 = -y.n_lo * iT, ddlg = ng >= 2 ? (y.n_lo - y.n_hi) * iT / (double)(ng - 1) : 0.0;
    // the forward gathers lines whose lower node j0 lies in the window
    // -(M-N)/2 .. (M+N)/2 - 1 and adds to the slots of j0 and j0 + 1 (mod M)
    const int64_t jlo = -(M - N) / 2, jhi = (M + N) / 2;
    double gl = 0.0;
    for (int r = 0; r < MODIT_LINES; ++r) {
        const int64_t l = ((int64_t)blockIdx.x * MODIT_LINES + r) * 256 + threadIdx.x;
        if (l >= nl) break;
        const double q = qv[l], fq = floor(q), wq = q - fq;
        const int64_t j0 = (int64_t)fq;
        if (j0 < jlo || j0 >= jhi) continue;
        const double u = uT * nu_hat[l], eu = exp_tab(-u), om = one_minus(u, eu);
        const double S = exp_tab(fma(-elower[l], kE, ln_S0[l]) - kq) * (om * sinv[l]) * scale;
        const double dlnS = fma(elower[l], bT, -qT) - (u * iT) * (eu / om);
        int k0 = 0;
        double wk = 0.0, dt = 0.0;
        if (dlg > 0.0) {
            const double t = (line_lg(lgref[l], n_temp[l], lnTr) - lg0) * idlg;
            k0 = min(max((int)floor(t), 0), ng - 2);
            wk = t - (double)k0;
            dt = (-n_temp[l] * iT - dlg0 - t * ddlg) * idlg;
        }
        const int k1 = (dlg > 0.0) ? k0 + 1 : 0;
        double A = 0.0, B = 0.0;
#pragma unroll
        for (int d = 0; d < 2; ++d) {
            int64_t sl = j0 + d; // in -(M-N)/2 .. (M+N)/2
            if (sl < 0) sl += M;
            else if (sl >= M) sl -= M;
            const double w = d ? wq : 1.0 - wq;
            const double c0 = (double)corr[((size_t)n * ng + k0) * (M + 2) + sl];
            const double c1 = (double)corr[((size_t)n * ng + k1) * (M + 2) + sl];
            A += w * ((1.0 - wk) * c0 + wk * c1);
            B += w * (c1 - c0);
        }
        gl = fma(S, fma(dlnS, A, B * dt), gl);
    }
    gl = block_sum(gl, red);
    if (threadIdx.x == 0) part[(size_t)n * gridDim.x + blockIdx.x] = gl;
}

// g_T[n] = sum of the layer's line and kernel partials, gbl[n] the s_b kernel
// partials (one block per layer, fixed order)
__global__ void __launch_bounds__(256) modit_adj_reduce(const double* __restrict__ partL, int nbl,
                                                        const double* __restrict__ partT,
                                                        const double* __restrict__ partB, int nbk,
                                                        double* __restrict__ g_T, double* __restrict__ gbl)
{
    __shared__ double red[256];
    const int n = blockIdx.x;
    double a = 0.0, b = 0.0;
    for (int i = threadIdx.x; i < nbl; i += blockDim.x) a += partL[(size_t)n * nbl + i];
    for (int i = threadIdx.x; i < nbk; i += blockDim.x) {
        a += partT[(size_t)n * nbk + i];
        b += partB[(size_t)n * nbk + i];
    }
    a = block_sum(a, red);
    b = block_sum(b, red);
    if (threadIdx.x == 0) {
        g_T[n] = a;
        gbl[n] = b;
    }
}

// g_b = sum over layers (one warp, fixed order)
__global__ void modit_broad_sum(const double* __restrict__ gbl, int L, double* __restrict__ g_b)
{
    double s = 0.0;
    for (int n = threadIdx.x; n < L; n += 32) s += gbl[n];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (threadIdx.x == 0) g_b[0] = s;
}

} // namespace xsd

namespace {

using namespace xsd;

size_t al256(size_t b) { return (b + 255) / 256 * 256; }

// frequencies a thread of the forward's and the adjoint's product takes
constexpr int MODIT_F = 8, MODIT_F_ADJ = 4;

struct ModitPlan {
    size_t range, lines, lsd, Z, A, Ahat, Y, work, total, work_bytes;
    size_t mu, gbl, partL, partT, partB; // adjoint only
    int nbl, nbk;
};

ModitPlan modit_plan(int64_t nl, int32_t L, int32_t ng, int64_t M, int prec, bool adjoint = false)
{
    const size_t rs = (prec == XS_PREC_MIXED) ? sizeof(float) : sizeof(double);
    const size_t H = (size_t)M / 2 + 1;
    ModitPlan p{};
    size_t off = 0;
    auto take = [&](size_t b) {
        size_t o = off;
        off += al256(b);
        return o;
    };
    p.range = take(sizeof(ModitLayer) * (size_t)L);
    p.lines = take(3 * sizeof(double) * (size_t)std::max<int64_t>(nl, 1)); // q, 1/stim denominator, ln gamma'_ref
    p.lsd = take(rs * (size_t)L * ng * (M + 2)); // reused: the inverse transforms' output, the adjoint's X_k in place
    p.Z = take(2 * rs * (size_t)L * ng * H);
    p.A = take(rs * (size_t)M);
    p.Ahat = take(2 * rs * H);
    p.Y = take(2 * rs * (size_t)L * H);
    // cuFFT work area: reserved at the size of the largest complex array
    p.work_bytes = std::max<size_t>((size_t)16 << 20, 2 * rs * (size_t)L * ng * H);
    p.work = take(p.work_bytes);
    if (adjoint) {
        p.nbl = (int)((std::max<int64_t>(nl, 1) + 256 * MODIT_LINES - 1) / (256 * MODIT_LINES));
        p.nbk = (int)((H + MODIT_STEP * MODIT_F_ADJ - 1) / (MODIT_STEP * MODIT_F_ADJ));
        p.mu = take(rs * (size_t)L * M);
        p.gbl = take(sizeof(double) * (size_t)L);
        p.partL = take(sizeof(double) * (size_t)L * p.nbl);
        p.partT = take(sizeof(double) * (size_t)L * p.nbk);
        p.partB = take(sizeof(double) * (size_t)L * p.nbk);
    }
    p.total = off;
    return p;
}

// cuFFT plans, created once per (device, length, batch, type) without their own
// work area (the caller's workspace provides it).
std::mutex g_fft_mu;
std::map<std::tuple<int, int64_t, int64_t, int, bool>, std::pair<cufftHandle, size_t>> g_fft_plans;

// in_place: the real rows are padded to M + 2 values, as the complex ones
int fft_plan(int64_t M, int64_t batch, cufftType type, bool in_place, cufftHandle* out, size_t* work)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return XS_ECUDA;
    auto key = std::make_tuple(dev, M, batch, (int)type, in_place);
    auto it = g_fft_plans.find(key);
    if (it != g_fft_plans.end()) {
        *out = it->second.first;
        *work = it->second.second;
        return XS_OK;
    }
    cufftHandle h;
    if (cufftCreate(&h) != CUFFT_SUCCESS) return XS_ECUDA;
    if (cufftSetAutoAllocation(h, 0) != CUFFT_SUCCESS) return XS_ECUDA;
    long long n = M;
    size_t ws = 0;
    const bool fwd = (type == CUFFT_D2Z || type == CUFFT_R2C);
    const long long real = in_place ? M + 2 : M;
    long long idist = fwd ? real : M / 2 + 1, odist = fwd ? M / 2 + 1 : real;
    if (cufftMakePlanMany64(h, 1, &n, nullptr, 1, idist, nullptr, 1, odist, type, batch, &ws) != CUFFT_SUCCESS) {
        cufftDestroy(h);
        return XS_ECUDA;
    }
    g_fft_plans[key] = {h, ws};
    *out = h;
    *work = ws;
    return XS_OK;
}

template <class R>
int fft_exec(int64_t M, int64_t batch, bool forward, void* in, void* out, void* work, size_t work_bytes,
             cudaStream_t st)
{
    constexpr bool D = std::is_same<R, double>::value;
    const cufftType type = forward ? (D ? CUFFT_D2Z : CUFFT_R2C) : (D ? CUFFT_Z2D : CUFFT_C2R);
    std::lock_guard<std::mutex> lk(g_fft_mu);
    cufftHandle h;
    size_t ws = 0;
    int r = fft_plan(M, batch, type, in == out, &h, &ws);
    if (r != XS_OK) return r;
    if (ws > work_bytes) return XS_ETOOBIG;
    if (cufftSetStream(h, st) != CUFFT_SUCCESS || cufftSetWorkArea(h, work) != CUFFT_SUCCESS) return XS_ECUDA;
    cufftResult e;
    if (D) {
        e = forward ? cufftExecD2Z(h, (cufftDoubleReal*)in, (cufftDoubleComplex*)out)
                    : cufftExecZ2D(h, (cufftDoubleComplex*)in, (cufftDoubleReal*)out);
    } else {
        e = forward ? cufftExecR2C(h, (cufftReal*)in, (cufftComplex*)out)
                    : cufftExecC2R(h, (cufftComplex*)in, (cufftReal*)out);
    }
    xsi::count_launch();
    return e == CUFFT_SUCCESS ? XS_OK : XS_ECUDA;
}

// Layer constants, per-line terms, the distribution and its transform (Z), the image sum's
// transform (Ahat).
template <class R>
int modit_distribution(const xs_lines* ln, double nu_min, double R0, int64_t N, const double* T, const double* P,
                       int32_t L, double sb, int32_t ng, int64_t M, char* ws, const ModitPlan& p, bool keep_adj,
                       cudaStream_t st)
{
    constexpr bool FAST = std::is_same<R, float>::value;
    const int64_t nl = ln->n;
    auto* lay = (ModitLayer*)(ws + p.range);
    R* lsd = (R*)(ws + p.lsd);
    double* qv = (double*)(ws + p.lines);
    double* sinv = qv + nl;
    double* lgref = sinv + nl;
    void* work = ws + p.work;
    const dim3 lines((unsigned)((nl + 256 * MODIT_LINES - 1) / (256 * MODIT_LINES)), (unsigned)L);
    modit_layer_init_kernel<<<(L + 63) / 64, 64, 0, st>>>(T, P, sb, ln->q_exponent, L, lay);
    modit_prepass_kernel<<<(unsigned)((nl + 255) / 256), 256, 0, st>>>(ln->nu_hat, ln->gamma_ref, nl, nu_min, R0, qv,
                                                                        sinv, lgref);
    modit_range_kernel<<<lines, 256, 0, st>>>(lgref, ln->n_temp, nl, lay);
    if (keep_adj) modit_extreme_kernel<<<lines, 256, 0, st>>>(lgref, ln->n_temp, nl, lay);
    modit_layer_kernel<<<L, MODIT_MAX_GAMMA, 0, st>>>(ng, ln->mass_amu, R0, keep_adj ? ln->n_temp : nullptr, nl, lay);
    modit_lsd_kernel<R><<<dim3((unsigned)((M + MODIT_THREADS - 2) / (MODIT_THREADS - 1)), (unsigned)L), MODIT_THREADS, 0,
                          st>>>(ln->nu_hat, ln->ln_S0, ln->elower, ln->n_temp, qv, sinv, lgref, nl,
                                FAST ? MIXED_SCALE : 1.0, N, M, ng, lay, lsd);
    modit_images_kernel<R><<<(unsigned)((M + 255) / 256), 256, 0, st>>>(M, (R*)(ws + p.A));
    xsi::count_launch(keep_adj ? 7 : 6);
    if (cudaGetLastError() != cudaSuccess) return XS_ECUDA;
    int r = fft_exec<R>(M, (int64_t)L * ng, true, lsd, ws + p.Z, work, p.work_bytes, st);
    if (r != XS_OK) return r;
    return fft_exec<R>(M, 1, true, ws + p.A, ws + p.Ahat, work, p.work_bytes, st);
}

template <class R>
int run_modit(const xs_lines* ln, double nu_min, double nu_max, int64_t N, const double* T, const double* P,
              int32_t L, double sb, int32_t ng, int64_t M, void* sigma, char* ws, const ModitPlan& p, bool keep_adj,
              cudaStream_t st)
{
    using C = typename CplxOf<R>::type;
    constexpr bool FAST = std::is_same<R, float>::value;
    const double R0 = (double)(N - 1) / log(nu_max / nu_min);
    const int64_t H = M / 2 + 1;
    R* y = (R*)(ws + p.lsd); // y reuses the distribution's memory
    C* Y = (C*)(ws + p.Y);
    if (ln->n == 0) {
        const size_t es = FAST ? sizeof(float) : sizeof(double);
        return cudaMemsetAsync(sigma, 0, es * (size_t)L * N, st) == cudaSuccess ? XS_OK : XS_ECUDA;
    }
    int r = modit_distribution<R>(ln, nu_min, R0, N, T, P, L, sb, ng, M, ws, p, keep_adj, st);
    if (r != XS_OK) return r;
    modit_multiply_kernel<R, MODIT_F>
        <<<dim3((unsigned)((H + MODIT_STEP * MODIT_F - 1) / (MODIT_STEP * MODIT_F)), (unsigned)L), MODIT_STEP, 0, st>>>(
            (const C*)(ws + p.Z), (const C*)(ws + p.Ahat), M, ng, (const ModitLayer*)(ws + p.range), Y);
    xsi::count_launch();
    r = fft_exec<R>(M, L, false, Y, y, ws + p.work, p.work_bytes, st);
    if (r != XS_OK) return r;
    modit_finish_kernel<R><<<dim3((unsigned)((N + 255) / 256), (unsigned)L), 256, 0, st>>>(
        y, M, N, L, R0, nu_min, FAST ? MIXED_UNSCALE : 1.0, sigma);
    xsi::count_launch();
    return cudaGetLastError() == cudaSuccess ? XS_OK : XS_ECUDA;
}

// reuse: the distribution's transform, the layer constants and per-line terms of an
// immediately preceding forward (keep_adj) with the same inputs and workspace are
// still there; the adjoint leaves them as they are.
template <class R>
int run_modit_adjoint(const xs_lines* ln, double nu_min, double nu_max, int64_t N, const double* T, const double* P,
                      int32_t L, double sb, int32_t ng, int64_t M, const double* g_sigma, double* g_T, double* g_b,
                      char* ws, const ModitPlan& p, bool reuse, cudaStream_t st)
{
    using C = typename CplxOf<R>::type;
    constexpr bool FAST = std::is_same<R, float>::value;
    const double R0 = (double)(N - 1) / log(nu_max / nu_min);
    const int64_t nl = ln->n;
    auto* lay = (const ModitLayer*)(ws + p.range);
    C* X = (C*)(ws + p.lsd); // the distribution is no longer needed
    R* mu = (R*)(ws + p.mu);
    double* qv = (double*)(ws + p.lines);
    double* partL = (double*)(ws + p.partL);
    double* partT = (double*)(ws + p.partT);
    double* partB = (double*)(ws + p.partB);
    double* gbl = (double*)(ws + p.gbl);
    void* work = ws + p.work;
    if (nl == 0) {
        if (cudaMemsetAsync(g_T, 0, sizeof(double) * L, st) != cudaSuccess) return XS_ECUDA;
        return cudaMemsetAsync(g_b, 0, sizeof(double), st) == cudaSuccess ? XS_OK : XS_ECUDA;
    }
    int r = XS_OK;
    if (!reuse) r = modit_distribution<R>(ln, nu_min, R0, N, T, P, L, sb, ng, M, ws, p, true, st);
    if (r != XS_OK) return r;
    modit_mu_kernel<R><<<dim3((unsigned)((M + 255) / 256), (unsigned)L), 256, 0, st>>>(
        g_sigma, N, M, R0, nu_min, (FAST ? MIXED_UNSCALE : 1.0) / (double)M, mu);
    xsi::count_launch();
    r = fft_exec<R>(M, L, true, mu, ws + p.Y, work, p.work_bytes, st);
    if (r != XS_OK) return r;
    modit_adj_kernel_term<R, MODIT_F_ADJ><<<dim3((unsigned)p.nbk, (unsigned)L), MODIT_STEP, 0, st>>>(
        (const C*)(ws + p.Z), X, (const C*)(ws + p.Y), (const C*)(ws + p.Ahat), M, ng, sb, lay, partT, partB);
    xsi::count_launch();
    r = fft_exec<R>(M, (int64_t)L * ng, false, X, X, work, p.work_bytes, st); // correlations, in place
    if (r != XS_OK) return r;
    modit_adj_line_term<R><<<dim3((unsigned)p.nbl, (unsigned)L), 256, 0, st>>>(
        ln->nu_hat, ln->ln_S0, ln->elower, ln->n_temp, qv, qv + nl, qv + 2 * nl, nl, ln->q_exponent,
        FAST ? MIXED_SCALE : 1.0, N, M, ng, lay, (const R*)X, partL);
    modit_adj_reduce<<<L, 256, 0, st>>>(partL, p.nbl, partT, partB, p.nbk, g_T, gbl);
    modit_broad_sum<<<1, 32, 0, st>>>(gbl, L, g_b);
    xsi::count_launch(3);
    return cudaGetLastError() == cudaSuccess ? XS_OK : XS_ECUDA;
}

bool pow2(int64_t v) { return v > 0 && (v & (v - 1)) == 0; }

// the argument checks that both directions share
bool modit_args(const xs_lines* lines, double nu_min, double nu_max, int64_t N, const double* T, const double* P_bar,
                int32_t L, double broad_scale, int32_t n_gamma, int64_t n_fft, int prec, const void* workspace)
{
    if (!lines || lines->n < 0 || !T || !P_bar || !workspace || L <= 0 || N < 2) return false;
    if (lines->n > 0 && (!lines->nu_hat || !lines->ln_S0 || !lines->elower || !lines->gamma_ref || !lines->n_temp))
        return false;
    if (!(nu_min > 0.0) || !(nu_max > nu_min) || !(broad_scale > 0.0) || !(lines->mass_amu > 0.0)) return false;
    if (n_gamma < 1 || n_gamma > MODIT_MAX_GAMMA || !pow2(n_fft) || n_fft < N + 2) return false;
    return prec == XS_PREC_FP64 || prec == XS_PREC_MIXED;
}

} // namespace

namespace xsi {

int modit_forward(const xs_lines* lines, double nu_min, double nu_max, int64_t N, const double* T, const double* P_bar,
                  int32_t L, double broad_scale, int32_t n_gamma, int64_t n_fft, int prec, void* sigma,
                  void* workspace, size_t workspace_bytes, cudaStream_t st, int flags)
{
    if (!modit_args(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, prec, workspace) || !sigma)
        return XS_EINVAL;
    const ModitPlan p = modit_plan(lines->n, L, n_gamma, n_fft, prec);
    if (workspace_bytes < p.total) return XS_EINVAL;
    const bool keep = flags & XS_RUN_KEEP_ADJ;
    if (prec == XS_PREC_FP64)
        return run_modit<double>(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, sigma,
                                 (char*)workspace, p, keep, st);
    return run_modit<float>(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, sigma,
                            (char*)workspace, p, keep, st);
}

int modit_adjoint(const xs_lines* lines, double nu_min, double nu_max, int64_t N, const double* T, const double* P_bar,
                  int32_t L, double broad_scale, int32_t n_gamma, int64_t n_fft, int prec, const double* g_sigma,
                  double* g_T, double* g_broad, void* workspace, size_t workspace_bytes, cudaStream_t st, int flags)
{
    if (!modit_args(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, prec, workspace) || !g_sigma ||
        !g_T || !g_broad)
        return XS_EINVAL;
    // the offsets that a reused forward has filled are the same in both plans
    const ModitPlan p = modit_plan(lines->n, L, n_gamma, n_fft, prec, true);
    if (workspace_bytes < p.total) return XS_EINVAL;
    const bool reuse = flags & XS_RUN_REUSE;
    if (prec == XS_PREC_FP64)
        return run_modit_adjoint<double>(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, g_sigma,
                                         g_T, g_broad, (char*)workspace, p, reuse, st);
    return run_modit_adjoint<float>(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, g_sigma, g_T,
                                    g_broad, (char*)workspace, p, reuse, st);
}

} // namespace xsi

extern "C" {

size_t modit_adjoint_workspace_bytes(int64_t n_lines, int32_t L, int32_t n_gamma, int64_t n_fft, int prec)
{
    if (n_lines < 0 || L <= 0 || n_gamma < 1 || n_gamma > MODIT_MAX_GAMMA || !pow2(n_fft)) return 0;
    if (prec != XS_PREC_FP64 && prec != XS_PREC_MIXED) return 0;
    return modit_plan(n_lines, L, n_gamma, n_fft, prec, true).total;
}

int modit_compute_adjoint(const xs_lines* lines, double nu_min, double nu_max, int64_t N, const double* T,
                          const double* P_bar, int32_t L, double broad_scale, int32_t n_gamma, int64_t n_fft,
                          int prec, const double* g_sigma, double* g_T, double* g_broad, void* workspace,
                          size_t workspace_bytes, xs_stream stream)
{
    XS_NVTX("modit_compute_adjoint");
    return xsi::modit_adjoint(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, prec, g_sigma, g_T,
                              g_broad, workspace, workspace_bytes, (cudaStream_t)stream, 0);
}

size_t modit_workspace_bytes(int64_t n_lines, int32_t L, int32_t n_gamma, int64_t n_fft, int prec)
{
    if (n_lines < 0 || L <= 0 || n_gamma < 1 || n_gamma > MODIT_MAX_GAMMA || !pow2(n_fft)) return 0;
    if (prec != XS_PREC_FP64 && prec != XS_PREC_MIXED) return 0;
    return modit_plan(n_lines, L, n_gamma, n_fft, prec).total;
}

int modit_compute(const xs_lines* lines, double nu_min, double nu_max, int64_t N, const double* T,
                  const double* P_bar, int32_t L, double broad_scale, int32_t n_gamma, int64_t n_fft, int prec,
                  void* sigma, void* workspace, size_t workspace_bytes, xs_stream stream)
{
    XS_NVTX("modit_compute");
    return xsi::modit_forward(lines, nu_min, nu_max, N, T, P_bar, L, broad_scale, n_gamma, n_fft, prec, sigma,
                              workspace, workspace_bytes, (cudaStream_t)stream, 0);
}

} // extern "C"

XS_CHECK_ACCESSOR(modit)
