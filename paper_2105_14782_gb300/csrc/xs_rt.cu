// Layer optical depth (Eq. dtau_line), the pure-absorption emission solve of
// Sec. 3 (Eqs. rerr, rerr_tq, trans, sourcepla) with its adjoint, the Gaussian
// log-likelihood and the power-law temperature profile.  All double precision: the emission
// solve and its adjoint are bound by the FP64 pipe, the optical depth and the likelihood by
// memory or, on short rows, by latency.
#include <algorithm>
#include <cooperative_groups.h>
#include <type_traits>

#include "xs_device.cuh"
#include "xs_internal.h"

namespace xsd {

constexpr int RT_THREADS = 256;

// E2(x) and E3(x), x >= 0.  Double-precision operations run at 2 lanes a clock and SM
// here, so what bounds the emission solve is their number; neither branch divides.
//   x <= 1.5: E1 = -gamma - ln x - sum_k (-x)^k/(k k!), then E_{n+1} = (e^{-x} - x E_n)/n;
//   x > 1.5:  e^x E2(x) by a polynomial per half octave of x, [1.5 2^(i/2), 1.5 2^((i+1)/2)].
// The polynomials interpolate the continued fraction
//   e^x E2(x) = 1/(x + 2 - 1*2/(x + 4 - 2*3/(x + 6 - ...)))
// at Chebyshev nodes, at compile time.  The nearest singularity is x = 0, so on every
// interval the error falls as 11.7^-n: degree 15 is at rounding.  (A continued fraction
// of up to 70 divisions and a series with divisions before: 100 layers x 20,000 points,
// emission 3.38 ms, its adjoint 3.41 ms.)
constexpr int E2_N = 16;    // coefficients
constexpr int E2_PIECES = 18; // 1.5 .. 768, where e^-x has underflowed
constexpr int E1_N = 22;
struct ExpIntTable {
    double c[E2_PIECES][E2_N]; // powers of t = (x - mid) inv
    double mid[E2_PIECES], inv[E2_PIECES];
    double e1[E1_N + 1]; // (-1)^k/(k k!)
};
constexpr ExpIntTable make_exp_int_table()
{
    ExpIntTable r{};
    constexpr ChebTable<E2_N> ch = make_cheb<E2_N>();
    double edge = 1.5;
    for (int i = 0; i < E2_PIECES; ++i) {
        const double next = (i & 1) ? 1.5 * (double)(1 << ((i + 1) / 2)) : 1.5 * (double)(1 << (i / 2)) * SQRT2;
        const double mid = 0.5 * (edge + next), half = 0.5 * (next - edge);
        r.mid[i] = mid;
        r.inv[i] = 1.0 / half;
        double f[E2_N] = {};
        for (int m = 0; m < E2_N; ++m) {
            const double x = mid + half * ch.T[1][m];
            double v = x + 2.0 + 2.0 * 100;
            for (int k = 100; k >= 1; --k) v = x + 2.0 * k - (double)k * (double)(k + 1) / v;
            f[m] = 1.0 / v;
        }
        // Chebyshev coefficients, then powers: T_{k+1} = 2 t T_k - T_{k-1}
        double a[E2_N] = {}, b[E2_N] = {}; // T_k, T_{k+1}
        a[0] = 1.0;
        b[1] = 1.0;
        for (int k = 0; k < E2_N; ++k) {
            double ck = 0.0;
            for (int m = 0; m < E2_N; ++m) ck += f[m] * ch.T[k][m];
            ck *= (k ? 2.0 : 1.0) / E2_N;
            for (int j = 0; j <= k; ++j) r.c[i][j] += ck * a[j];
            double up[E2_N] = {};
            for (int j = 0; j < E2_N; ++j) up[j] = (j ? 2.0 * b[j - 1] : 0.0) - a[j];
            for (int j = 0; j < E2_N; ++j) {
                a[j] = b[j];
                b[j] = up[j];
            }
        }
        edge = next;
    }
    double fact = 1.0;
    for (int k = 1; k <= E1_N; ++k) {
        fact *= -k;
        r.e1[k] = 1.0 / (k * fact);
    }
    return r;
}
__device__ const ExpIntTable EXPINT = make_exp_int_table();

__device__ __forceinline__ void exp_int23(double x, double* E2, double* E3)
{
    const double ex = exp_tab(-x);
    double e2;
    if (x <= 1.5) {
        if (x == 0.0) {
            *E2 = 1.0;
            *E3 = 0.5;
            return;
        }
        double s = EXPINT.e1[E1_N];
#pragma unroll
        for (int k = E1_N - 1; k >= 1; --k) s = fma(s, x, EXPINT.e1[k]);
        const double e1 = -0.57721566490153286061 - log(x) - s * x;
        e2 = ex - x * e1;
    } else {
        // half octave of x/1.5 from its exponent and leading bits
        const double y = fmin(x, 767.0) * (1.0 / 1.5);
        const int hi = __double2hiint(y);
        const int i = min(max(2 * ((hi >> 20) - 1023) + ((hi & 0xfffff) >= 0x6a09e ? 1 : 0), 0), E2_PIECES - 1);
        const double t = (fmin(x, 767.0) - EXPINT.mid[i]) * EXPINT.inv[i];
        const double* c = EXPINT.c[i];
        double p = c[E2_N - 1];
#pragma unroll
        for (int k = E2_N - 2; k >= 0; --k) p = fma(p, t, c[k]);
        e2 = (x == x) ? ex * p : x; // fmin drops a NaN
    }
    *E2 = e2;
    *E3 = 0.5 * (ex - x * e2);
}

// a/(e^u - 1), u > 0: from e^-u where that loses nothing, the quotient corrected by its
// residual
__device__ __forceinline__ double bose(double a, double u)
{
    if (!(u >= 0.5)) return a / expm1(u);
    const double e = exp_tab(-u), d = 1.0 - e, y = rcp64(d), n = a * e;
    const double q = n * y;
    return fma(fma(-q, d, n), y, q);
}

// pi B(nu, T) = planck_c nu^3/(e^u - 1), u = c2 nu/T.  An error of u grows u-fold in
// e^u and stands undiminished in the adjoint's F_{n+1} - S_n, so u is formed to half an ulp:
// the quotient by 1/T gets its residual, with what rounding c2 nu lost, back.  One function
// for every layer's source and the bottom's, so that the bottom layer, which lies on its own
// temperature, sees F_L - S_{L-1} = 0 exactly.  Against quadruple precision, 24 layers x 300
// points, rms of F and g_dtau 3.4e-16 and 3.6e-16; with a rounded product c2 nu (1/T) 4.9e-16
// and 5.7e-16, with a division 4.5e-16 and 4.6e-16; no difference in time beyond the runs'.
constexpr double PLANCK_C = PI * 2.0 * hP * cL * cL;
struct Planck {
    double kv, cv, cl; // planck_c nu^3; c2 nu and its rounding error
    __device__ __forceinline__ explicit Planck(double v)
        : kv(PLANCK_C * v * v * v), cv(c2 * v), cl(fma(c2, v, -cv))
    {
    }
    __device__ __forceinline__ double operator()(double T) const
    {
        const int e = __double2hiint(T) & 0x7ff00000;
        double u;
        if (e < 0x20b00000 || e > 0x5f300000) { // beyond 2^-500..2^500: 0, infinities, NaN
            u = cv / T;
        } else {
            const double y = rcp64(T), q = cv * y;
            u = fma(fma(-q, T, cv) + cl, y, q);
        }
        return bose(kv, u);
    }
};

struct SigPtrs {
    const void* p[XS_MAX_SPECIES];
};
struct GSigPtrs {
    double* p[XS_MAX_SPECIES];
};

// A row of a layer per block row: the layer's factors are formed once a block (a division
// for them and one of the index an element before: 101 x 49,999, two species, 236 us).
__global__ void tau_kernel(SigPtrs sig, int S, const double* __restrict__ vmr, const double* __restrict__ P,
                           const double* __restrict__ dP, int L, int64_t N, double g, double mu, double kappa,
                           int is_float, double* __restrict__ dtau)
{
    __shared__ double f[XS_MAX_SPECIES + 1];
    for (int64_t n = blockIdx.y; n < L; n += gridDim.y) {
        __syncthreads();
        if (threadIdx.x <= S) {
            const int m = threadIdx.x;
            f[m] = m < S ? dP[n] * 1e6 / (mu * amu * g) * vmr[(size_t)m * L + n] : kappa * P[n] * dP[n] * 1e6 / g;
        }
        __syncthreads();
        for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
            const size_t i = (size_t)n * N + j;
            double s = f[S];
            for (int m = 0; m < S; ++m)
                s = fma(f[m], is_float ? (double)((const float*)sig.p[m])[i] : ((const double*)sig.p[m])[i], s);
            dtau[i] = s;
        }
    }
}

// Sum over a cluster of C blocks, fixed order; the result is valid in thread 0 of rank 0.
// One block cannot draw enough of the chip for a row of 1e4-1e5 points.
constexpr int RT_CLUSTER = 8;
template <int C>
__device__ __forceinline__ double cluster_sum(double v, double* red, double* slot)
{
    namespace cg = cooperative_groups;
    red[threadIdx.x] = v;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    double t = 0.0;
    if constexpr (C == 1) {
        t = red[0];
        __syncthreads(); // read before it is written again
    } else {
        cg::cluster_group cl = cg::this_cluster();
        if (threadIdx.x == 0) *slot = red[0];
        cl.sync();
        if (threadIdx.x == 0 && cl.block_rank() == 0)
            for (int b = 0; b < C; ++b) t += *cl.map_shared_rank(slot, b);
        cl.sync(); // the slots are read before they are written again or a block ends
    }
    return t;
}

// g_sigma[m] = g_dtau col vmr; g_vmr[m][n] = col sum_j g_dtau sigma_m.  A cluster of C
// blocks per layer, one pass over the row for all species (one block per layer and a pass
// per species before: 101 layers x 49,999 points 178 us, 4 layers x 100,000 points 304 us).
// M: the number of species, XS_MAX_SPECIES for any.
template <int C, int M>
__global__ void __launch_bounds__(RT_THREADS)
    tau_adjoint_kernel(SigPtrs sig, GSigPtrs gsig, int species, const double* __restrict__ vmr,
                       const double* __restrict__ dP, int L, int64_t N, double g, double mu, int is_float,
                       const double* __restrict__ g_dtau, double* __restrict__ g_vmr)
{
    __shared__ double red[RT_THREADS], slot;
    const int S = M < XS_MAX_SPECIES ? M : species;
    const int n = blockIdx.x / C, rank = blockIdx.x % C;
    const double col = dP[n] * 1e6 / (mu * amu * g);
    double acc[M], cv[M];
#pragma unroll
    for (int m = 0; m < M; ++m) {
        acc[m] = 0.0;
        cv[m] = m < S ? col * vmr[(size_t)m * L + n] : 0.0;
    }
#pragma unroll (M <= 2 ? 4 : 1)
    for (int64_t j = (int64_t)rank * blockDim.x + threadIdx.x; j < N; j += C * blockDim.x) {
        const size_t i = (size_t)n * N + j;
        const double gd = g_dtau[i];
#pragma unroll
        for (int m = 0; m < M; ++m) {
            if (m >= S) break;
            const double v = is_float ? (double)((const float*)sig.p[m])[i] : ((const double*)sig.p[m])[i];
            acc[m] = fma(gd, v, acc[m]);
            if (gsig.p[m]) gsig.p[m][i] = gd * cv[m];
        }
    }
#pragma unroll
    for (int m = 0; m < M; ++m) {
        if (m >= S) break;
        const double t = cluster_sum<C>(acc[m], red, &slot);
        if (threadIdx.x == 0 && rank == 0) g_vmr[(size_t)m * L + n] = col * t;
    }
}

// Emission solve (Sec. 2.3):  F0 = sum_n Phi_n (1 - T_n) S_n + Phi_L S_B, with
// Phi_n = prod_{k<n} T_k, T_n = 2 E3(dtau_n), S_n = pi B(nu, T_n), S_B = pi B(nu, T_{L-1}).
// A block takes PTS grid points (neighbouring lanes, so rows of dtau are read in whole
// sectors) and its RT_THREADS/PTS groups of lanes take contiguous segments of the layers:
// each reduces its segment to (prod T, local sum), and the segments are chained in
// order.  Bound by FP64 operations (about 70 a point and layer) on the SMs that have
// blocks: see emission_points.
__device__ __forceinline__ void seg_range(int L, int w, int segs, int* n0, int* n1)
{
    *n0 = (int)(((int64_t)L * w) / segs);
    *n1 = (int)(((int64_t)L * (w + 1)) / segs);
}

// KEEP: the layer's T_n, E2_n and S_n are stored for the adjoint of the same call.
template <int PTS, bool KEEP>
__global__ void __launch_bounds__(RT_THREADS) emission_kernel(const double* __restrict__ dtau,
                                                              const double* __restrict__ T,
                                                              const double* __restrict__ nu, int L, int64_t N,
                                                              double* __restrict__ F0, double* __restrict__ w_tr,
                                                              double* __restrict__ w_e2, double* __restrict__ w_S)
{
    constexpr int SEG = RT_THREADS / PTS;
    __shared__ double segP[SEG][PTS], segF[SEG][PTS];
    const int lane = threadIdx.x % PTS, w = threadIdx.x / PTS;
    const int64_t j = (int64_t)blockIdx.x * PTS + lane;
    const bool valid = j < N;
    const double v = valid ? nu[j] : nu[0];
    const Planck planck(v);
    int n0, n1;
    seg_range(L, w, SEG, &n0, &n1);
    double phi = 1.0, F = 0.0;
    if (valid) {
        for (int n = n0; n < n1; ++n) {
            double e2, e3;
            const size_t i = (size_t)n * N + j;
            exp_int23(dtau[i], &e2, &e3);
            const double tr = 2.0 * e3, Sn = planck(T[n]);
            if (KEEP) {
                w_tr[i] = tr;
                w_e2[i] = e2;
                w_S[i] = Sn;
            }
            F += phi * (1.0 - tr) * Sn;
            phi *= tr;
        }
    }
    segP[w][lane] = phi;
    segF[w][lane] = F;
    __syncthreads();
    if (w == 0 && valid) {
        double Ft = 0.0, ph = 1.0;
        for (int s = 0; s < SEG; ++s) {
            Ft += ph * segF[s][lane];
            ph *= segP[s][lane];
        }
        F0[j] = Ft + ph * planck(T[L - 1]);
    }
}

// Adjoint of the emission solve for lambda = dlogL/dF0:
//   dF0/ddtau_n = Phi_n (F_{n+1} - S_n) dT_n/ddtau_n,  dT/ddtau = -2 E2(dtau),
//   dF0/dS_n = Phi_n (1 - T_n) (+ Phi_L for the bottom source, n = L-1),
// where F_{n+1} = upward flux below layer n: F_L = S_B, F_n = T_n F_{n+1} + (1 - T_n) S_n.
// Three passes over each group's layer segment: (1) T, E2, S stored and the
// segment's maps F_top = A F_bottom + C and prod T; (2) after chaining the
// segments, F_{n+1} down the segment; (3) Phi_n along it, g_dtau and the
// per-layer sums of lambda dF0/dS_n dS_n/dT_n over the block's points.  REUSE: the
// factors of (1) are the forward's (KEEP) and only chained.
template <int PTS, bool REUSE>
__global__ void __launch_bounds__(RT_THREADS) emission_adjoint_kernel(
    const double* __restrict__ g_F0, const double* __restrict__ dtau, const double* __restrict__ T,
    const double* __restrict__ nu, int L, int64_t N, double* __restrict__ g_dtau, double* __restrict__ part,
    double* __restrict__ w_tr, double* __restrict__ w_e2, double* __restrict__ w_S)
{
    constexpr int SEG = RT_THREADS / PTS;
    __shared__ double segA[SEG][PTS], segC[SEG][PTS], segFin[SEG][PTS], segPhi[SEG][PTS];
    const int lane = threadIdx.x % PTS, w = threadIdx.x / PTS;
    const int64_t j = (int64_t)blockIdx.x * PTS + lane;
    const bool valid = j < N;
    const double v = valid ? nu[j] : nu[0];
    const double lam = valid ? g_F0[j] : 0.0;
    const Planck planck(v);
    int n0, n1;
    seg_range(L, w, SEG, &n0, &n1);
    // (1) per-layer factors and the segment's backward map
    double A = 1.0, Cm = 0.0;
    if (valid) {
        for (int n = n1 - 1; n >= n0; --n) {
            const size_t i = (size_t)n * N + j;
            double tr, Sn;
            if (REUSE) {
                tr = w_tr[i];
                Sn = w_S[i];
            } else {
                double e2, e3;
                exp_int23(dtau[i], &e2, &e3);
                tr = 2.0 * e3;
                Sn = planck(T[n]);
                w_tr[i] = tr;
                w_e2[i] = e2;
                w_S[i] = Sn;
            }
            Cm = tr * Cm + (1.0 - tr) * Sn;
            A *= tr;
        }
    }
    segA[w][lane] = A;
    segC[w][lane] = Cm;
    __syncthreads();
    if (w == 0) {
        // flux entering each segment from below, and Phi at each segment's top
        double Fb = valid ? planck(T[L - 1]) : 0.0;
        for (int s = SEG - 1; s >= 0; --s) {
            segFin[s][lane] = Fb;
            Fb = segA[s][lane] * Fb + segC[s][lane];
        }
        double ph = 1.0;
        for (int s = 0; s < SEG; ++s) {
            segPhi[s][lane] = ph;
            ph *= segA[s][lane];
        }
    }
    __syncthreads();
    // (2) F_{n+1} for each layer of the segment, kept in g_dtau until (3)
    if (valid) {
        double F = segFin[w][lane];
        for (int n = n1 - 1; n >= n0; --n) {
            const size_t i = (size_t)n * N + j;
            g_dtau[i] = F;
            const double tr = w_tr[i];
            F = tr * F + (1.0 - tr) * w_S[i];
        }
    }
    // (3) forward along the segment (as many steps in every group of a warp, for the sums)
    double phi = segPhi[w][lane];
    const double phiL = segPhi[SEG - 1][lane] * segA[SEG - 1][lane];
    const double inv_kv = 1.0 / planck.kv;
    const int most = (L + SEG - 1) / SEG;
    for (int k = 0; k < most; ++k) {
        const int n = n0 + k;
        double gT = 0.0;
        if (valid && n < n1) {
            const size_t i = (size_t)n * N + j;
            const double tr = w_tr[i], Sn = w_S[i], invT = rcp64_any(T[n]);
            g_dtau[i] = lam * phi * (g_dtau[i] - Sn) * (-2.0 * w_e2[i]);
            double gS = lam * phi * (1.0 - tr);
            if (n == L - 1) gS += lam * phiL;
            phi *= tr;
            // d(pi B)/dT = B (u/T)/(1 - e^-u), and 1/(1 - e^-u) = 1 + 1/(e^u - 1) = 1 + B/kv
            gT = gS * Sn * (planck.cv * invT * invT) * fma(Sn, inv_kv, 1.0);
        }
        for (int o = PTS / 2; o > 0; o >>= 1) gT += __shfl_xor_sync(0xffffffffu, gT, o, PTS);
        if (lane == 0 && n < n1) part[(size_t)n * gridDim.x + blockIdx.x] = gT;
    }
}

__global__ void layer_sum_kernel(const double* __restrict__ part, int nb, int L, double* __restrict__ out)
{
    __shared__ double red[RT_THREADS];
    int n = blockIdx.x;
    double a = 0.0;
    for (int i = threadIdx.x; i < nb; i += blockDim.x) a += part[(size_t)n * nb + i];
    red[threadIdx.x] = a;
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x == 0) out[n] = red[0];
}

// One cluster; one division a point (one block and two divisions before: 20,000 points
// 100 us, 100,000 points 475 us).
__global__ void __cluster_dims__(RT_CLUSTER, 1, 1)
    loglike_kernel(const double* __restrict__ F, const double* __restrict__ d, const double* __restrict__ s, int64_t N,
                   double* __restrict__ logL, double* __restrict__ gF)
{
    __shared__ double red[1024], slot;
    double acc = 0.0;
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < N; j += RT_CLUSTER * blockDim.x) {
        const double is = 1.0 / s[j];
        const double r = (d[j] - F[j]) * is;
        acc = fma(r, r, acc);
        if (gF) gF[j] = r * is;
    }
    const double t = cluster_sum<RT_CLUSTER>(acc, red, &slot);
    if (threadIdx.x == 0 && blockIdx.x == 0) logL[0] = -0.5 * t;
}

struct VmrArgs {
    double lg[XS_MAX_SPECIES];
};

// layer temperatures T0 P^alpha (T != nullptr) and mixing ratios 10^lg (vmr != nullptr)
__global__ void atmosphere_kernel(double T0, double alpha, const double* __restrict__ P, int L, double* __restrict__ T,
                                  VmrArgs a, int S, double* __restrict__ vmr)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (T && i < L) T[i] = T0 * pow(P[i], alpha);
    if (vmr && i < S * L) vmr[i] = pow(10.0, a.lg[i / L]);
}

__device__ __forceinline__ double warp_sum(double v)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// dlogL/dtheta from the per-layer pieces, one warp, fixed order:
//   T0:    sum_n g_T[n] T_n / T0
//   alpha: sum_n g_T[n] T_n ln P_n
//   log10 vmr_m: ln10 sum_n g_vmr[m][n] vmr_m
//   broadening scale: sum_m g_b[m]
// (100 layers: 200 us when one thread did it.)
__global__ void theta_grad_kernel(int S, int L, double T0, const double* __restrict__ vmr, const double* __restrict__ T,
                                  const double* __restrict__ P, const double* __restrict__ g_T,
                                  const double* __restrict__ g_vmr, const double* __restrict__ g_b,
                                  double* __restrict__ out)
{
    const int lane = threadIdx.x;
    double gT0 = 0.0, ga = 0.0;
    for (int n = lane; n < L; n += 32) {
        const double t = g_T[n] * T[n];
        gT0 += t;
        ga = fma(t, log(P[n]), ga);
    }
    gT0 = warp_sum(gT0);
    ga = warp_sum(ga);
    double gb = 0.0;
    for (int m = 0; m < S; ++m) {
        double s = 0.0;
        for (int n = lane; n < L; n += 32) s += g_vmr[(size_t)m * L + n];
        s = warp_sum(s);
        if (lane == 0) out[3 + m] = 2.30258509299404568402 * vmr[(size_t)m * L] * s;
        gb += g_b[m];
    }
    if (lane == 0) {
        out[1] = gT0 / T0;
        out[2] = ga;
        out[3 + S] = gb;
    }
}

// Collision-induced absorption (Sec. 2.4, Eq. taucont): dtau += n1 n2 alpha(T, nu) H dP/P,
// n_i = vmr_i P/(kB T), H = kB T/(mu m_u g), alpha linear in T between the table's
// temperatures (clamped).  = vmr1 vmr2 P dP alpha/(kB T mu m_u g) with P, dP in dyn/cm^2.
__device__ __forceinline__ void cia_interp(const double* Tg, int nT, double T, int* k, double* w, double* dw)
{
    if (nT < 2 || T <= Tg[0]) {
        *k = 0;
        *w = 0.0;
        *dw = 0.0;
        return;
    }
    if (T >= Tg[nT - 1]) {
        *k = nT - 2;
        *w = 1.0;
        *dw = 0.0;
        return;
    }
    int lo = 0, hi = nT - 1; // Tg[lo] <= T < Tg[hi]
    while (hi - lo > 1) {
        const int m = (lo + hi) >> 1;
        if (Tg[m] <= T) lo = m; else hi = m;
    }
    *k = lo;
    *dw = 1.0 / (Tg[lo + 1] - Tg[lo]);
    *w = (T - Tg[lo]) * *dw;
}

__global__ void tau_cia_kernel(const double* __restrict__ alpha, const double* __restrict__ Tg, int nT,
                               const double* __restrict__ T, const double* __restrict__ P,
                               const double* __restrict__ dP, int L, int64_t N, double c12, int accumulate,
                               double* __restrict__ dtau)
{
    const int n = blockIdx.y;
    int k;
    double w, dw;
    cia_interp(Tg, nT, T[n], &k, &w, &dw);
    const double f = c12 * P[n] * dP[n] / T[n];
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < N; j += (int64_t)gridDim.x * blockDim.x) {
        const double a0 = alpha[(size_t)k * N + j];
        const double a = (nT > 1) ? a0 + w * (alpha[(size_t)(k + 1) * N + j] - a0) : a0;
        const size_t i = (size_t)n * N + j;
        dtau[i] = (accumulate ? dtau[i] : 0.0) + f * a;
    }
}

// g_T[n] += sum_j g_dtau[n][j] d dtau[n][j]/dT_n, d/dT of f(T) alpha(T) with f ~ 1/T
// (one block per layer, fixed-order sum)
__global__ void tau_cia_adjoint_kernel(const double* __restrict__ g_dtau, const double* __restrict__ alpha,
                                       const double* __restrict__ Tg, int nT, const double* __restrict__ T,
                                       const double* __restrict__ P, const double* __restrict__ dP, int64_t N,
                                       double c12, double* __restrict__ g_T)
{
    __shared__ double red[RT_THREADS];
    const int n = blockIdx.x;
    int k;
    double w, dw;
    cia_interp(Tg, nT, T[n], &k, &w, &dw);
    const double f = c12 * P[n] * dP[n] / T[n];
    double s = 0.0;
    for (int64_t j = threadIdx.x; j < N; j += blockDim.x) {
        const double a0 = alpha[(size_t)k * N + j];
        const double a1 = (nT > 1) ? alpha[(size_t)(k + 1) * N + j] : a0;
        const double a = a0 + w * (a1 - a0);
        const double da = (a1 - a0) * dw;
        s += g_dtau[(size_t)n * N + j] * f * (da - a / T[n]);
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) g_T[n] += red[0];
}

// Gradient for per-layer temperatures: out[1 + n] = dlogL/dT_n, then
// dlogL/dlog10 vmr_m and dlogL/ds_b (out[0], logL, is left as it is).
__global__ void layer_grad_kernel(int S, int L, const double* __restrict__ vmr, const double* __restrict__ g_T,
                                  const double* __restrict__ g_vmr, const double* __restrict__ g_b,
                                  double* __restrict__ out)
{
    const int lane = threadIdx.x;
    for (int n = lane; n < L; n += 32) out[1 + n] = g_T[n];
    double gb = 0.0;
    for (int m = 0; m < S; ++m) {
        double s = 0.0;
        for (int n = lane; n < L; n += 32) s += g_vmr[(size_t)m * L + n];
        s = warp_sum(s);
        if (lane == 0) out[1 + L + m] = 2.30258509299404568402 * vmr[(size_t)m * L] * s;
        gb += g_b[m];
    }
    if (lane == 0) out[1 + L + S] = gb;
}

__global__ void accumulate_kernel(double* __restrict__ dst, const double* __restrict__ src, int64_t n, int first)
{
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) dst[i] = first ? src[i] : dst[i] + src[i];
}

} // namespace xsd

using namespace xsd;

namespace xsi {

static inline int last_status() { return cudaGetLastError() == cudaSuccess ? XS_OK : XS_ECUDA; }
static inline int launched(int n)
{
    count_launch(n);
    return last_status();
}

int rt_tau(const void* const* sigma, int32_t S, const double* vmr, const double* P, const double* dP, int32_t L,
           int64_t N, double g, double mu, double kappa, int prec, double* dtau, cudaStream_t st)
{
    SigPtrs sp{};
    for (int m = 0; m < S; ++m) sp.p[m] = sigma[m];
    const unsigned gx = (unsigned)std::min<int64_t>((N + 4 * RT_THREADS - 1) / (4 * RT_THREADS), 1024);
    tau_kernel<<<dim3(gx, (unsigned)std::min(L, 65535)), RT_THREADS, 0, st>>>(sp, S, vmr, P, dP, L, N, g, mu, kappa,
                                                                 prec == XS_PREC_MIXED, dtau);
    return launched(1);
}

int rt_tau_adjoint(const void* const* sigma, int32_t S, const double* vmr, const double* P, const double* dP,
                   int32_t L, int64_t N, double g, double mu, int prec, const double* g_dtau, double* const* g_sigma,
                   double* g_vmr, cudaStream_t st)
{
    (void)P;
    SigPtrs sp{};
    GSigPtrs gp{};
    for (int m = 0; m < S; ++m) {
        sp.p[m] = sigma[m];
        gp.p[m] = g_sigma ? g_sigma[m] : nullptr;
    }
    // blocks a layer: up to 8, fewer where the layers alone fill the chip or a block had less
    // than 1,024 points (4,096 from 128 layers on): a cluster costs more to launch and to join
    // than so short a row (1,000 layers of 50 points 154 us with 8 blocks, 300 of 9,727 88 us)
    const int64_t points = L < 128 ? 1024 : 4096;
    int c = 1;
    while (c < RT_CLUSTER && (int64_t)c * L < 256 && 2 * c * points <= N) c *= 2;
    auto pick = [&](auto M) {
        constexpr int m = decltype(M)::value;
        return c == 8   ? tau_adjoint_kernel<8, m>
               : c == 4 ? tau_adjoint_kernel<4, m>
               : c == 2 ? tau_adjoint_kernel<2, m>
                        : tau_adjoint_kernel<1, m>;
    };
    auto* k = S == 1   ? pick(std::integral_constant<int, 1>{})
              : S == 2 ? pick(std::integral_constant<int, 2>{})
                       : pick(std::integral_constant<int, XS_MAX_SPECIES>{});
    int threads = RT_THREADS;
    while (threads > 32 && threads * (int64_t)c * 4 > N) threads /= 2; // four points a thread
    cudaLaunchAttribute cluster{};
    cluster.id = cudaLaunchAttributeClusterDimension;
    cluster.val.clusterDim.x = (unsigned)c;
    cluster.val.clusterDim.y = cluster.val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)(c * L));
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = st;
    cfg.attrs = &cluster;
    cfg.numAttrs = c > 1 ? 1 : 0;
    if (cudaLaunchKernelEx(&cfg, k, sp, gp, (int)S, vmr, dP, (int)L, N, g, mu, (int)(prec == XS_PREC_MIXED), g_dtau, g_vmr) !=
        cudaSuccess)
        return XS_ECUDA;
    return launched(1);
}

// Points a block of the emission kernels takes.  A group of lanes of a warp is a segment, so a
// warp's time is its longest segment's layers, and what counts is the sum of that over a
// block's warps times the blocks an SM gets: in whole blocks while they are few (below four
// an SM), on average then.  A few layers leave most segments of the small blocks empty (3
// layers x 9,000 points 47 us with 8, 12 with 32; 20 x 2,003 23 with 8, 19 with 16); 60 x 3,000
// take 8 points, for more SMs.
static int emission_points(int32_t L, int64_t N)
{
    int best = 32;
    double least = 0.0;
    for (int pts = 32; pts >= 8; pts /= 2) {
        const int segs = RT_THREADS / pts, group = 32 / pts; // segments of a block and of a warp
        int layers = 0;
        for (int w = 0; w < segs; w += group) {
            int most = 0;
            for (int g = w; g < w + group; ++g)
                most = std::max(most, (int)((int64_t)L * (g + 1) / segs - (int64_t)L * g / segs));
            layers += most;
        }
        const int64_t nb = (N + pts - 1) / pts;
        const double cost = layers * (nb >= 4 * SMS ? (double)nb / SMS : (double)((nb + SMS - 1) / SMS));
        if (pts == 32 || cost < least) {
            least = cost;
            best = pts;
        }
    }
    return best;
}

// [L][nb] per-block layer partials, then T_n, E2_n and S_n as [L][N] each.  The partials'
// space is that of the smallest blocks, so that the size grows with N and a workspace that
// serves a grid serves every smaller one.
struct EmissionWs {
    double *part, *tr, *e2, *S;
    size_t bytes;
};
static EmissionWs emission_ws(int32_t L, int64_t N, void* ws)
{
    const int64_t nb = (N + 7) / 8;
    auto al = [](size_t b) { return (b + 255) / 256 * 256; };
    const size_t part = al(sizeof(double) * (size_t)L * (size_t)nb), LN = al(sizeof(double) * (size_t)L * (size_t)N);
    char* base = (char*)ws;
    return {(double*)base, (double*)(base + part), (double*)(base + part + LN), (double*)(base + part + 2 * LN),
            part + 3 * LN};
}

template <int PTS>
static void launch_emission(const double* dtau, const double* T, const double* nu, int32_t L, int64_t N, double* F0,
                            void* keep, cudaStream_t st)
{
    const unsigned nb = (unsigned)((N + PTS - 1) / PTS);
    const EmissionWs w = emission_ws(L, N, keep);
    if (keep) emission_kernel<PTS, true><<<nb, RT_THREADS, 0, st>>>(dtau, T, nu, L, N, F0, w.tr, w.e2, w.S);
    else emission_kernel<PTS, false><<<nb, RT_THREADS, 0, st>>>(dtau, T, nu, L, N, F0, nullptr, nullptr, nullptr);
}

int rt_emission(const double* dtau, const double* T, const double* nu, int32_t L, int64_t N, double* F0,
                cudaStream_t st, void* keep)
{
    const int pts = emission_points(L, N);
    if (pts == 32) launch_emission<32>(dtau, T, nu, L, N, F0, keep, st);
    else if (pts == 16) launch_emission<16>(dtau, T, nu, L, N, F0, keep, st);
    else launch_emission<8>(dtau, T, nu, L, N, F0, keep, st);
    return launched(1);
}

size_t rt_emission_ws(int32_t L, int64_t N) { return emission_ws(L, N, nullptr).bytes; }

template <int PTS>
static void launch_emission_adjoint(const double* g_F0, const double* dtau, const double* T, const double* nu, int32_t L,
                                    int64_t N, double* g_dtau, const EmissionWs& w, bool reuse, cudaStream_t st)
{
    const unsigned nb = (unsigned)((N + PTS - 1) / PTS);
    auto* k = reuse ? emission_adjoint_kernel<PTS, true> : emission_adjoint_kernel<PTS, false>;
    k<<<nb, RT_THREADS, 0, st>>>(g_F0, dtau, T, nu, L, N, g_dtau, w.part, w.tr, w.e2, w.S);
}

int rt_emission_adjoint(const double* g_F0, const double* dtau, const double* T, const double* nu, int32_t L,
                        int64_t N, double* g_dtau, double* g_T, void* ws, cudaStream_t st, bool reuse)
{
    const int pts = emission_points(L, N);
    const EmissionWs w = emission_ws(L, N, ws);
    if (pts == 32) launch_emission_adjoint<32>(g_F0, dtau, T, nu, L, N, g_dtau, w, reuse, st);
    else if (pts == 16) launch_emission_adjoint<16>(g_F0, dtau, T, nu, L, N, g_dtau, w, reuse, st);
    else launch_emission_adjoint<8>(g_F0, dtau, T, nu, L, N, g_dtau, w, reuse, st);
    layer_sum_kernel<<<L, RT_THREADS, 0, st>>>(w.part, (int)((N + pts - 1) / pts), L, g_T);
    return launched(2);
}

int rt_loglike(const double* F, const double* d, const double* s, int64_t N, double* logL, double* g_F,
               cudaStream_t st)
{
    loglike_kernel<<<RT_CLUSTER, 1024, 0, st>>>(F, d, s, N, logL, g_F);
    return launched(1);
}

int rt_atmosphere(double T0, double alpha, const double* P, int32_t L, double* T, int32_t S, const double* lg,
                  double* vmr, cudaStream_t st)
{
    VmrArgs a{};
    for (int m = 0; m < S; ++m) a.lg[m] = lg[m];
    const int many = vmr ? std::max(S, 1) * L : L;
    atmosphere_kernel<<<(many + 127) / 128, 128, 0, st>>>(T0, alpha, P, L, T, a, S, vmr);
    return launched(1);
}

int rt_theta_grad(int32_t S, int32_t L, double T0, const double* vmr, const double* T, const double* P,
                  const double* g_T, const double* g_vmr, const double* g_b, double* out, cudaStream_t st)
{
    theta_grad_kernel<<<1, 32, 0, st>>>(S, L, T0, vmr, T, P, g_T, g_vmr, g_b, out);
    return launched(1);
}

static double cia_c12(double vmr1, double vmr2, double g, double mu)
{
    return vmr1 * vmr2 * 1e12 / (kB * mu * amu * g); // P dP in bar^2 -> (dyn/cm^2)^2
}

int rt_tau_cia(const double* alpha, const double* Tg, int32_t nT, const double* T, const double* P, const double* dP,
               int32_t L, int64_t N, double vmr1, double vmr2, double g, double mu, int accumulate, double* dtau,
               cudaStream_t st)
{
    const unsigned gx = (unsigned)std::min<int64_t>((N + RT_THREADS - 1) / RT_THREADS, 1024);
    tau_cia_kernel<<<dim3(gx, (unsigned)L), RT_THREADS, 0, st>>>(alpha, Tg, nT, T, P, dP, L, N,
                                                                 cia_c12(vmr1, vmr2, g, mu), accumulate, dtau);
    return launched(1);
}

int rt_tau_cia_adjoint(const double* g_dtau, const double* alpha, const double* Tg, int32_t nT, const double* T,
                       const double* P, const double* dP, int32_t L, int64_t N, double vmr1, double vmr2, double g,
                       double mu, double* g_T, cudaStream_t st)
{
    tau_cia_adjoint_kernel<<<L, RT_THREADS, 0, st>>>(g_dtau, alpha, Tg, nT, T, P, dP, N, cia_c12(vmr1, vmr2, g, mu),
                                                     g_T);
    return launched(1);
}

int rt_layer_grad(int32_t S, int32_t L, const double* vmr, const double* g_T, const double* g_vmr, const double* g_b,
                  double* out, cudaStream_t st)
{
    layer_grad_kernel<<<1, 32, 0, st>>>(S, L, vmr, g_T, g_vmr, g_b, out);
    return launched(1);
}

int rt_accumulate(double* dst, const double* src, int64_t n, int first, cudaStream_t st)
{
    accumulate_kernel<<<(unsigned)((n + 255) / 256), 256, 0, st>>>(dst, src, n, first);
    return launched(1);
}

} // namespace xsi

XS_CHECK_ACCESSOR(rt)
