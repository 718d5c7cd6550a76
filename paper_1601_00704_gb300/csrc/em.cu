// EM fit of a one-dimensional Gaussian mixture on the GPU (Sec. 2.2,
// Eqs. 20-24): the pore-size statistics that the paper splits into organic
// (OM) and inorganic (IOM) components before the DGM/GMS permeabilities are
// assigned.  FP64 throughout.
//
// One iteration is one launch (k_em_step): the E-step responsibilities w_j(i)
// (Eqs. 20-21, exponent with its minus sign) and, in the same pass, the sums
// of w, w d and w d^2 with d = x - mu_j (the old mean), from which
//   Phi_j = S0/m,  mu_j += S1/S0,  sigma_j^2 = S2/S0 - (S1/S0)^2   (Eqs. 22-24).
// The subtraction is harmless while the mean moves by less than a few sigma.
// Where it would cancel (a component collapsing onto few samples) the launch
// leaves the estimate alone and asks for the two-pass iteration instead
// (k_em_pass1/2: sums of w and w x, then of w (x - mu_new)^2).
// Each launch writes per-block partials that the last block adds in a fixed
// order, so a fit is bit-for-bit reproducible.
//
#include "fixed.cuh"
#include "glbm.h"

#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>

extern __attribute__((visibility("hidden"))) thread_local char g_create_err[512];

namespace {

constexpr int KMAX = 8;
constexpr int EM_THREADS = 256;   // two-pass kernels
constexpr int STEP_THREADS = 256;  // k_em_step
constexpr int STEP_BLOCKS = 2;     // of it per SM

// Progress of a fit on the device.
struct EmState {
    double ll, prev;   // mean log-likelihood of this and the previous E-step
    int it;            // iterations done
    int done;          // converged: later launches return at once
    int cancel;        // the next iteration needs the two passes; likewise
    unsigned ticket;
};

struct EmParams {
    int k;
    double phi[KMAX], mu[KMAX], var[KMAX];  // current estimate (E-step uses these)
    double mu_new[KMAX];                    // pass-1 result used by pass 2
    double amp[KMAX], hiv[KMAX];            // phi / sqrt(2 pi var), -1 / (2 var)
};

__host__ __device__ inline void em_factor(double phi, double var, double &amp, double &hiv) {
    amp = phi * (0.39894228040143267794 / sqrt(var));
    hiv = -0.5 / var;
}
__host__ __device__ inline void em_factors(EmParams &p) {
    for (int j = 0; j < p.k; ++j) em_factor(p.phi[j], p.var[j], p.amp[j], p.hiv[j]);
}

__device__ __forceinline__ void responsibilities(double x, const EmParams &p, double (&w)[KMAX], double &den) {
    const double inv_sqrt_2pi = 0.39894228040143267794;
    den = 0.0;
#pragma unroll
    for (int j = 0; j < KMAX; ++j) {
        if (j >= p.k) break;
        const double d = x - p.mu[j];
        const double g = inv_sqrt_2pi / sqrt(p.var[j]) * exp(-0.5 * d * d / p.var[j]);
        w[j] = g * p.phi[j];
        den += w[j];
    }
    const double inv = 1.0 / den;
#pragma unroll
    for (int j = 0; j < KMAX; ++j)
        if (j < p.k) w[j] *= inv;
}

// Block sum of `cnt` doubles held per thread in v[]; thread 0 writes them.
template <int CNT>
__device__ __forceinline__ void block_sums(double (&v)[CNT], int cnt, double *__restrict__ out) {
    __shared__ double sh[EM_THREADS / 32][CNT];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
    for (int c = 0; c < CNT; ++c) {
        if (c >= cnt) break;
        double s = v[c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) sh[warp][c] = s;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int c = 0; c < cnt; ++c) {
            double s = 0.0;
            for (int w = 0; w < EM_THREADS / 32; ++w) s += sh[w][c];
            out[c] = s;
        }
    }
}

// Sum of logarithms as a running product: significands multiply, exponents
// add, and one log at the very end replaces one per sample.  Factors that are
// zero, subnormal, infinite or NaN go through log().
__device__ __forceinline__ double split_exponent(double f, long long &exps) {  // f normal, positive
    const long long b = __double_as_longlong(f);
    exps += (b >> 52) - 1023;
    return __longlong_as_double((b & 0x000fffffffffffffll) | 0x3ff0000000000000ll);  // in [1, 2)
}

// A number beyond FP64's normal range, or one whose products with others of
// its kind might leave it, is handled in FP64 instructions.
__device__ __forceinline__ bool tame(double x) {
    const int f = fx::field(x);
    return f >= 1 && f <= 2046;
}
constexpr int kNever = 1 << 16;  // exponent that no product brings back into range

__device__ const fx::Table g_exp_table = fx::make_table();

// One EM iteration.  Bound by FP64 issue (GB300 has two FP64 lanes per SM), so
// what is not a sum runs on the integer units, which issue 64 instructions for
// one of FP64 (fixed.cuh): exponent, exponential, weight, reciprocal and the
// product under the logarithm.  FP64 keeps d, the sum of the weights, w d and
// the three sums: 6 instructions per sample and component instead of 38.
// Component factors are formed once per iteration by the last block, and block
// sums go through shared memory (13 FP64 instructions per sum and block of 8
// warps instead of 40 by shuffles).  2 blocks of 8 warps per SM.  10^6 samples, 2
// components, us an iteration: two passes with a one-thread sum of the block
// partials 1154, one pass in FP64 instructions 131, as written 55
// (4 blocks of 4 warps 62, 4 of 8 60, 2 of 16 60); the FP64 pipe is busy 74 % of
// the time its SM works.
// K = 7 and 8 hold 50 and 56 KB of static shared memory, more than 48, which CUDA 13
// admits for sm_103a; at 188 and 210 registers one block fits an SM, and the grid
// runs in two waves (10^6 samples, 8 components: 222 us an iteration, two passes 2610).
// part: 3K sums, product, rest (doubles) and exponents, [3K + 3][blocks].
template <int K>
__global__ void __launch_bounds__(STEP_THREADS)
k_em_step(const double *__restrict__ x, long long m, EmParams *__restrict__ pp, EmState *__restrict__ st, double tol,
          double *__restrict__ part) {
    if (st->done || st->cancel) return;
    constexpr int W = 3 * K + 3, PROD = 3 * K, REST = 3 * K + 1, EXPS = 3 * K + 2, NW = STEP_THREADS / 32;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int nb = gridDim.x;
    __shared__ uint64_t table[128];
    static_assert(STEP_THREADS >= 128, "one table entry per thread");
    if (threadIdx.x < 128) table[threadIdx.x] = g_exp_table.t[threadIdx.x];
    double mu[K], v[3 * K];
    fx::Num amp[K], rate[K];  // weight is amp 2^(-rate d^2)
#pragma unroll
    for (int j = 0; j < K; ++j) {
        mu[j] = pp->mu[j];
        amp[j] = fx::unpack(pp->amp[j]);
        rate[j] = fx::mul(fx::unpack(pp->hiv[j]), fx::Num{fx::kLog2e, 0});
        if (!tame(pp->amp[j]) || !tame(pp->hiv[j])) rate[j].e = kNever;
        v[j] = v[K + j] = v[2 * K + j] = 0.0;
    }
    __syncthreads();
    fx::Num prod{1ull << 63, 0};
    double rest = 0.0;
    long long exps = 0;
    for (long long i = blockIdx.x * (long long)STEP_THREADS + threadIdx.x; i < m; i += (long long)nb * STEP_THREADS) {
        const double xi = x[i];
        double d[K], w[K], den = 0.0;
#pragma unroll
        for (int j = 0; j < K; ++j) {
            d[j] = xi - mu[j];
            const fx::Num a = fx::unpack(d[j]), t = fx::mul(fx::mul(a, a), rate[j]);
            fx::Num n{0, kNever};
            if (t.e <= 9) n = fx::mul(fx::exp2_neg(t, table), amp[j]);
            if (n.e >= -1022 && n.e <= 1000) w[j] = fx::pack(n);
            else w[j] = pp->amp[j] * exp(pp->hiv[j] * (d[j] * d[j]));
            den = j ? den + w[j] : w[0];
        }
        const bool normal = tame(den) && den > 0.0;
        const fx::Num dn = fx::unpack(den), inv = fx::reciprocal(dn);
        if (normal) {
            prod = fx::mul(prod, dn);
            exps += prod.e;
            prod.e = 0;
        } else {
            rest += log(den);
        }
#pragma unroll
        for (int j = 0; j < K; ++j) {
            const fx::Num n = fx::mul(fx::unpack(w[j]), inv);
            double r;
            if (normal && tame(w[j]) && n.e >= -1022) r = fx::pack(n);
            else r = w[j] * (1.0 / den);
            const double rd = r * d[j];
            v[j] += r;
            v[K + j] += rd;
            v[2 * K + j] += rd * d[j];
        }
    }
    // sums of the block, then of all blocks by the last one, in fixed order
    __shared__ double sh[W][STEP_THREADS];
    __shared__ bool last;
#pragma unroll
    for (int c = 0; c < 3 * K; ++c) sh[c][threadIdx.x] = v[c];
    sh[PROD][threadIdx.x] = fx::pack(prod);
    sh[REST][threadIdx.x] = rest;
    sh[EXPS][threadIdx.x] = __longlong_as_double(exps);
    __syncthreads();
    // column c of n values: sum, product or integer sum, in lane 0
    auto column = [&](int c, auto value, int n) {
        if (c == EXPS) {
            long long t = 0;
            for (int q = lane; q < n; q += 32) t += __double_as_longlong(value(q));
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
            return __longlong_as_double(t);
        }
        double t = c == PROD ? 1.0 : 0.0;
        for (int q = lane; q < n; q += 32) t = c == PROD ? t * value(q) : t + value(q);
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double u = __shfl_down_sync(0xffffffffu, t, o);
            t = c == PROD ? t * u : t + u;
        }
        return t;
    };
    for (int c = warp; c < W; c += NW) {
        const double t = column(c, [&](int q) { return sh[c][q]; }, STEP_THREADS);  // product: 256 factors up to 2
        if (lane == 0) {
            __stcg(part + (long long)c * nb + blockIdx.x, t);
            __threadfence();
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(&st->ticket, 1u) == unsigned(nb) - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    long long moved = 0;  // exponents taken off the blocks' products (then 2^nb bounds theirs, nb <= 304)
    for (int c = warp; c < W; c += NW) {
        const double *p = part + (long long)c * nb;
        const double t = column(
            c, [&](int q) { return c == PROD ? split_exponent(__ldcg(p + q), moved) : __ldcg(p + q); }, nb);
        if (lane == 0) sh[0][c] = t;
        if (c == PROD) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) moved += __shfl_down_sync(0xffffffffu, moved, o);
            if (lane == 0) sh[0][W] = __longlong_as_double(moved);
        }
    }
    __syncthreads();
    if (warp != 0) return;
    // lane j finishes component j, lane K the log-likelihood
    const double *tot = sh[0];
    const int j = lane < K ? lane : 0;
    const double s0 = tot[j], shift = tot[K + j] / s0, second = tot[2 * K + j] / s0;
    const bool cancel = __any_sync(0xffffffffu, second - shift * shift < second * (1.0 / 64.0));
    if (lane == 0) {
        st->ticket = 0u;
        if (cancel) st->cancel = 1;
    }
    if (cancel) return;
    if (lane < K) {
        const double phi = s0 / double(m), var = second - shift * shift;
        pp->phi[j] = phi;
        pp->mu[j] += shift;
        pp->var[j] = var;
        em_factor(phi, var, pp->amp[j], pp->hiv[j]);
    } else if (lane == K) {
        const long long exps = __double_as_longlong(tot[EXPS]) + __double_as_longlong(tot[W]);
        const double ll = (tot[REST] + (log(tot[PROD]) + double(exps) * 0.693147180559945309417)) / double(m);
        st->it++;
        st->ll = ll;
        if (tol > 0.0 && fabs(ll - st->prev) < tol) st->done = 1;
        st->prev = ll;
    }
}

// pass 1 partials per block: [sum w_j (k), sum w_j x (k), sum log den]
__global__ void __launch_bounds__(EM_THREADS)
k_em_pass1(const double *__restrict__ x, long long m, const EmParams *__restrict__ pp, double *__restrict__ part) {
    const EmParams p = *pp;
    double v[2 * KMAX + 1];
#pragma unroll
    for (int c = 0; c < 2 * KMAX + 1; ++c) v[c] = 0.0;
    for (long long i = blockIdx.x * (long long)EM_THREADS + threadIdx.x; i < m;
         i += (long long)gridDim.x * EM_THREADS) {
        double w[KMAX], den;
        const double xi = x[i];
        responsibilities(xi, p, w, den);
#pragma unroll
        for (int j = 0; j < KMAX; ++j)
            if (j < p.k) {
                v[j] += w[j];
                v[KMAX + j] += w[j] * xi;
            }
        v[2 * KMAX] += log(den);
    }
    block_sums<2 * KMAX + 1>(v, 2 * KMAX + 1, part + (long long)blockIdx.x * (2 * KMAX + 1));
}

// pass 2 partials per block: [sum w_j (x - mu_new_j)^2 (k)]
__global__ void __launch_bounds__(EM_THREADS)
k_em_pass2(const double *__restrict__ x, long long m, const EmParams *__restrict__ pp, double *__restrict__ part) {
    const EmParams p = *pp;
    double v[KMAX];
#pragma unroll
    for (int c = 0; c < KMAX; ++c) v[c] = 0.0;
    for (long long i = blockIdx.x * (long long)EM_THREADS + threadIdx.x; i < m;
         i += (long long)gridDim.x * EM_THREADS) {
        double w[KMAX], den;
        const double xi = x[i];
        responsibilities(xi, p, w, den);
#pragma unroll
        for (int j = 0; j < KMAX; ++j)
            if (j < p.k) {
                const double d = xi - p.mu_new[j];
                v[j] += w[j] * d * d;
            }
    }
    block_sums<KMAX>(v, KMAX, part + (long long)blockIdx.x * KMAX);
}

// Fixed-order totals of the block partials, one warp per sum; pass 1 sets
// mu_new and the log-likelihood, pass 2 phi and the variances, moves mu_new
// into mu and ends the iteration.
__global__ void __launch_bounds__(EM_THREADS)
k_em_finalize(const double *__restrict__ part, int nblocks, long long m, int pass, double tol,
              EmParams *__restrict__ pp, EmState *__restrict__ st, double *__restrict__ sw_keep) {
    __shared__ double tot[2 * KMAX + 1];
    const int W = pass == 1 ? 2 * KMAX + 1 : KMAX;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = warp; c < W; c += EM_THREADS / 32) {
        double s = 0.0;
        for (int b = lane; b < nblocks; b += 32) s += part[(long long)b * W + c];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) tot[c] = s;
    }
    __syncthreads();
    if (threadIdx.x != 0) return;
    EmParams &p = *pp;
    if (pass == 1) {
        for (int j = 0; j < p.k; ++j) {
            sw_keep[j] = tot[j];
            p.mu_new[j] = tot[KMAX + j] / tot[j];
        }
        st->ll = tot[2 * KMAX] / double(m);
    } else {
        for (int j = 0; j < p.k; ++j) {
            p.phi[j] = sw_keep[j] / double(m);
            p.mu[j] = p.mu_new[j];
            p.var[j] = tot[j] / sw_keep[j];
        }
        em_factors(p);
        st->it++;
        st->cancel = 0;
        if (tol > 0.0 && fabs(st->ll - st->prev) < tol) st->done = 1;
        st->prev = st->ll;
    }
}

template <int K>
void launch_em_step(int k, int nb, cudaStream_t s, const double *x, long long m, EmParams *pp, EmState *st, double tol,
                    double *part) {
    if (k == K) k_em_step<K><<<nb, STEP_THREADS, 0, s>>>(x, m, pp, st, tol, part);
    else if constexpr (K < KMAX) launch_em_step<K + 1>(k, nb, s, x, m, pp, st, tol, part);
}

glbm_status emfail(glbm_status s, const char *fmt, const char *detail) {
    snprintf(g_create_err, 512, fmt, detail);
    return s;
}

}  // namespace

extern "C" glbm_status glbm_em_gmm1d(const double *x, long long m, int k, double *phi, double *mu, double *var,
                                     int max_iter, double tol, int *iters, double *loglik, int device_ptrs,
                                     void *stream) {
    if (iters) *iters = 0;
    if (!x || !phi || !mu || !var || m < 1 || k < 1 || k > KMAX || max_iter < 0 || !std::isfinite(tol))
        return emfail(GLBM_EINVAL, "em_gmm1d: %s", "need x, m >= 1, 1 <= k <= 8, phi/mu/var and max_iter >= 0");
    EmParams hp{};
    hp.k = k;
    double fsum = 0.0;
    for (int j = 0; j < k; ++j) {
        if (!(phi[j] > 0.0) || !(var[j] > 0.0) || !std::isfinite(mu[j]))
            return emfail(GLBM_EINVAL, "em_gmm1d: %s", "initial fractions and variances must be > 0");
        hp.phi[j] = phi[j];
        hp.mu[j] = mu[j];
        hp.var[j] = var[j];
        fsum += phi[j];
    }
    for (int j = 0; j < k; ++j) hp.phi[j] /= fsum;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    const int nb = int(std::min<long long>((m + EM_THREADS - 1) / EM_THREADS, 152LL * 8));
    const int nbs = int(std::min<long long>((m + STEP_THREADS - 1) / STEP_THREADS, 152LL * STEP_BLOCKS));
    // one workspace: estimate, progress, Phi sums, block partials of either form
    const size_t parts = std::max(size_t(nbs) * (3 * k + 3), size_t(nb) * (2 * KMAX + 1));
    em_factors(hp);
    struct Head {
        EmParams p;
        EmState s;
        double sw[KMAX];
    };
    EmState hs{};
    hs.ll = hs.prev = -INFINITY;
    Head head{hp, hs, {}};
    double *dx = nullptr;
    Head *dh = nullptr;
    cudaError_t e = cudaSuccess;
    if (!device_ptrs) {
        e = cudaMalloc(&dx, sizeof(double) * m);
        if (e == cudaSuccess) e = cudaMemcpyAsync(dx, x, sizeof(double) * m, cudaMemcpyHostToDevice, st);
    }
    if (e == cudaSuccess) e = cudaMalloc(&dh, sizeof(Head) + sizeof(double) * parts);
    if (e == cudaSuccess) e = cudaMemcpyAsync(dh, &head, sizeof(Head), cudaMemcpyHostToDevice, st);
    double *part = reinterpret_cast<double *>(dh + 1);
    const double *xs = device_ptrs ? x : dx;
    // Iterations are enqueued in batches; the launches after one that
    // converged, or that asks for the two-pass form, return at once.
    int batch = tol > 0.0 ? 2 : max_iter;
    while (e == cudaSuccess && hs.it < max_iter && !hs.done) {
        const int n = std::min(batch, max_iter - hs.it);
        if (hs.cancel) {
            k_em_pass1<<<nb, EM_THREADS, 0, st>>>(xs, m, &dh->p, part);
            k_em_finalize<<<1, EM_THREADS, 0, st>>>(part, nb, m, 1, tol, &dh->p, &dh->s, dh->sw);
            k_em_pass2<<<nb, EM_THREADS, 0, st>>>(xs, m, &dh->p, part);
            k_em_finalize<<<1, EM_THREADS, 0, st>>>(part, nb, m, 2, tol, &dh->p, &dh->s, dh->sw);
        } else {
            for (int i = 0; i < n; ++i) launch_em_step<1>(k, nbs, st, xs, m, &dh->p, &dh->s, tol, part);
            batch = 2 * std::min(batch, 8);
        }
        e = cudaGetLastError();
        if (e == cudaSuccess) e = cudaMemcpyAsync(&hs, &dh->s, sizeof(EmState), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    }
    if (e == cudaSuccess) e = cudaMemcpyAsync(&hp, &dh->p, sizeof(EmParams), cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaStreamSynchronize(st);
    if (dx) cudaFree(dx);
    if (dh) cudaFree(dh);
    if (e != cudaSuccess) return emfail(GLBM_ECUDA, "em_gmm1d: %s", cudaGetErrorString(e));
    bool finite = true;
    for (int j = 0; j < k; ++j) {
        phi[j] = hp.phi[j];
        mu[j] = hp.mu[j];
        var[j] = hp.var[j];
        finite = finite && std::isfinite(phi[j]) && std::isfinite(mu[j]) && std::isfinite(var[j]);
    }
    if (iters) *iters = hs.it;
    if (loglik) *loglik = max_iter > 0 ? hs.ll : NAN;
    // a component that collapses onto a single sample has zero variance and
    // the next E-step is undefined
    if (!finite) return emfail(GLBM_ENAN, "em_gmm1d: %s", "estimate not finite (a component collapsed)");
    return GLBM_OK;
}
