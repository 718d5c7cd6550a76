// glbm_kernels.cuh -- shared by glbm.cu (single lattice) and batch.cu (many lattices).
// Device code of the GB300 (sm_103a) generalized lattice Boltzmann model
// (GLBM) time loop of Wang, Chen, Kang & Rahman, arXiv:1601.00704, Sec. 2.3.
//
// Hot path: one fused pull-stream + collide kernel per time step (Eq. 29 with
// Eqs. 27, 30-37) over a structure-of-arrays distribution layout, followed every
// chunk by a deterministic FP64 mean-velocity reduction that stays on the
// device.  The C ABI is declared in include/glbm.h.
//
// Design notes
//  * Distributions are stored as deviations g_i = f_i - w_i (rho0 = 1).  At
//    the Darcy velocities of shale media (u ~ 1e-9 lattice units) the
//    momentum signal sits ~8 decades below f_i ~ w_i; deviations keep it
//    inside FP32 (and FP16/BF16 with a power-of-two scale) precision.
//  * Layout: plane i (D2Q9 order below) holds g_i for node n = y*nx + x; the
//    plane stride is nx*ny rounded up to 64 elements, so every plane and, when
//    nx is a multiple of the vector width, every row starts 16-byte aligned.
//  * Each thread owns VEC consecutive nodes of one row (VEC*sizeof(T) = 16 B)
//    and moves them with 128-bit loads/stores.  Populations with e_x = +-1
//    need the x-1 / x+1 neighbour: it comes from the adjacent lane by a warp
//    shuffle; lanes 0/31 and the periodic row ends fetch one scalar.  A scalar
//    (VEC = 1) instantiation serves lattices whose nx is not a multiple of VEC.
//  * Per-node coefficients are packed once per medium (Eqs. 36-37):
//      alpha = eps*nu/K   (c0 = 1/2 + alpha/4, Darcy drag alpha*u),
//      eps, beta = eps*F_eps/sqrt(K)  (c1 = beta/2, only with Forchheimer).
//    Storing alpha rather than c0 keeps full relative precision of the drag
//    for nearly clear nodes, where 4*c0 - 2 would cancel.
//  * Halfway bounce-back walls at y = -1/2 and y = ny-1/2 and periodic x are
//    index arithmetic inside the kernel; no ghost layers, no extra bytes.
//  * The velocity solve (Eqs. 32-35) uses explicitly rounded intrinsics so
//    the velocity export kernel reproduces the step kernel's u bit for bit.
//  * step_body() is the whole per-thread time step; k_step (one lattice) and
//    k_batch_step (many lattices, batch.cu) only map blocks to rows.
//  * Kernels that run once per medium or per export (validation, coefficient
//    packing, equilibrium start, FP16 rescale, f export) are in
//    setup_kernels.cuh, so this file holds the time loop alone.

#pragma once

#include "odd_constants.h"

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>
#include <utility>

namespace {

// ---------------------------------------------------------------------------
// D2Q9: e0=(0,0); e1..e4=(1,0),(0,1),(-1,0),(0,-1);
//       e5..e8=(1,1),(-1,1),(-1,-1),(1,-1); w = 4/9, 1/9 (x4), 1/36 (x4).
// ---------------------------------------------------------------------------
__host__ __device__ constexpr int cx(int i) {
    return (i == 1 || i == 5 || i == 8) ? 1 : ((i == 3 || i == 6 || i == 7) ? -1 : 0);
}
__host__ __device__ constexpr int cy(int i) {
    return (i == 2 || i == 5 || i == 6) ? 1 : ((i == 4 || i == 7 || i == 8) ? -1 : 0);
}
__host__ __device__ constexpr int opp(int i) {
    return i == 0 ? 0 : (i <= 4 ? ((i + 1) % 4) + 1 : ((i - 3) % 4) + 5);
}
template <typename R>
__host__ __device__ constexpr R wgt(int i) {
    return i == 0 ? R(4) / R(9) : (i <= 4 ? R(1) / R(9) : R(1) / R(36));
}
static_assert(opp(1) == 3 && opp(2) == 4 && opp(3) == 1 && opp(4) == 2, "opp");
static_assert(opp(5) == 7 && opp(6) == 8 && opp(7) == 5 && opp(8) == 6, "opp");

// ---------------------------------------------------------------------------
// Explicitly rounded arithmetic (no FMA contraction differences between
// kernels that must agree bitwise).
// ---------------------------------------------------------------------------
__device__ __forceinline__ float radd(float a, float b) { return __fadd_rn(a, b); }
__device__ __forceinline__ float rsub(float a, float b) { return __fsub_rn(a, b); }
__device__ __forceinline__ float rmul(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float rfma(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ float rdiv(float a, float b) { return __fdiv_rn(a, b); }
__device__ __forceinline__ float rsqrt_(float a) { return __fsqrt_rn(a); }
__device__ __forceinline__ double radd(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ double rsub(double a, double b) { return __dsub_rn(a, b); }
__device__ __forceinline__ double rmul(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double rfma(double a, double b, double c) { return __fma_rn(a, b, c); }
__device__ __forceinline__ double rdiv(double a, double b) { return __ddiv_rn(a, b); }
__device__ __forceinline__ double rsqrt_(double a) { return __dsqrt_rn(a); }
// Reciprocals of rho ~ 1, 2*c0 >= 1 and eps in (0, 1]: the hardware
// approximation (within 1 ulp) is ample and a fraction of IEEE rcp's cost.
__device__ __forceinline__ float rrcp(float a) {
    float r;  // hardware approximate reciprocal (within 1 ulp); every argument here is >= 1/2
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
    return r;
}
__device__ __forceinline__ double rrcp(double a) { return __drcp_rn(a); }

// ---------------------------------------------------------------------------
// Storage formats.  R is the collision arithmetic type.
// ---------------------------------------------------------------------------
// Stochastic rounding: round |x| up with probability equal to the dropped
// fraction, using uniform random bits r; unbiased in expectation, so slow
// modes whose per-step change is below half an ulp do not freeze.
// FP16: stochastic in the normal range [2^-14, 65504]; values below it are
// rounded to nearest -- with the scale keeping the largest stored magnitude
// near 2^12 they lie 2^26 below it, where a biased last bit is immaterial --
// and overflow, inf and NaN convert as usual.
__device__ __forceinline__ __half f2h_sr(float x, uint32_t r) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t a = b & 0x7fffffffu;
    const uint32_t t = (b + (r & 0x1FFFu)) & ~0x1FFFu;  // drop 13 mantissa bits
    const bool normal = a - 0x38800000u < 0x477fe000u - 0x38800000u;
    return normal ? __float2half_rz(__uint_as_float(t)) : __float2half_rn(x);
}
__device__ __forceinline__ __nv_bfloat16 f2bf_sr(float x, uint32_t r) {
    const uint32_t b = __float_as_uint(x);
    const uint32_t t = (b + (r & 0xFFFFu)) & 0xFFFF0000u;  // drop 16 mantissa bits
    const bool finite = (b & 0x7f800000u) != 0x7f800000u;
    return finite ? __float2bfloat16_rz(__uint_as_float(t)) : __float2bfloat16_rn(x);
}

template <typename T> struct Store;
template <> struct Store<float> {
    using R = float;
    static constexpr bool kSmall = false;
    __device__ static float ld(float v, float) { return v; }
    __device__ static float st(float v, float) { return v; }
    __device__ static float st_sr(float v, float, uint32_t) { return v; }
};
template <> struct Store<double> {
    using R = double;
    static constexpr bool kSmall = false;
    __device__ static double ld(double v, double) { return v; }
    __device__ static double st(double v, double) { return v; }
    __device__ static double st_sr(double v, double, uint32_t) { return v; }
};
template <> struct Store<__half> {
    using R = float;
    static constexpr bool kSmall = true;
    __device__ static float ld(__half v, float inv_s) { return __half2float(v) * inv_s; }
    __device__ static __half st(float v, float s) { return __float2half_rn(v * s); }
    __device__ static __half st_sr(float v, float s, uint32_t r) { return f2h_sr(v * s, r); }
    static constexpr bool kScaled = true;
    // Two scaled values -> packed pair with hardware stochastic rounding
    // (cvt.rs): `lo` lands in the low half (lower address), `hi` in the high.
    __device__ static uint32_t pack_sr(float lo, float hi, uint32_t rbits) {
        uint32_t d;
        asm("cvt.rs.f16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
        return d;
    }
};
template <> struct Store<__nv_bfloat16> {
    using R = float;
    static constexpr bool kSmall = true;
    // BF16 has FP32's exponent range: stored unscaled (the scale is always 1)
    __device__ static float ld(__nv_bfloat16 v, float) { return __bfloat162float(v); }
    __device__ static __nv_bfloat16 st(float v, float) { return __float2bfloat16_rn(v); }
    __device__ static __nv_bfloat16 st_sr(float v, float, uint32_t r) { return f2bf_sr(v, r); }
    static constexpr bool kScaled = false;
    __device__ static uint32_t pack_sr(float lo, float hi, uint32_t rbits) {
        uint32_t d;
        asm("cvt.rs.bf16x2.f32 %0, %1, %2, %3;" : "=r"(d) : "f"(hi), "f"(lo), "r"(rbits));
        return d;
    }
};

// Nodes per thread: 16-byte vectors for 32/64-bit storage, 8-byte vectors
// (4 nodes) for 16-bit storage.
template <typename T>
constexpr int kVecOf = sizeof(T) == 2 ? 4 : int(16 / sizeof(T));

// Integer hash ("lowbias32" multiply-xorshift) for the stochastic rounding
// bits: one 32-bit word per (node, step, population pair).
__host__ __device__ __forceinline__ uint32_t mix32(uint32_t x) {
    x ^= x >> 16;
    x *= 0x7feb352du;
    x ^= x >> 15;
    x *= 0x846ca68bu;
    x ^= x >> 16;
    return x;
}

template <typename R>
struct Phys {
    R omega;     // 1/tau
    R A;         // 1 - 1/(2 tau)
    R gx, gy;    // external force G
    R scale;     // storage scale S (stored = g*S); 1 for FP32/FP64
    R inv_scale; // 1/S
    uint32_t step_key;  // per-step key of the stochastic-rounding hash
    int sr;             // 16-bit storage: 1 = stochastic rounding, 0 = nearest
    // 16-bit storage inside a replayed CUDA graph: when `clock` is set the
    // kernel forms its key from the device step counter instead,
    // step_key = mix32((*clock + step_off) * 0x9E3779B9 + seed), the same
    // value the host forms for step *clock + step_off.
    const unsigned *clock = nullptr;
    uint32_t step_off = 0;
    uint32_t seed = 0;
    uint32_t step_key2 = 0;  // key of the following step, for k_pair
    uint32_t tstep = 0;      // the step itself, for kernels that form several keys
    OddConstants<R> odd{};   // FP32 and FP64 storage: the odd half's constants
};

// Stochastic-rounding key of time step t (host and device agree).
__host__ __device__ __forceinline__ uint32_t step_key_of(uint32_t t, uint32_t seed) {
    return mix32(t * 0x9E3779B9u + seed);
}

struct Geo {
    int nx, ny;
    long long plane;  // elements per population plane
    int bpr;          // blocks per row
};

// Vector moves of 8 bytes or a multiple of 16 bytes.  CG: load through L2
// only (ld.global.cg), for data that other blocks of the same launch wrote
// (the persistent batch kernel), which a non-coherent L1 line could hide.
template <typename X, int N, bool CG = false>
__device__ __forceinline__ void ld16(const X *__restrict__ p, X (&out)[N]) {
    constexpr int B = int(N * sizeof(X));
    static_assert(B == 8 || B % 16 == 0, "8-byte or 16-byte multiple");
    if constexpr (B == 8) {
        uint2 u = CG ? __ldcg(reinterpret_cast<const uint2 *>(p)) : *reinterpret_cast<const uint2 *>(p);
        memcpy(&out[0], &u, 8);
    } else {
#pragma unroll
        for (int j = 0; j < B / 16; ++j) {
            uint4 u = CG ? __ldcg(reinterpret_cast<const uint4 *>(p) + j) : reinterpret_cast<const uint4 *>(p)[j];
            memcpy(&out[j * (16 / sizeof(X))], &u, 16);
        }
    }
}
// One element, optionally through L2 only (see ld16).
template <bool CG, typename X>
__device__ __forceinline__ X ld1(const X *p) {
    if constexpr (CG) {
        if constexpr (sizeof(X) == 2) {
            const unsigned short u = __ldcg(reinterpret_cast<const unsigned short *>(p));
            X v;
            memcpy(&v, &u, 2);
            return v;
        } else {
            return __ldcg(p);
        }
    } else {
        return *p;
    }
}
template <typename X, int N>
__device__ __forceinline__ void st16(X *__restrict__ p, const X (&in)[N]) {
    constexpr int B = int(N * sizeof(X));
    if constexpr (B == 8) {
        uint2 u;
        memcpy(&u, &in[0], 8);
        __stcs(reinterpret_cast<uint2 *>(p), u);
    } else {
#pragma unroll
        for (int j = 0; j < B / 16; ++j) {
            uint4 u;
            memcpy(&u, &in[j * (16 / sizeof(X))], 16);
            __stcs(reinterpret_cast<uint4 *>(p) + j, u);
        }
    }
}

// ---------------------------------------------------------------------------
// Per-node physics.
// ---------------------------------------------------------------------------

// Eqs. 32, 33, 35, 36, 37, 34: density deviation and the node velocity from
// the streamed deviations g[9].  Explicit rounding: see file header.
template <typename R, bool FORCH>
__device__ __forceinline__ void node_velocity(const R (&g)[9], R alpha, R eps, R beta,
                                              const Phys<R> &ph, R &drho, R &ux, R &uy) {
    drho = radd(radd(radd(g[0], radd(g[1], g[3])), radd(g[2], g[4])),
                radd(radd(g[5], g[7]), radd(g[6], g[8])));
    const R mx = radd(radd(rsub(g[1], g[3]), rsub(g[5], g[7])), rsub(g[8], g[6]));
    const R my = radd(radd(rsub(g[2], g[4]), rsub(g[5], g[7])), rsub(g[6], g[8]));
    const R rho = radd(R(1), drho);
    const R inv_rho = rrcp(rho);
    const R heps = rmul(R(0.5), eps);
    const R vx = rfma(mx, inv_rho, rmul(heps, ph.gx));
    const R vy = rfma(my, inv_rho, rmul(heps, ph.gy));
    const R c0 = rfma(R(0.25), alpha, R(0.5));
    R den;
    if (FORCH) {
        const R c1 = rmul(R(0.5), beta);
        const R vmag = rsqrt_(rfma(vx, vx, rmul(vy, vy)));
        den = radd(c0, rsqrt_(rfma(c1, vmag, rmul(c0, c0))));
    } else {
        den = rfma(R(0.5), alpha, R(1));  // 2*c0
    }
    const R inv_den = rrcp(den);
    ux = rmul(vx, inv_den);
    uy = rmul(vy, inv_den);
}

// Eq. 27 force, Eq. 30 equilibrium and Eq. 31 forcing (with the 1/eps on the
// u.F term, the mass-conserving reading), then the BGK update of Eq. 29,
// g* = g + (g_eq - g)/tau + F_i, for FP32 and FP64 storage.
//
// Rounding: at Darcy velocities every deviation is dominated by its density
// carrier w_i (rho - 1), several decades above the velocity terms.  The update
// is therefore regrouped as
//     g* = w d + [ (1 - 1/tau)(g - w d) + w (even +- odd) ],   d = rho - 1,
// where the bracket holds only small terms and w d enters by fused
// multiply-add, so the carrier is rounded once per population instead of at
// every term.
//
// Operation count: with H = 1.5 u/tau + 3A F, J = 3 u/tau + 3A F and
// A = 1 - 1/(2 tau) the direction sums of Eqs. 30 and 31 collapse to
//     w even = w (3 rho/eps) [ (e.u)(e.H) - (u.H)/3 ],   w odd = w rho (e.J),
// shared by opposite directions: 106 FP32 operations per node with the mass
// closure below.  The form before it (separate f_eq and F_i terms, and TwoSum
// sums of the populations before and after the collision) took 241 and was
// bound by them where the lattice fits L2: 1024^2 FP32 10.8 -> 8.8 us a step.
// w rho J is c rho (a u + b F) with constants whose rounding loses no momentum
// (odd_constants.h); H goes with the same b, so that w (3/eps) becomes 3c/eps.
template <typename R>
__device__ __forceinline__ R collide_pair(R &gi, R &gj, R w, R d, R k1, R eu, R eH, R eJ, R q, R we, R wo) {
    const R ev = rmul(we, rfma(eu, eH, -q));
    const R ni = rfma(w, d, rfma(k1, rfma(-w, d, gi), rfma(wo, eJ, ev)));
    const R nj = rfma(w, d, rfma(k1, rfma(-w, d, gj), rfma(-wo, eJ, ev)));
    const R lost = radd(rsub(gi, ni), rsub(gj, nj));  // what this pair hands to the rest population
    gi = ni;
    gj = nj;
    return lost;
}

template <typename R, bool FORCH>
__device__ __forceinline__ void collide(R (&g)[9], R alpha, R eps, R beta,
                                        const Phys<R> &ph, R &ux, R &uy) {
    R drho;
    node_velocity<R, FORCH>(g, alpha, eps, beta, ph, drho, ux, uy);
    const R rho = radd(R(1), drho);
    R drag = alpha;
    if (FORCH) drag = rfma(beta, rsqrt_(rfma(ux, ux, rmul(uy, uy))), alpha);
    const R Fx = rfma(-drag, ux, rmul(eps, ph.gx));
    const R Fy = rfma(-drag, uy, rmul(eps, ph.gy));
    const R k1 = R(1) - ph.omega, omJ = ph.odd.a, omH = R(0.5) * omJ;
    const R AFx = rmul(ph.odd.b, Fx), AFy = rmul(ph.odd.b, Fy);
    const R Hx = rfma(omH, ux, AFx), Hy = rfma(omH, uy, AFy);
    const R Jx = rfma(omJ, ux, AFx), Jy = rfma(omJ, uy, AFy);
    const R q = rmul(R(1.0 / 3.0), rfma(ux, Hx, rmul(uy, Hy)));
    // weights of the axis class (w = 1/9) and the diagonal class (1/36)
    const R we1 = rmul(R(3) * ph.odd.c, rmul(rrcp(eps), rho)), we2 = rmul(R(0.25), we1);
    const R wo1 = rmul(ph.odd.c, rho), wo2 = rmul(R(0.25), wo1);
    const R w1 = wgt<R>(1), w2 = R(0.25) * wgt<R>(1);
    // Mass closure: the collision conserves each node's mass exactly in
    // arithmetic, but rounding the nine stored populations does not, and the
    // slow pressure mode integrates that per-node error over thousands of
    // steps.  The rest population therefore takes up exactly what the eight
    // moving ones lose, g0* = g0 + sum_i (g_i - g_i*): each difference is of
    // neighbouring densities (exact by Sterbenz's lemma once within a factor
    // of two), so one rounding per node remains instead of nine: errors 30x below
    // the unclosed update's.  Against FP64, relative to the separate f_eq and F_i
    // terms with TwoSum sums before and after, geometric means over tau = 0.55 .. 2:
    // four two-phase media velocity 0.65, density 0.46; blocks of clear and porous
    // rock (35 lattices of 24 to 48 nodes a side) 0.66 and 0.88 +- 0.02, with TwoSum
    // sums 0.77; clear channels, where rounding scatters tenfold from tau to tau,
    // 0.95 and 0.63.
    const R l1 = collide_pair<R>(g[1], g[3], w1, drho, k1, ux, Hx, Jx, q, we1, wo1);
    const R l2 = collide_pair<R>(g[2], g[4], w1, drho, k1, uy, Hy, Jy, q, we1, wo1);
    const R l5 = collide_pair<R>(g[5], g[7], w2, drho, k1, radd(ux, uy), radd(Hx, Hy), radd(Jx, Jy), q, we2, wo2);
    const R l6 = collide_pair<R>(g[6], g[8], w2, drho, k1, rsub(uy, ux), rsub(Hy, Hx), rsub(Jy, Jx), q, we2, wo2);
    g[0] = radd(g[0], radd(radd(l1, l2), radd(l5, l6)));
}

// The same update for 16-bit storage, whose own rounding (2^-8 / 2^-11)
// dwarfs any FP32 regrouping error: every population is k1 g + c_i with
//   c_i = w_i [om (rho-1) + om rho (3 e.u + 9/(2 eps)(e.u)^2 - 3/(2 eps) u^2)
//              + rho A (3 e.F + 9/eps (e.u)(e.F) - 3/eps u.F)],
// folded per weight class into c = C + e.u (P e.u + Q e.F) +- (T e.u + U e.F)
// (even part C + ..., odd part T e.u + U e.F); w_diagonal = w_axis / 4 and
// w_0 = 4 w_axis, so the other classes are exact power-of-two multiples.
template <typename R, bool FORCH>
__device__ __forceinline__ void collide_small(R (&g)[9], R alpha, R eps, R beta,
                                              const Phys<R> &ph, R &ux, R &uy) {
    R drho;
    node_velocity<R, FORCH>(g, alpha, eps, beta, ph, drho, ux, uy);
    const R rho = R(1) + drho;
    R Fx = eps * ph.gx - alpha * ux;
    R Fy = eps * ph.gy - alpha * uy;
    if (FORCH) {
        const R bu = beta * sqrt(ux * ux + uy * uy);
        Fx -= bu * ux;
        Fy -= bu * uy;
    }
    const R om = ph.omega, k1 = R(1) - om;
    const R w1 = R(1.0 / 9.0);
    const R cA = R(3) * w1 * ph.A;    // 3 w A
    const R cO = R(1.5) * w1 * om;    // (3/2) w om
    const R ier = rrcp(eps) * rho;    // rho / eps
    const R uu = ux * ux + uy * uy, uF = ux * Fx + uy * Fy;
    const R C1 = (w1 * om) * drho - ier * (cA * uF + cO * uu);
    const R P1 = (R(3) * cO) * ier, Q1 = (R(3) * cA) * ier;
    const R T1 = (R(2) * cO) * rho, U1 = cA * rho;
    g[0] = k1 * g[0] + R(4) * C1;
    auto pair = [&](R &gi, R &gj, R eu, R eF, R s) {
        const R E = s * (C1 + eu * (P1 * eu + Q1 * eF));
        const R O = s * (T1 * eu + U1 * eF);
        gi = k1 * gi + (E + O);
        gj = k1 * gj + (E - O);
    };
    pair(g[1], g[3], ux, Fx, R(1));
    pair(g[2], g[4], uy, Fy, R(1));
    pair(g[5], g[7], ux + uy, Fx + Fy, R(0.25));
    pair(g[6], g[8], uy - ux, Fy - Fx, R(0.25));
}

// ---------------------------------------------------------------------------
// The same collisions for two nodes at once on packed FP32 pairs
// (add/mul/fma.rn.f32x2): the lane rate is that of the scalar instructions,
// but each pair takes one issue slot, and the multi-step kernels are bound by
// issue.  Every operation and its rounding is that of the scalar functions
// above (negated factors stand in for subtractions), so the bits are theirs.
// ---------------------------------------------------------------------------
struct f2 {
    unsigned long long v;
};
__host__ __device__ __forceinline__ f2 mk2(float lo, float hi) {
#ifdef __CUDA_ARCH__
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r.v) : "f"(lo), "f"(hi));
    return r;
#else
    uint32_t a, b;
    memcpy(&a, &lo, 4);
    memcpy(&b, &hi, 4);
    return f2{(unsigned long long)b << 32 | a};
#endif
}
__host__ __device__ __forceinline__ f2 bc2(float x) { return mk2(x, x); }
__device__ __forceinline__ float lo2(f2 a) {
    return __uint_as_float(uint32_t(a.v));
}
__device__ __forceinline__ float hi2(f2 a) {
    return __uint_as_float(uint32_t(a.v >> 32));
}
__device__ __forceinline__ f2 radd(f2 a, f2 b) {
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 rsub(f2 a, f2 b) {
    f2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 rmul(f2 a, f2 b) {
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r.v) : "l"(a.v), "l"(b.v));
    return r;
}
__device__ __forceinline__ f2 rfma(f2 a, f2 b, f2 c) {
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r.v) : "l"(a.v), "l"(b.v), "l"(c.v));
    return r;
}
__device__ __forceinline__ f2 rrcp(f2 a) { return mk2(rrcp(lo2(a)), rrcp(hi2(a))); }
__device__ __forceinline__ f2 rsqrt_(f2 a) { return mk2(rsqrt_(lo2(a)), rsqrt_(hi2(a))); }

// Launch constants as pairs, made on the host so that they sit in the
// constant bank.
struct Pair2 {
    f2 one, half, quarter, hgx, hgy, ngx, ngy, k1;
    f2 omH, omJ, nA3, nthird, we, wo, nwo, w1, nw1, w2, nw2;  // 32-bit storage
    f2 cA, ncO, w1om, four, cO3, ncA3, cO2, ncA;     // 16-bit storage
    f2 inv_s;
};
inline Pair2 make_pair2(const Phys<float> &p) {
    Pair2 c;
    const float w1 = 1.0f / 9.0f, om = p.omega, cA = (3.0f * w1) * p.A, cO = (1.5f * w1) * om;
    c.one = bc2(1.0f), c.half = bc2(0.5f), c.quarter = bc2(0.25f);
    const float gx = p.gx * p.scale, gy = p.gy * p.scale;  // FP16: with the storage scale (else 1)
    c.hgx = bc2(0.5f * gx), c.hgy = bc2(0.5f * gy), c.ngx = bc2(-gx), c.ngy = bc2(-gy);
    c.k1 = bc2(1.0f - om);
    c.omH = bc2(0.5f * p.odd.a), c.omJ = bc2(p.odd.a), c.nA3 = bc2(-p.odd.b);
    c.nthird = bc2(-(1.0f / 3.0f)), c.we = bc2(3.0f * p.odd.c), c.wo = bc2(p.odd.c), c.nwo = bc2(-p.odd.c);
    c.w1 = bc2(w1), c.nw1 = bc2(-w1);
    c.w2 = bc2(0.25f * w1), c.nw2 = bc2(-0.25f * w1);
    c.cA = bc2(cA), c.ncA = bc2(-cA), c.ncO = bc2(-cO), c.w1om = bc2(w1 * om), c.four = bc2(4.0f);
    c.cO3 = bc2(3.0f * cO), c.ncA3 = bc2(-(3.0f * cA)), c.cO2 = bc2(2.0f * cO);
    c.inv_s = bc2(p.inv_scale);
    return c;
}

// node_velocity for a pair.  SCALED: populations as stored in FP16, g S with S
// a power of two.  A power of two commutes with every rounding, so the whole
// update runs on S drho, S u and S F (the launch constants bring S G) and S
// leaves only rho, the products of two of them (rho / eps in collide_small2) and
// the square roots' arguments: 2 multiplications (4 with Forchheimer) instead of
// one per population on the way in and on the way out, and the same bits (2048^2
// FP16 27.0 -> 25.2 us a step).  Nothing is multiplied by S rho / eps, which
// leaves FP32's range where eps^2 G is below 1e-35.
template <bool FORCH, bool SCALED = false>
__device__ __forceinline__ void node_velocity2(const f2 (&g)[9], f2 alpha, f2 eps, f2 beta, const Pair2 &c, f2 &drho,
                                               f2 &rho, f2 &ux, f2 &uy) {
    drho = radd(radd(radd(g[0], radd(g[1], g[3])), radd(g[2], g[4])), radd(radd(g[5], g[7]), radd(g[6], g[8])));
    rho = radd(c.one, SCALED ? rmul(drho, c.inv_s) : drho);
    const f2 d57 = rsub(g[5], g[7]), d86 = rsub(g[8], g[6]);
    const f2 mx = radd(radd(rsub(g[1], g[3]), d57), d86);
    const f2 my = rsub(radd(rsub(g[2], g[4]), d57), d86);
    const f2 ir = rrcp(rho);
    const f2 vx = rfma(mx, ir, rmul(eps, c.hgx)), vy = rfma(my, ir, rmul(eps, c.hgy));
    f2 den;
    if (FORCH) {
        const f2 c0 = rfma(c.quarter, alpha, c.half), c1 = rmul(c.half, beta);
        f2 vmag = rsqrt_(rfma(vx, vx, rmul(vy, vy)));
        if (SCALED) vmag = rmul(vmag, c.inv_s);
        den = radd(c0, rsqrt_(rfma(c1, vmag, rmul(c0, c0))));
    } else {
        den = rfma(c.half, alpha, c.one);
    }
    const f2 iden = rrcp(den);
    ux = rmul(vx, iden);
    uy = rmul(vy, iden);
}

__device__ __forceinline__ f2 collide_pair2(f2 &gi, f2 &gj, f2 w, f2 nw, f2 d, f2 k1, f2 eu, f2 eH, f2 eJ, f2 nq,
                                            f2 we, f2 wo, f2 nwo) {
    const f2 ev = rmul(we, rfma(eu, eH, nq));
    const f2 ni = rfma(w, d, rfma(k1, rfma(nw, d, gi), rfma(wo, eJ, ev)));
    const f2 nj = rfma(w, d, rfma(k1, rfma(nw, d, gj), rfma(nwo, eJ, ev)));
    const f2 lost = radd(rsub(gi, ni), rsub(gj, nj));
    gi = ni;
    gj = nj;
    return lost;
}

// collide for a pair.
template <bool FORCH>
__device__ __forceinline__ void collide2(f2 (&g)[9], f2 alpha, f2 eps, f2 beta, const Pair2 &c) {
    f2 drho, rho, ux, uy;
    node_velocity2<FORCH>(g, alpha, eps, beta, c, drho, rho, ux, uy);
    f2 drag = alpha;
    if (FORCH) drag = rfma(beta, rsqrt_(rfma(ux, ux, rmul(uy, uy))), alpha);
    const f2 AFx = rmul(c.nA3, rfma(drag, ux, rmul(eps, c.ngx)));  // -3A (-F)
    const f2 AFy = rmul(c.nA3, rfma(drag, uy, rmul(eps, c.ngy)));
    const f2 Hx = rfma(c.omH, ux, AFx), Hy = rfma(c.omH, uy, AFy);
    const f2 Jx = rfma(c.omJ, ux, AFx), Jy = rfma(c.omJ, uy, AFy);
    const f2 nq = rmul(c.nthird, rfma(ux, Hx, rmul(uy, Hy)));
    const f2 we1 = rmul(c.we, rmul(rrcp(eps), rho)), we2 = rmul(c.quarter, we1);
    const f2 wo1 = rmul(c.wo, rho), wo2 = rmul(c.quarter, wo1);
    const f2 nwo1 = rmul(c.nwo, rho), nwo2 = rmul(c.quarter, nwo1);
    const f2 l1 = collide_pair2(g[1], g[3], c.w1, c.nw1, drho, c.k1, ux, Hx, Jx, nq, we1, wo1, nwo1);
    const f2 l2 = collide_pair2(g[2], g[4], c.w1, c.nw1, drho, c.k1, uy, Hy, Jy, nq, we1, wo1, nwo1);
    const f2 l5 = collide_pair2(g[5], g[7], c.w2, c.nw2, drho, c.k1, radd(ux, uy), radd(Hx, Hy), radd(Jx, Jy), nq, we2,
                                wo2, nwo2);
    const f2 l6 = collide_pair2(g[6], g[8], c.w2, c.nw2, drho, c.k1, rsub(uy, ux), rsub(Hy, Hx), rsub(Jy, Jx), nq, we2,
                                wo2, nwo2);
    g[0] = radd(g[0], radd(radd(l1, l2), radd(l5, l6)));
}

// collide_small for a pair (SCALED: see node_velocity2).
template <bool FORCH, bool SCALED>
__device__ __forceinline__ void collide_small2(f2 (&g)[9], f2 alpha, f2 eps, f2 beta, const Pair2 &c) {
    f2 drho, rho, ux, uy;
    node_velocity2<FORCH, SCALED>(g, alpha, eps, beta, c, drho, rho, ux, uy);
    f2 nFx = rfma(eps, c.ngx, rmul(alpha, ux)), nFy = rfma(eps, c.ngy, rmul(alpha, uy));  // -F
    const f2 uu = rfma(ux, ux, rmul(uy, uy));
    if (FORCH) {
        const f2 umag = SCALED ? rmul(rsqrt_(uu), c.inv_s) : rsqrt_(uu);
        const f2 bu = rmul(beta, umag);
        nFx = rfma(bu, ux, nFx);
        nFy = rfma(bu, uy, nFy);
    }
    const f2 ier = rmul(rrcp(eps), SCALED ? rmul(rho, c.inv_s) : rho);
    const f2 nuF = rfma(ux, nFx, rmul(uy, nFy));
    const f2 C1 = rfma(c.w1om, drho, rmul(ier, rfma(c.ncO, uu, rmul(c.cA, nuF))));
    const f2 P1 = rmul(c.cO3, ier), Q1 = rmul(c.ncA3, ier);
    const f2 T1 = rmul(c.cO2, rho), U1 = rmul(c.ncA, rho);
    g[0] = rfma(c.k1, g[0], rmul(c.four, C1));
    auto pair = [&](f2 &gi, f2 &gj, f2 eu, f2 neF, bool diag) {
        f2 E = rfma(eu, rfma(P1, eu, rmul(Q1, neF)), C1);
        f2 O = rfma(T1, eu, rmul(U1, neF));
        if (diag) E = rmul(c.quarter, E), O = rmul(c.quarter, O);
        gi = rfma(c.k1, gi, radd(E, O));
        gj = rfma(c.k1, gj, rsub(E, O));
    };
    pair(g[1], g[3], ux, nFx, false);
    pair(g[2], g[4], uy, nFy, false);
    pair(g[5], g[7], radd(ux, uy), radd(nFx, nFy), true);
    pair(g[6], g[8], rsub(uy, ux), rsub(nFy, nFx), true);
}

// Per-node coefficients of VEC consecutive nodes.
template <typename R, int VEC>
__device__ __forceinline__ void load_coef(const R *__restrict__ p, R (&c)[VEC]) {
    if constexpr (VEC == 1) c[0] = p[0];
    else ld16<R, VEC>(p, c);
}

// ---------------------------------------------------------------------------
// Pull-streaming gather of VEC consecutive nodes (x0..x0+VEC-1, row y) and
// of their coefficients (alpha, eps and, with Forchheimer, beta at node n0).
// Phase 1 issues every load of the thread (9 vectors + up to 6 edge scalars +
// 2-3 coefficient vectors) before phase 2 consumes any, so all of them are in
// flight together.
// ---------------------------------------------------------------------------
// INTERIOR: 0 < y < ny-1, so no population crosses a wall or the periodic
// y boundary and every shift mode is a compile-time constant.  x0 must be a
// valid node (callers clamp idle threads to x0 = 0 and discard their result).
template <typename T, int VEC, bool WALLS, bool INTERIOR, bool FORCH, bool CG = false>
__device__ __forceinline__ void gather(const T *__restrict__ src, const Geo &geo, int x0, int y,
                                       int lane, typename Store<T>::R inv_s,
                                       const typename Store<T>::R *__restrict__ alpha,
                                       const typename Store<T>::R *__restrict__ epsv,
                                       const typename Store<T>::R *__restrict__ betav, long long n0,
                                       typename Store<T>::R (&g)[VEC][9], typename Store<T>::R (&a)[VEC],
                                       typename Store<T>::R (&e)[VEC], typename Store<T>::R (&b)[VEC]) {
    using R = typename Store<T>::R;
    const int nx = geo.nx, ny = geo.ny;
    load_coef<R, VEC>(alpha + n0, a);
    load_coef<R, VEC>(epsv + n0, e);
    if (FORCH) load_coef<R, VEC>(betav + n0, b);
    else {
#pragma unroll
        for (int k = 0; k < VEC; ++k) b[k] = R(0);
    }
    if constexpr (VEC == 1) {
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            int ys = y - cy(i);
            const T *p;
            if (!INTERIOR && (ys < 0 || ys >= ny)) {
                if (WALLS) {
                    // halfway bounce-back: the opposite population that left
                    // this node towards the wall returns reversed
                    p = src + (long long)opp(i) * geo.plane + (long long)y * nx + x0;
                    g[0][i] = Store<T>::ld(ld1<CG>(p), inv_s);
                    continue;
                }
                ys = ys < 0 ? ys + ny : ys - ny;
            }
            int xs = x0 - cx(i);
            xs = xs < 0 ? xs + nx : (xs >= nx ? xs - nx : xs);
            p = src + (long long)i * geo.plane + (long long)ys * nx + xs;
            g[0][i] = Store<T>::ld(ld1<CG>(p), inv_s);
        }
    } else {
        // shift mode per population: 0 none, +1 take x-1, -1 take x+1;
        // bounce-back rows take the same node's opposite population unshifted
        T v[9][VEC];
        T edge[9];
        int mode[9];
        const bool first = lane == 0 || x0 == 0;
        const bool last = lane == 31 || x0 + VEC >= nx;
        const int xl = x0 == 0 ? nx - 1 : x0 - 1;
        const int xr = x0 + VEC >= nx ? 0 : x0 + VEC;
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            int ys = y - cy(i);
            int pl = i;
            mode[i] = cx(i);
            if (!INTERIOR && (ys < 0 || ys >= ny)) {
                if (WALLS) {
                    pl = opp(i);
                    ys = y;
                    mode[i] = 0;
                } else {
                    ys = ys < 0 ? ys + ny : ys - ny;
                }
            }
            const T *row = src + (long long)pl * geo.plane + (long long)ys * nx;
            ld16<T, VEC, CG>(row + x0, v[i]);
            edge[i] = T(0);
            if (mode[i] == 1 && first) edge[i] = ld1<CG>(row + xl);
            if (mode[i] == -1 && last) edge[i] = ld1<CG>(row + xr);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            R r[VEC];
#pragma unroll
            for (int k = 0; k < VEC; ++k) r[k] = Store<T>::ld(v[i][k], inv_s);
            if (mode[i] == 0) {
#pragma unroll
                for (int k = 0; k < VEC; ++k) g[k][i] = r[k];
            } else if (mode[i] == 1) {
                // node x takes x-1: shift right by one, left neighbour from lane-1
                R left = __shfl_up_sync(0xffffffffu, r[VEC - 1], 1);
                if (first) left = Store<T>::ld(edge[i], inv_s);
                g[0][i] = left;
#pragma unroll
                for (int k = 1; k < VEC; ++k) g[k][i] = r[k - 1];
            } else {
                // node x takes x+1: shift left by one, right neighbour from lane+1
                R right = __shfl_down_sync(0xffffffffu, r[0], 1);
                if (last) right = Store<T>::ld(edge[i], inv_s);
#pragma unroll
                for (int k = 0; k < VEC - 1; ++k) g[k][i] = r[k + 1];
                g[VEC - 1][i] = right;
            }
        }
    }
}


// Deterministic block sum of two doubles; thread 0 returns the totals.
__device__ __forceinline__ void block_sum2(double &a, double &b) {
    __shared__ double sh[2][32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        a += __shfl_down_sync(0xffffffffu, a, o);
        b += __shfl_down_sync(0xffffffffu, b, o);
    }
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) {
        sh[0][warp] = a;
        sh[1][warp] = b;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        a = 0.0;
        b = 0.0;
        for (int w = 0; w < int(blockDim.x >> 5); ++w) {
            a += sh[0][w];
            b += sh[1][w];
        }
    }
}

constexpr int kThreads = 128;

// Block maximum of a non-negative float; thread 0 returns it.
__device__ __forceinline__ float block_max(float m) {
    __shared__ float shm[32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_down_sync(0xffffffffu, m, o));
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (lane == 0) shm[warp] = m;
    __syncthreads();
    if (threadIdx.x == 0)
        for (int w = 1; w < int(blockDim.x >> 5); ++w) m = fmaxf(m, shm[w]);
    return m;
}

// One time step for the VEC consecutive nodes x0.. of row y of one lattice
// (src/dst/coefficients point at that lattice's plane 0).  Adds this thread's
// FP64 velocity sums to sx, sy and, for 16-bit storage, the largest stored
// magnitude to gm.
template <typename T, int VEC, bool WALLS, bool FORCH, bool REDUCE, bool CG = false>
__device__ __forceinline__ void step_body(const T *__restrict__ src, T *__restrict__ dst,
                                          const typename Store<T>::R *__restrict__ alpha,
                                          const typename Store<T>::R *__restrict__ epsv,
                                          const typename Store<T>::R *__restrict__ betav, const Geo &geo,
                                          const Phys<typename Store<T>::R> &ph, int x0, int y, double &sx,
                                          double &sy, float &gm) {
    using R = typename Store<T>::R;
    const bool active = x0 < geo.nx;
    x0 = active ? x0 : 0;  // idle threads read node 0 of the row and store nothing
    const int lane = threadIdx.x & 31;
    const long long n0 = (long long)y * geo.nx + x0;

    R g[VEC][9], a[VEC], e[VEC], b[VEC];
    if (y > 0 && y < geo.ny - 1)
        gather<T, VEC, WALLS, true, FORCH, CG>(src, geo, x0, y, lane, ph.inv_scale, alpha, epsv, betav, n0, g, a, e,
                                               b);
    else
        gather<T, VEC, WALLS, false, FORCH, CG>(src, geo, x0, y, lane, ph.inv_scale, alpha, epsv, betav, n0, g, a, e,
                                                b);

#pragma unroll
    for (int k = 0; k < VEC; ++k) {
        R ux, uy;
        if constexpr (Store<T>::kSmall) collide_small<R, FORCH>(g[k], a[k], e[k], b[k], ph, ux, uy);
        else collide<R, FORCH>(g[k], a[k], e[k], b[k], ph, ux, uy);
        if (REDUCE && active) {
            sx += double(ux);
            sy += double(uy);
        }
    }
    bool stored = false;
    if constexpr (Store<T>::kSmall && VEC == 4) {
        if (active && ph.sr) {
            // 16-bit storage, 4 nodes: two hardware stochastic-rounding
            // conversions per population.  The random words are successive
            // states of a full-period LCG seeded by one hash per thread; each
            // state is a bijective image of the seed, hence uniform like it,
            // which is all that unbiased rounding needs.
            uint32_t x = mix32(uint32_t(n0) ^ ph.step_key);
#pragma unroll
            for (int i = 0; i < 9; ++i) {
                float v[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) v[k] = Store<T>::kScaled ? g[k][i] * ph.scale : g[k][i];
                if (REDUCE)
                    gm = fmaxf(gm, fmaxf(fmaxf(fabsf(v[0]), fabsf(v[1])), fmaxf(fabsf(v[2]), fabsf(v[3]))));
                x = x * 0x2C1B3C6Du + 0x297A2D39u;
                const uint32_t r0 = x;
                x = x * 0x2C1B3C6Du + 0x297A2D39u;
                const uint32_t r1 = x;
                uint2 u;
                u.x = Store<T>::pack_sr(v[0], v[1], r0);
                u.y = Store<T>::pack_sr(v[2], v[3], r1);
                __stcs(reinterpret_cast<uint2 *>(dst + (long long)i * geo.plane + n0), u);
            }
            stored = true;
        }
    }
    if (active && !stored) {
        uint32_t hk[VEC];
        if constexpr (Store<T>::kSmall) {
#pragma unroll
            for (int k = 0; k < VEC; ++k) hk[k] = mix32(uint32_t(n0 + k) ^ ph.step_key);
        }
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            T v[VEC];
#pragma unroll
            for (int k = 0; k < VEC; ++k) {
                if constexpr (Store<T>::kSmall) {
                    if (ph.sr) {
                        // one multiply-xorshift per word on top of the node's full hash
                        uint32_t r = (hk[k] ^ (uint32_t(i >> 1) * 0x9E3779B9u)) * 0x2C1B3C6Du;
                        r ^= r >> 15;
                        v[k] = Store<T>::st_sr(g[k][i], ph.scale, (i & 1) ? (r >> 16) : r);
                    } else {
                        v[k] = Store<T>::st(g[k][i], ph.scale);
                    }
                    if (REDUCE) gm = fmaxf(gm, fabsf(float(v[k])));
                } else {
                    v[k] = Store<T>::st(g[k][i], ph.scale);
                }
            }
            T *p = dst + (long long)i * geo.plane + n0;
            if constexpr (VEC == 1) p[0] = v[0];
            else st16<T, VEC>(p, v);
        }
    }
}

// ---------------------------------------------------------------------------
// K2: fused pull-stream + collide (one time step).  REDUCE additionally
// writes this block's FP64 sums of u_x, u_y to partial[2*block] and, for
// 16-bit storage, the largest stored magnitude |g*S| to pmax[block].
// ---------------------------------------------------------------------------
// Programmatic dependent launch.  A step kernel launched with programmatic
// stream serialisation may be scheduled while the previous kernel of the
// stream drains.  It waits here, before touching any global memory (reads of
// the previous step's output and writes into the buffer that step read), for
// that kernel to complete and flush; then it lets the next launch start
// placing its blocks, so launch latency and the last partial wave overlap.
// Without the launch attribute both instructions return at once.
__device__ __forceinline__ void pdl_enter() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Host: launch `kern` on `st`, with programmatic stream serialisation when
// `pdl` (callers pass it for non-default streams).
template <typename... P, typename... A>
inline cudaError_t launch_kernel_smem(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st,
                                      bool pdl, A &&...args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = block;
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = pdl ? at : nullptr;
    cfg.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}
template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kern)(P...), dim3 grid, dim3 block, cudaStream_t st, bool pdl,
                                 A &&...args) {
    return launch_kernel_smem(kern, grid, block, 0, st, pdl, std::forward<A>(args)...);
}

// Grid: x = blocks of a row (geo.bpr), row y = blockIdx.y + kMaxGridY *
// blockIdx.z (step_grid).  Blocks of 128 threads resident per SM, fixed by
// measurement on GB300: FP32 and FP16 fit 64 registers (8 blocks, 32 warps);
// BF16 spills at 64 and runs faster at 72 (7 blocks); FP64 is left free.
constexpr int kMaxGridY = 65535;
inline dim3 step_grid(const Geo &g) {
    const int gy = g.ny < kMaxGridY ? g.ny : kMaxGridY;
    return dim3(unsigned(g.bpr), unsigned(gy), unsigned((g.ny + kMaxGridY - 1) / kMaxGridY));
}
template <typename T>
constexpr int kMinBlocks = sizeof(T) == 8 ? 1 : (std::is_same<T, __nv_bfloat16>::value ? 7 : 8);

template <typename T, int VEC, bool WALLS, bool FORCH, bool REDUCE>
__global__ void __launch_bounds__(kThreads, kMinBlocks<T>)
k_step(const T *__restrict__ src, T *__restrict__ dst, const typename Store<T>::R *__restrict__ alpha,
       const typename Store<T>::R *__restrict__ epsv, const typename Store<T>::R *__restrict__ betav,
       Geo geo, Phys<typename Store<T>::R> ph, double *__restrict__ partial, float *__restrict__ pmax) {
    pdl_enter();
    if constexpr (Store<T>::kSmall) {
        if (ph.clock) ph.step_key = step_key_of(*ph.clock + ph.step_off, ph.seed);
    }
    const int y = int(blockIdx.y) + kMaxGridY * int(blockIdx.z);
    if (y >= geo.ny) return;  // padding of the last z slice (whole block)
    const int bx = int(blockIdx.x);
    const int x0 = (bx * kThreads + threadIdx.x) * VEC;
    const long long blk = (long long)y * geo.bpr + bx;  // reduction slot, row-major
    double sx = 0.0, sy = 0.0;
    float gm = 0.0f;
    step_body<T, VEC, WALLS, FORCH, REDUCE>(src, dst, alpha, epsv, betav, geo, ph, x0, y, sx, sy, gm);
    if (REDUCE) {
        block_sum2(sx, sy);
        if (threadIdx.x == 0) {
            partial[2 * blk] = sx;
            partial[2 * blk + 1] = sy;
        }
        if constexpr (Store<T>::kSmall) {
            gm = block_max(gm);
            if (threadIdx.x == 0) pmax[blk] = gm;
        }
    }
}

// ---------------------------------------------------------------------------
// K2b: two time steps in one pass over memory.
//
// The one-step kernel is bound by HBM on large lattices (FP32: 80 B per node
// and step at 1.03 of the copy bandwidth) while its arithmetic needs less than
// half of that time, so two steps share one read and one write.  Each warp
// marches up a strip of 128 columns (4 per lane), one row per iteration: it
// gathers row r and collides it (first step), then streams and collides row
// r - 1 (second step) from the first-step populations of rows r - 2, r - 1
// and r.  Level ones stay in registers for a row, upward ones in shared memory
// for two, downward ones are used at once.  x neighbours come by warp shuffle
// as in gather(); the outermost lane on each side has none beyond it, so it
// only is the halo of the next one and a strip stores 30 of its 32 lanes'
// columns (6 %).  Rows y0 - 1 and y1 of a segment [y0, y1) are recomputed by
// its neighbours' warps (2/rows).  One warp per block and no barriers.
//
// The arithmetic runs on packed pairs because issue would be the next bound
// (scalar: 147 instructions per node and step, packed: 107).  Registers
// are what is scarce: with the upward rows and the next row's loads in
// registers, or at 5 warps per scheduler, the loop spills and loses 20 %.
// FP32 runs best at 12 warps per SM (fewer DRAM streams), 16-bit at 16;
// cp.async.cg, a barrier per row and 128-thread blocks were slower.
// 4096^2, us a step: FP32 191 -> 108 (Forchheimer 201 -> 116), BF16 110 -> 87;
// 2048^2: FP32 49.5 -> 28.0, FP16 30.0 -> 25.2.  FP32 then moves 0.9 of the copy
// bandwidth; 16-bit storage is bound by latency at 4 warps per scheduler (issue
// active 60 % of the time, 0.64 of the copy bandwidth).
//
// Both steps round, and draw their stochastic-rounding words, exactly as the
// one-step kernel does, so the results are its bits.
// ---------------------------------------------------------------------------
constexpr int kPairThreads = 32;
template <typename T>
constexpr int kPairWarps = sizeof(T) == 2 ? 16 : 12;  // resident warps per SM
// Fewest nodes for which k_pair is considered: below, the lattice stays in L2, there
// is less than a warp's worth of rows per segment and the one-step kernel is
// faster (1024^2: FP32 8.4 against 8.9 us a step, BF16 6.9 against 8.4; 1280^2:
// 16.4 against 11.6 and 11.5 against 10.9).
constexpr long long kPairNodes = 5ll << 18;
constexpr int kStripLanes = 30;              // lanes of a strip that store
constexpr int kStripCols = 4 * kStripLanes;  // columns of a strip

template <typename F, size_t... I>
__device__ __forceinline__ void for_pops_(F f, std::index_sequence<I...>) {
    (f(std::integral_constant<int, int(I)>{}), ...);
}
template <typename F>
__device__ __forceinline__ void for_pops(F f) {
    for_pops_(f, std::make_index_sequence<9>{});
}

// Four nodes of a lane as two packed pairs.
struct Quad {
    f2 p[2];
};

// The LCG's state after n steps is a_n x + c_n: taken directly from the seed
// the 18 words of a lane do not wait for one another.
struct LcgStep {
    uint32_t a, c;
};
__host__ __device__ constexpr LcgStep lcg_step(int n) {
    LcgStep s{1u, 0u};
    for (int i = 0; i < n; ++i) s = LcgStep{s.a * 0x2C1B3C6Du, s.c * 0x2C1B3C6Du + 0x297A2D39u};
    return s;
}

// Stored form of 4 nodes' population I of 16-bit storage, stochastically
// rounded with states 2I+1 and 2I+2 of the LCG as in step_body (the FP16 scale
// is in the values).
template <typename T, int I>
__device__ __forceinline__ uint2 round4(Quad q, uint32_t seed) {
    constexpr LcgStep s0 = lcg_step(2 * I + 1), s1 = lcg_step(2 * I + 2);
    return make_uint2(Store<T>::pack_sr(lo2(q.p[0]), hi2(q.p[0]), seed * s0.a + s0.c),
                      Store<T>::pack_sr(lo2(q.p[1]), hi2(q.p[1]), seed * s1.a + s1.c));
}
// Loaded 4 nodes of storage T as pairs (FP16: with their scale).
template <typename T>
__device__ __forceinline__ Quad unpack4(const T (&t)[4]) {
    return Quad{{mk2(Store<T>::ld(t[0], 1.0f), Store<T>::ld(t[1], 1.0f)), mk2(Store<T>::ld(t[2], 1.0f), Store<T>::ld(t[3], 1.0f))}};
}

// x shifts within a strip: RIGHT: node x takes x - 1; else node x takes x + 1.
template <bool RIGHT>
__device__ __forceinline__ Quad shift4(const Quad &r) {
    Quad o;
    if (RIGHT) {
        const float n = __shfl_up_sync(0xffffffffu, hi2(r.p[1]), 1);
        o.p[0] = mk2(n, lo2(r.p[0]));
        o.p[1] = mk2(hi2(r.p[0]), lo2(r.p[1]));
    } else {
        const float n = __shfl_down_sync(0xffffffffu, lo2(r.p[0]), 1);
        o.p[0] = mk2(hi2(r.p[0]), lo2(r.p[1]));
        o.p[1] = mk2(hi2(r.p[1]), n);
    }
    return o;
}

template <typename T, bool FORCH>
__device__ __forceinline__ void collide4(Quad (&g)[9], const Quad &a, const Quad &e, const Quad &b, const Pair2 &c) {
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        f2 n[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) n[i] = g[i].p[k];
        if constexpr (Store<T>::kSmall) collide_small2<FORCH, Store<T>::kScaled>(n, a.p[k], e.p[k], b.p[k], c);
        else collide2<FORCH>(n, a.p[k], e.p[k], b.p[k], c);
#pragma unroll
        for (int i = 0; i < 9; ++i) g[i].p[k] = n[i];
    }
}

// Shared memory of one warp.  Every lane reads back only what it wrote or
// copied itself, so no barrier is needed.
//  f, coef  row r + 1 travels here by cp.async while row r is computed; the
//           coefficients stay for the second step of row r, a row later
//  up       first-step upward populations of the last two rows
template <typename T, bool FORCH>
struct StripSmem {
    struct Vec {
        T v[4];
    };
    float4 coef[3][FORCH ? 3 : 2][32];
    float4 up[2][3][32];
    alignas(16) Vec f[9][32];
};
template <int B>
__device__ __forceinline__ void cp_async(void *smem, const void *gmem) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(unsigned(__cvta_generic_to_shared(smem))),
                 "l"(gmem), "n"(B)
                 : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Rows [y0, y1) of the strip whose stored columns begin at xs, two steps.
// nx must be a multiple of 4; ph.step_key / step_key2 key the two steps;
// `sm` is this warp's own.
template <typename T, bool WALLS, bool FORCH>
__device__ __forceinline__ void march_strip(StripSmem<T, FORCH> &sm, const T *__restrict__ src, T *__restrict__ dst,
                                            const float *__restrict__ alpha, const float *__restrict__ epsv,
                                            const float *__restrict__ betav, const Geo &geo, const Phys<float> &ph,
                                            const Pair2 &c, int xs, int y0, int y1) {
    const int nx = geo.nx, ny = geo.ny;
    const int lane = threadIdx.x & 31;
    const int groups = nx >> 2;
    int grp = (xs >> 2) + lane - 1;  // this lane's column group, wrapped around the period
    grp = grp < 0 ? grp + groups : grp;
    grp = grp >= groups ? grp % groups : grp;
    const int x0 = grp << 2;
    const bool store = lane >= 1 && lane <= kStripLanes && xs + 4 * (lane - 1) < nx;
    const bool at_lo = WALLS && y0 == 0, at_hi = WALLS && y1 == ny;

    const Quad zero{{f2{0}, f2{0}}};
    Quad c0 = zero, c1 = zero, c3 = zero;  // first-step rest and level populations of row r - 1 (x-shifted)
    int slot = 0;                          // coefficient slot of row r
    auto row_of = [&](int r) { return WALLS ? r : (r < 0 ? r + ny : (r >= ny ? r - ny : r)); };
    // start the copies of row r: population i comes from row r - e_y, at a wall
    // from its opposite in row r (halfway bounce-back)
    auto fetch = [&](int r, int cs) {
        const int rr = row_of(r);
        const bool lo = WALLS && rr == 0, hi = WALLS && rr == ny - 1;
        const long long row = (long long)rr * nx + x0;
        const long long rm = !WALLS && rr == 0 ? (long long)(ny - 1) * nx + x0 : row - nx;
        const long long rp = !WALLS && rr == ny - 1 ? x0 : row + nx;
        cp_async<16>(&sm.coef[cs][0][lane], alpha + row);
        cp_async<16>(&sm.coef[cs][1][lane], epsv + row);
        if (FORCH) cp_async<16>(&sm.coef[cs][FORCH ? 2 : 0][lane], betav + row);
        constexpr int B = 4 * sizeof(T);
        const long long pl = geo.plane;
        cp_async<B>(&sm.f[0][lane], src + row);
        cp_async<B>(&sm.f[1][lane], src + pl + row);
        cp_async<B>(&sm.f[3][lane], src + 3 * pl + row);
        cp_async<B>(&sm.f[2][lane], src + (lo ? 4 * pl + row : 2 * pl + rm));
        cp_async<B>(&sm.f[5][lane], src + (lo ? 7 * pl + row : 5 * pl + rm));
        cp_async<B>(&sm.f[6][lane], src + (lo ? 8 * pl + row : 6 * pl + rm));
        cp_async<B>(&sm.f[4][lane], src + (hi ? 2 * pl + row : 4 * pl + rp));
        cp_async<B>(&sm.f[7][lane], src + (hi ? 5 * pl + row : 7 * pl + rp));
        cp_async<B>(&sm.f[8][lane], src + (hi ? 6 * pl + row : 8 * pl + rp));
    };
    // row ny of a walled lattice is the upper wall's mirror, made from row ny - 1
    const int r_first = at_lo ? 0 : y0 - 1, r_last = at_hi ? ny - 1 : y1;
    fetch(r_first, 0);
    cp_async_commit();
    for (int r = r_first; r <= y1; ++r) {
        const int next = slot == 2 ? 0 : slot + 1, prev = slot == 0 ? 2 : slot - 1;
        Quad h0, h2, h4, s1, s3, s5, s6, s7, s8;
        if (at_hi && r == ny) {
            // halfway bounce-back: what left row ny - 1 upwards returns reversed
            // to its own node (undo the x shift of 5 and 6)
            Quad u5, u6;
            memcpy(&h4, &sm.up[(r - 1) & 1][0][lane], 16);
            memcpy(&u5, &sm.up[(r - 1) & 1][1][lane], 16);
            memcpy(&u6, &sm.up[(r - 1) & 1][2][lane], 16);
            s7 = shift4<false>(u5);
            s8 = shift4<true>(u6);
            h0 = s1 = s3 = h2 = s5 = s6 = zero;
        } else {
            const int rr = row_of(r);
            const bool lo = WALLS && rr == 0, hi = WALLS && rr == ny - 1;
            Quad h[9], a, e, b = zero;
            cp_async_wait<0>();
            memcpy(&a, &sm.coef[slot][0][lane], 16);
            memcpy(&e, &sm.coef[slot][1][lane], 16);
            if (FORCH) memcpy(&b, &sm.coef[slot][FORCH ? 2 : 0][lane], 16);
            Quad f[9];
#pragma unroll
            for (int i = 0; i < 9; ++i) f[i] = unpack4<T>(sm.f[i][lane].v);
            h[0] = f[0], h[2] = f[2], h[4] = f[4];
            h[1] = shift4<true>(f[1]);
            h[3] = shift4<false>(f[3]);
            h[5] = lo ? f[5] : shift4<true>(f[5]);
            h[6] = lo ? f[6] : shift4<false>(f[6]);
            h[7] = hi ? f[7] : shift4<false>(f[7]);
            h[8] = hi ? f[8] : shift4<true>(f[8]);
            if (r + 1 <= r_last) fetch(r + 1, next);  // row r is in registers by now
            cp_async_commit();
            collide4<T, FORCH>(h, a, e, b, c);
            if constexpr (Store<T>::kSmall) {
                const uint32_t seed = mix32(uint32_t((long long)rr * nx + x0) ^ ph.step_key);
                for_pops([&](auto i) {
                    const uint2 w = round4<T, i.value>(h[i.value], seed);
                    T t[4];
                    memcpy(t, &w, 8);
                    h[i.value] = unpack4<T>(t);
                });
            }
            h0 = h[0], h2 = h[2], h4 = h[4];
            s1 = shift4<true>(h[1]);
            s3 = shift4<false>(h[3]);
            s5 = shift4<true>(h[5]);
            s6 = shift4<false>(h[6]);
            s7 = shift4<false>(h[7]);
            s8 = shift4<true>(h[8]);
            if (lo) {  // the lower wall returns row 0's own downward populations
                memcpy(&sm.up[1][0][lane], &h[4], 16);
                memcpy(&sm.up[1][1][lane], &h[7], 16);
                memcpy(&sm.up[1][2][lane], &h[8], 16);
            }
        }
        Quad g[9] = {c0, c1, zero, c3, h4, zero, zero, s7, s8};
        if (r > y0) {
            Quad a, e, b = zero;
            memcpy(&g[2], &sm.up[r & 1][0][lane], 16);
            memcpy(&g[5], &sm.up[r & 1][1][lane], 16);
            memcpy(&g[6], &sm.up[r & 1][2][lane], 16);
            memcpy(&a, &sm.coef[prev][0][lane], 16);
            memcpy(&e, &sm.coef[prev][1][lane], 16);
            if (FORCH) memcpy(&b, &sm.coef[prev][FORCH ? 2 : 0][lane], 16);
            collide4<T, FORCH>(g, a, e, b, c);
            const long long n0 = (long long)(r - 1) * nx + x0;
            uint32_t seed = 0;
            if constexpr (Store<T>::kSmall) seed = mix32(uint32_t(n0) ^ ph.step_key2);
            for_pops([&](auto i) {
                T *p = dst + (long long)i.value * geo.plane + n0;
                if constexpr (Store<T>::kSmall) {
                    const uint2 w = round4<T, i.value>(g[i.value], seed);
                    if (store) __stcs(reinterpret_cast<uint2 *>(p), w);
                } else {
                    uint4 w;
                    memcpy(&w, &g[i.value], 16);
                    if (store) __stcs(reinterpret_cast<uint4 *>(p), w);
                }
            });
        }
        memcpy(&sm.up[r & 1][0][lane], &h2, 16);
        memcpy(&sm.up[r & 1][1][lane], &s5, 16);
        memcpy(&sm.up[r & 1][2][lane], &s6, 16);
        c0 = h0, c1 = s1, c3 = s3;
        slot = next;
    }
}

// One lattice: block w takes strip w % strips of segment w / strips
// (neighbouring strips run side by side, so their shared columns hit L1 or L2).
template <typename T, bool WALLS, bool FORCH>
__global__ void __launch_bounds__(kPairThreads, kPairWarps<T>)
k_pair(const T *__restrict__ src, T *__restrict__ dst, const float *__restrict__ alpha,
       const float *__restrict__ epsv, const float *__restrict__ betav, Geo geo, Phys<float> ph,
       const __grid_constant__ Pair2 c, int strips, int rows) {
    extern __shared__ __align__(16) unsigned char strip_smem[];
    pdl_enter();
    if constexpr (Store<T>::kSmall) {
        if (ph.clock) {
            const uint32_t t = *ph.clock + ph.step_off;
            ph.step_key = step_key_of(t, ph.seed);
            ph.step_key2 = step_key_of(t + 1, ph.seed);
        }
    }
    const int seg = blockIdx.x / strips;
    const int y0 = seg * rows;
    const int y1 = y0 + rows < geo.ny ? y0 + rows : geo.ny;
    march_strip<T, WALLS, FORCH>(*reinterpret_cast<StripSmem<T, FORCH> *>(strip_smem), src, dst, alpha, epsv, betav,
                                 geo, ph, c, (blockIdx.x - seg * strips) * kStripCols, y0, y1);
}

// ---------------------------------------------------------------------------
// K2c: several time steps of a tile per launch, for lattices that one wave of
// blocks covers and for row lengths that are not a multiple of the vector.
//
// Small lattices are bound by the latency of a launch (a 128^2 step is 0.2 us
// of arithmetic in a 2 us launch), odd row lengths by scalar loads.  A block
// loads a tile with a halo, advances it `nsteps` steps and stores the inside.
// A thread keeps 4 nodes of a row: rest and level populations stay in its
// registers (x neighbours by shuffle among the Q lanes of the row), the six
// that move in y go through shared memory, two buffers, one barrier per step.
// The first step gathers from memory itself, so rows need a halo of
// nsteps - 1; columns lose one per step, rounded up to 4.  Values beyond the
// halo's reach are computed from stale neighbours and never stored.  Wall
// rows write what the wall returns into the shared row beyond it.
// Columns of an odd-length row are fetched one by one, each wrapped around
// the period; everything after that is the same.
// Rounding and stochastic-rounding words are the one-step kernel's (per lane
// of 4 for whole vectors, per node otherwise), so the results are its bits.
// ---------------------------------------------------------------------------
constexpr int kTileThreads = 640;  // most per block: 96 registers a thread
constexpr int kTileQ = 16;         // most lanes of a row
// Shared memory of a tile of `rows` rows (with halo) and q lanes: two buffers of
// six populations, with a row beyond each edge; and the most of any plan.
constexpr size_t tile_bytes(int rows, int q) { return sizeof(float4) * 2 * 6 * size_t(rows + 2) * size_t(q); }
constexpr size_t kTileSmem = tile_bytes(kTileThreads / kTileQ, kTileQ);
static_assert(tile_bytes(kTileThreads / 8, 8) <= kTileSmem, "narrow tiles");

struct TilePlan {
    int steps;     // T: most steps per launch; 0: not used
    int q_log2;    // lanes per row, Q = 1 << q_log2
    int rows;      // rows per block with halo
    int hx, hy;    // halo
    int nx_tiles, ny_tiles;
};

// Stored 16-bit form of one node as the one-step kernel with one node per
// thread rounds it.
template <typename T, int I>
__device__ __forceinline__ T round1(float v, uint32_t hash) {
    uint32_t r = (hash ^ (uint32_t(I >> 1) * 0x9E3779B9u)) * 0x2C1B3C6Du;
    r ^= r >> 15;
    return Store<T>::st_sr(v, 1.0f, (I & 1) ? (r >> 16) : r);
}

template <typename T, bool WALLS, bool FORCH, bool ODD>
__global__ void __launch_bounds__(kTileThreads, 1)
k_tile(const T *__restrict__ src, T *__restrict__ dst, const float *__restrict__ alpha,
       const float *__restrict__ epsv, const float *__restrict__ betav, Geo geo, Phys<float> ph,
       const __grid_constant__ Pair2 c, TilePlan pl, int nsteps) {
    extern __shared__ __align__(16) float4 tile_smem[];
    const int Q = 1 << pl.q_log2, R = pl.rows;
    const int qx = threadIdx.x & (Q - 1), ly = threadIdx.x >> pl.q_log2;
    const int ty = blockIdx.x / pl.nx_tiles, tx = blockIdx.x - ty * pl.nx_tiles;
    const int nx = geo.nx, ny = geo.ny;
    const int gx = tx * (4 * Q - 2 * pl.hx) - pl.hx + 4 * qx;  // unwrapped
    const int gy = ty * (R - 2 * pl.hy) - pl.hy + ly;
    const bool inside = !WALLS || (gy >= 0 && gy < ny);
    int row = gy;  // wrapped; rows outside a walled lattice compute row 0 to no effect
    if (WALLS) row = inside ? gy : 0;
    else {
        row %= ny;
        row = row < 0 ? row + ny : row;
    }
    int col[ODD ? 4 : 1];  // this lane's columns, wrapped (whole vectors: the first)
#pragma unroll
    for (int k = 0; k < (ODD ? 4 : 1); ++k) {
        const int x = (gx + k) % nx;
        col[k] = x < 0 ? x + nx : x;
    }
    const bool lo = WALLS && inside && row == 0, hi = WALLS && inside && row == ny - 1;
    const bool out = inside && ly >= pl.hy && ly < R - pl.hy && gy < ny && 4 * qx >= pl.hx &&
                     4 * qx < 4 * Q - pl.hx && gx < nx;
    // rows of this warp (first and last), to skip those that do not matter
    const int wy0 = int(threadIdx.x & ~31u) >> pl.q_log2, wy1 = int(threadIdx.x | 31u) >> pl.q_log2;
    const bool beyond = WALLS && (gy - ly + wy1 < 0 || gy - ly + wy0 >= ny);

    const long long base = (long long)row * nx;
    auto coef = [&](const float *p) {
        Quad q;
        if constexpr (ODD) {
            q.p[0] = mk2(p[base + col[0]], p[base + col[1]]);
            q.p[1] = mk2(p[base + col[2]], p[base + col[3]]);
        } else {
            const uint4 w = *reinterpret_cast<const uint4 *>(p + base + col[0]);
            memcpy(&q, &w, 16);
        }
        return q;
    };
    const Quad zero{{f2{0}, f2{0}}};
    // no step kernel writes the coefficients: they load while the one before drains
    const Quad a = coef(alpha), e = coef(epsv), b = FORCH ? coef(betav) : zero;
    pdl_enter();
    uint32_t t0 = ph.tstep;
    if constexpr (Store<T>::kSmall) {
        if (ph.clock) t0 = *ph.clock + ph.step_off;
    }
    auto right = [&](const Quad &r) {  // node x takes x - 1 within the row's lanes
        const float n = __shfl_up_sync(0xffffffffu, hi2(r.p[1]), 1, Q);
        return Quad{{mk2(n, lo2(r.p[0])), mk2(hi2(r.p[0]), lo2(r.p[1]))}};
    };
    auto left = [&](const Quad &r) {
        const float n = __shfl_down_sync(0xffffffffu, lo2(r.p[0]), 1, Q);
        return Quad{{mk2(hi2(r.p[0]), lo2(r.p[1])), mk2(hi2(r.p[1]), n)}};
    };

    Quad g[9];
    {
        const int rm = row == 0 ? ny - 1 : row - 1, rp = row == ny - 1 ? 0 : row + 1;
        // at a wall the opposite population that left the node returns to it
        const int rlo = lo ? row : rm, rhi = hi ? row : rp;
        const int plane[9] = {0, 1, lo ? 4 : 2, 3, hi ? 2 : 4, lo ? 7 : 5, lo ? 8 : 6, hi ? 5 : 7, hi ? 6 : 8};
        const int from[9] = {row, row, rlo, row, rhi, rlo, rlo, rhi, rhi};
        Quad f[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const T *p = src + (long long)plane[i] * geo.plane + (long long)from[i] * nx;
            T t[4];
            if constexpr (ODD) {
#pragma unroll
                for (int k = 0; k < 4; ++k) t[k] = p[col[ODD ? k : 0]];
            } else {
                ld16<T, 4>(p + col[0], t);
            }
            f[i] = unpack4<T>(t);
        }
        g[0] = f[0], g[2] = f[2], g[4] = f[4];
        g[1] = right(f[1]), g[3] = left(f[3]);
        const Quad s5 = right(f[5]), s6 = left(f[6]), s7 = left(f[7]), s8 = right(f[8]);
        auto pick = [](bool first, const Quad &p, const Quad &q) {
            return Quad{{f2{first ? p.p[0].v : q.p[0].v}, f2{first ? p.p[1].v : q.p[1].v}}};
        };
        g[5] = pick(lo, f[5], s5), g[6] = pick(lo, f[6], s6);
        g[7] = pick(hi, f[7], s7), g[8] = pick(hi, f[8], s8);
    }
    for (int s = 0; s < nsteps; ++s) {
        const int reach = nsteps - 1 - s;  // rows beyond the inside that still matter
        const bool work = !beyond && wy1 >= pl.hy - reach && wy0 < R - pl.hy + reach;
        if (work) {
            collide4<T, FORCH>(g, a, e, b, c);
            T stored[9][4];
            if constexpr (Store<T>::kSmall) {
                const uint32_t key = step_key_of(t0 + uint32_t(s), ph.seed);
                if constexpr (ODD) {
                    uint32_t hash[4];
#pragma unroll
                    for (int k = 0; k < 4; ++k) hash[k] = mix32(uint32_t(base + col[ODD ? k : 0]) ^ key);
                    for_pops([&](auto i) {
                        const Quad &q = g[i.value];
                        const float v[4] = {lo2(q.p[0]), hi2(q.p[0]), lo2(q.p[1]), hi2(q.p[1])};
#pragma unroll
                        for (int k = 0; k < 4; ++k) stored[i.value][k] = round1<T, i.value>(v[k], hash[k]);
                    });
                } else {
                    const uint32_t seed = mix32(uint32_t(base + col[0]) ^ key);
                    for_pops([&](auto i) {
                        const uint2 w = round4<T, i.value>(g[i.value], seed);
                        memcpy(stored[i.value], &w, 8);
                    });
                }
            } else {
                memcpy(stored, g, sizeof(stored));
            }
            if (reach == 0) {
                if (out) {
#pragma unroll
                    for (int i = 0; i < 9; ++i) {
                        T *p = dst + (long long)i * geo.plane + base + gx;
                        if constexpr (ODD) {
#pragma unroll
                            for (int k = 0; k < 4; ++k)
                                if (gx + k < nx) p[k] = stored[i][k];
                        } else {
                            st16<T, 4>(p, stored[i]);
                        }
                    }
                }
                break;
            }
            if constexpr (Store<T>::kSmall) {
#pragma unroll
                for (int i = 0; i < 9; ++i) g[i] = unpack4<T>(stored[i]);
            }
            // slots: population set {2, 5, 6 | 4, 7, 8}, row + 1, lane
            float4 *buf = tile_smem + (s & 1) * 6 * (R + 2) * Q + qx;
            auto slot = [&](int set, int r) { return buf + (set * (R + 2) + r + 1) * Q; };
            if (inside) {
                if (lo) {
                    memcpy(slot(0, ly - 1), &g[4], 16);
                    memcpy(slot(1, ly - 1), &g[7], 16);
                    memcpy(slot(2, ly - 1), &g[8], 16);
                }
                if (hi) {
                    memcpy(slot(3, ly + 1), &g[2], 16);
                    memcpy(slot(4, ly + 1), &g[5], 16);
                    memcpy(slot(5, ly + 1), &g[6], 16);
                }
            }
            g[1] = right(g[1]), g[3] = left(g[3]);
            g[5] = right(g[5]), g[6] = left(g[6]), g[7] = left(g[7]), g[8] = right(g[8]);
            if (inside) {
                memcpy(slot(0, ly), &g[2], 16);
                memcpy(slot(1, ly), &g[5], 16);
                memcpy(slot(2, ly), &g[6], 16);
                memcpy(slot(3, ly), &g[4], 16);
                memcpy(slot(4, ly), &g[7], 16);
                memcpy(slot(5, ly), &g[8], 16);
            }
        } else if (reach == 0) {
            break;
        }
        __syncthreads();
        const float4 *buf = tile_smem + (s & 1) * 6 * (R + 2) * Q + qx;
        auto slot = [&](int set, int r) { return buf + (set * (R + 2) + r + 1) * Q; };
        memcpy(&g[2], slot(0, ly - 1), 16);
        memcpy(&g[5], slot(1, ly - 1), 16);
        memcpy(&g[6], slot(2, ly - 1), 16);
        memcpy(&g[4], slot(3, ly + 1), 16);
        memcpy(&g[7], slot(4, ly + 1), 16);
        memcpy(&g[8], slot(5, ly + 1), 16);
    }
}

// Device step counter of 16-bit storage (see Phys::clock): set to a value
// or advanced by a captured chunk's length, one thread, ordered on the
// stream after the chunk's last step kernel.
__global__ void k_clock(unsigned *__restrict__ clock, unsigned value, int add) {
    pdl_enter();
    *clock = add ? *clock + value : value;
}

// Device-side run status (A8 result and convergence test).
struct DevStatus {
    double ux, uy;     // mean velocity of the last reduced step
    double prev_ux;    // the previous check's mean u_x
    int have_prev;     // prev_ux valid
    int converged;     // set by the last finalize
    int nonfinite;     // mean velocity not finite
    float gmax;        // 16-bit storage: largest stored |g*S| at that step
    int streak;        // consecutive checks that passed the relative-change test
    int pad;
};

// K3 finalize: fixed-order FP64 sum of the block partials, mean, test.
// Converged once `patience` consecutive checks pass |Ux - Ux_prev| <=
// tol |Ux| (patience 1: the first pass).
__global__ void __launch_bounds__(256)
k_finalize(const double *__restrict__ partial, int nparts, double inv_n, double tol,
           DevStatus *__restrict__ st, const float *__restrict__ pmax, int patience = 1) {
    __shared__ double sh[2][256];
    double a = 0.0, b = 0.0;
    float m = 0.0f;
    for (int j = threadIdx.x; j < nparts; j += 256) {
        a += partial[2ll * j];
        b += partial[2ll * j + 1];
        if (pmax) m = fmaxf(m, pmax[j]);
    }
    sh[0][threadIdx.x] = a;
    sh[1][threadIdx.x] = b;
    if (pmax) m = block_max(m);
    __syncthreads();
    for (int s = 128; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            sh[0][threadIdx.x] += sh[0][threadIdx.x + s];
            sh[1][threadIdx.x] += sh[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        const double ux = sh[0][0] * inv_n, uy = sh[1][0] * inv_n;
        st->ux = ux;
        st->uy = uy;
        const bool fin = isfinite(ux) && isfinite(uy);
        st->nonfinite = fin ? 0 : 1;
        const bool pass = fin && tol > 0.0 && st->have_prev && fabs(ux - st->prev_ux) <= tol * fabs(ux);
        st->streak = pass ? st->streak + 1 : 0;
        st->converged = st->streak >= patience ? 1 : 0;
        st->prev_ux = ux;
        st->have_prev = 1;
        st->gmax = m;
    }
}

// Velocity export: re-run the step's gather and velocity solve on the
// pre-step state (scalar loads; same arithmetic as k_step).
template <typename T, bool WALLS, bool FORCH>
__global__ void __launch_bounds__(kThreads)
k_velocity(const T *__restrict__ src, const typename Store<T>::R *__restrict__ alpha,
           const typename Store<T>::R *__restrict__ epsv, const typename Store<T>::R *__restrict__ betav,
           Geo geo, Phys<typename Store<T>::R> ph, double *__restrict__ ux_out,
           double *__restrict__ uy_out, double *__restrict__ rho_out = nullptr) {
    using R = typename Store<T>::R;
    const int y = blockIdx.x / geo.bpr;
    const int bx = blockIdx.x - y * geo.bpr;
    const int x0 = bx * kThreads + threadIdx.x;
    const bool active = x0 < geo.nx;
    if (!active) return;  // no shuffles on the scalar path
    const long long n = (long long)y * geo.nx + x0;
    R g[1][9], a[1], e[1], b[1];
    gather<T, 1, WALLS, false, FORCH>(src, geo, x0, y, threadIdx.x & 31, ph.inv_scale, alpha, epsv, betav, n, g, a, e,
                                      b);
    R drho, ux, uy;
    node_velocity<R, FORCH>(g[0], a[0], e[0], b[0], ph, drho, ux, uy);
    ux_out[n] = double(ux);
    uy_out[n] = double(uy);
    if (rho_out) rho_out[n] = 1.0 + double(drho);
}

}  // namespace
