// Constants of the odd (momentum) half of the FP32/FP64 collision.
//
// Opposite populations differ by w_i rho (3 e.u/tau + 3 A e.F), A = 1 - 1/(2 tau),
// and keep k1 = 1 - 1/tau of what they had.  Summed over the directions a step
// leaves the momentum k1 m + u/tau + A F, which is m + F exactly; if 1/9, 3/tau
// and 3A are each rounded, the sum is off by a fixed fraction of u and of F (up
// to 6e-8 each), at every node and in every step, and the slow modes collect it:
// on a two-phase medium it is the largest error of an FP32 run.  The weight may
// carry any factor that the other two give back, so it is chosen such that both
// quotients are within 2^-31 or so of numbers of the type.
#pragma once

#include <cmath>
#include <type_traits>

namespace {

// odd part: c rho e.(a u + b F) for the axis directions, a quarter of it for
// the diagonal ones, with 3 c a = 1 - k1 and 3 c b = 1 - (1 - k1)/2.
template <typename R>
struct OddConstants {
    R c, a, b;
};

// Candidates c = 1/8 + i 2^-20 are short, so that 3c is exact and fma gives the
// residuals of the rounded quotients.  The first whose residuals sum to 2^-31
// (FP64: 2^-60), else the best of 1024: 3 us, once per handle.
template <typename R>
OddConstants<R> odd_constants(R omega) {
    constexpr double enough = std::is_same<R, float>::value ? 0x1p-31 : 0x1p-60;
    const R k1 = R(1) - omega, om = R(1) - k1;
    const R A = R(1) - R(0.5) * om, rest = R(-0.5) * om - (A - R(1));  // A + rest = 1 - om/2 exactly
    OddConstants<R> best{};
    double least = 4.0;
    for (int i = 0; i < 1024 && least > enough; ++i) {
        const R c = R(0.125) + R(i) * R(0x1p-20), c3 = R(3) * c, a = om / c3, b = A / c3;
        const double off = std::fabs(double(std::fma(a, c3, -om))) + std::fabs(double(std::fma(b, c3, -A) - rest));
        if (off < least) least = off, best = OddConstants<R>{c, a, b};
    }
    return best;
}

}  // namespace
