// A rough log10 of the condition number kappa = sum |terms| / |sum| of a pattern's signed sum, before any of its
// 2^n terms is formed: which of two arithmetics takes the pattern is then decided without trying one first.
//
// The pattern's modes in pairs, as if the pairs were independent: per pair the four terms, and the product
// of the pairs' kappas.  What the pairs leave out (the correlations between them) only lowers the true kappa:
// on 480 patterns of 12 to 18 clicks (Haar and local interferometers of 24 to 100 modes, transmission 0.3 to 1,
// squeezing 0.2 to 1.4) with kappa from 1e5 to 1e35 the guess was 1.05 to 1.6 times its exponent.  Beyond 33 were
// 30 of the 35 patterns with kappa above 1e26, 8 of 22 between 1e24 and 1e26, 7 of 39 between 1e22 and 1e24
// and 1 of 384 below.  (Blocks of four modes, at 25 times the work, told no better.)
//
// Measured on a GB300: GBS_DD on 40 patterns of 18 clicks at 100 modes 12.50 -> 8.54 ms (double-double alone
// 8.51), of 16 to 18 clicks (kappa 1e25 to 5e29, some guesses below the line) 7.68 -> 6.43 (5.17); the gradient of 64
// patterns of 15 to 17 clicks at 40 modes, 62 of them above 1e24, 63.7 -> 50.8 ms (double-double alone 50.0);
// batches without such patterns unchanged.
#pragma once
#include <stdint.h>

constexpr float kGuessRedo = 33.0f;   // decades: the pattern is double-double's
constexpr int kGuessFrom = 14;        // clicks: a smaller pattern is not worth the guess

// By one warp, a lane a pair (n <= 64).  det - 1 of a mode in FP64, where nearly dark detectors cancel; from there
// on every sum is of positive terms (for a state's O; any number serves for another) and FP32 does.
template <typename Mode>
__device__ __forceinline__ float kappa_guess(const double *__restrict__ O, int M, const Mode *modes, int n) {
    const int lane = threadIdx.x & 31, N2 = 2 * M;
    float k = 0.0f;
    if (2 * lane < n) {
        const int m0 = modes[2 * lane];
        auto at = [&](int i, int j) { return O[(size_t)i * N2 + j]; };
        // d = det^{-1/2} and d - 1 of one mode's block A = I - O
        auto mode = [&](int m, float &a00, float &a01, float &a11, float &d, float &e) {
            const double x = at(m, m), y = at(m, m + M), z = at(m + M, m + M);
            const float del = (float)(x * z - y * y - (x + z));  // det - 1
            a00 = (float)(1.0 - x), a01 = (float)-y, a11 = (float)(1.0 - z);
            const float r = sqrtf(1.0f + del);
            d = 1.0f / r;
            e = -del / (1.0f + del + r);
        };
        float p00, p01, p11, d0, e0, A, T;
        mode(m0, p00, p01, p11, d0, e0);
        if (2 * lane + 1 < n) {
            const int m1 = modes[2 * lane + 1];
            float q00, q01, q11, d1, e1;
            mode(m1, q00, q01, q11, d1, e1);
            const float b00 = (float)at(m0, m1), b01 = (float)at(m0, m1 + M), b10 = (float)at(m0 + M, m1),
                        b11 = (float)at(m0 + M, m1 + M), inv = d0 * d0;
            // X = B^T P^{-1} B, and det(Q - X) / det Q = 1 - f
            const float u00 = (p11 * b00 - p01 * b10) * inv, u01 = (p11 * b01 - p01 * b11) * inv,
                        u10 = (p00 * b10 - p01 * b00) * inv, u11 = (p00 * b11 - p01 * b01) * inv;
            const float x00 = b00 * u00 + b10 * u10, x01 = b00 * u01 + b10 * u11, x11 = b01 * u01 + b11 * u11;
            const float f = (q11 * x00 - 2.0f * q01 * x01 + q00 * x11 - (x00 * x11 - x01 * x01)) * d1 * d1;
            const float r = sqrtf(1.0f - f), h = f / (1.0f - f + r);  // (1 - f)^{-1/2} - 1
            A = 1.0f + d0 + d1 + d0 * d1 * (1.0f + h);
            T = e0 * e1 + d0 * d1 * h;
        } else {
            A = 1.0f + d0;
            T = e0;
        }
        const float v = log10f(A) - log10f(fabsf(T));
        k = v == v ? fminf(v, 40.0f) : 0.0f;  // no number: the sweep will tell
    }
#pragma unroll
    for (int off = 16; off; off >>= 1) k += __shfl_xor_sync(0xffffffffu, k, off);
    return k;
}
