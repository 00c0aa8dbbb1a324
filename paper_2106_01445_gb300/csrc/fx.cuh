// 128-bit signed fixed point on the integer pipes: value = X * 2^-112 (Q16.112),
// X two's complement in four 32-bit limbs (w[0] least significant).
//
// Used for the Schur updates of the exact sweep, whose entries are bounded: A = I - O
// = sigma_Q^{-1} <= 2 I, so every Schur complement of A has entries in [-2, 2]; with
// pivot determinants >= 2^-8 (checked, see fl_pivot_bad) the inverse pivots, the rows
// W = B P^{-1} and every intermediate of c - w0 b0 - w1 b1 stay below 2^15.  Products
// are truncated to 2^-112 (partial products below bit 96 are dropped, error < 2^-13
// of the last place); sums are exact.
#pragma once
#include <stdint.h>

#include "dd.cuh"

struct fx {
    uint32_t w[4];
};

__device__ __forceinline__ fx fx_zero() { return fx{{0u, 0u, 0u, 0u}}; }
__device__ __forceinline__ fx fx_one() { return fx{{0u, 0u, 0u, 1u << 16}}; }

__device__ __forceinline__ fx operator+(const fx &a, const fx &b) {
    fx r;
    asm("add.cc.u32 %0, %4, %8;\n\t"
        "addc.cc.u32 %1, %5, %9;\n\t"
        "addc.cc.u32 %2, %6, %10;\n\t"
        "addc.u32 %3, %7, %11;"
        : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3])
        : "r"(a.w[0]), "r"(a.w[1]), "r"(a.w[2]), "r"(a.w[3]), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]),
          "r"(b.w[3]));
    return r;
}
__device__ __forceinline__ fx operator-(const fx &a, const fx &b) {
    fx r;
    asm("sub.cc.u32 %0, %4, %8;\n\t"
        "subc.cc.u32 %1, %5, %9;\n\t"
        "subc.cc.u32 %2, %6, %10;\n\t"
        "subc.u32 %3, %7, %11;"
        : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2]), "=r"(r.w[3])
        : "r"(a.w[0]), "r"(a.w[1]), "r"(a.w[2]), "r"(a.w[3]), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]),
          "r"(b.w[3]));
    return r;
}
__device__ __forceinline__ fx operator-(const fx &a) { return fx_zero() - a; }
__device__ __forceinline__ fx &operator+=(fx &a, const fx &b) { return a = a + b; }
__device__ __forceinline__ bool fx_positive(const fx &a) {
    return (int32_t)a.w[3] > 0 || (a.w[3] == 0u && (a.w[2] | a.w[1] | a.w[0]) != 0u);
}

// Limbs 3..7 of the unsigned 256-bit product a*b, without the partial products of
// columns 0 and 1 and the low halves of column 2.  Row i adds a_i * b; after row i
// the partial sum is below 2^(32 (i + 5)), so each row's carry ends in its last limb.
__device__ __forceinline__ void fx_mul_upper(const fx &a, const fx &b, uint32_t &p3, uint32_t &p4,
                                             uint32_t &p5, uint32_t &p6, uint32_t &p7) {
    // row 0: lo(a0 b3) -> 3; hi(a0 b2) -> 3, hi(a0 b3) -> 4
    asm("mul.lo.u32 %0, %2, %3;\n\t"
        "mad.hi.cc.u32 %0, %2, %4, %0;\n\t"
        "madc.hi.u32 %1, %2, %3, 0;"
        : "=&r"(p3), "=&r"(p4)
        : "r"(a.w[0]), "r"(b.w[3]), "r"(b.w[2]));
    // row 1: lo(a1 b2) -> 3, lo(a1 b3) -> 4, carry -> 5; hi(a1 b1) -> 3, hi(a1 b2) -> 4, hi(a1 b3) -> 5
    asm("mad.lo.cc.u32 %0, %3, %5, %0;\n\t"
        "madc.lo.cc.u32 %1, %3, %6, %1;\n\t"
        "addc.u32 %2, 0, 0;\n\t"
        "mad.hi.cc.u32 %0, %3, %4, %0;\n\t"
        "madc.hi.cc.u32 %1, %3, %5, %1;\n\t"
        "madc.hi.u32 %2, %3, %6, %2;"
        : "+r"(p3), "+r"(p4), "=&r"(p5)
        : "r"(a.w[1]), "r"(b.w[1]), "r"(b.w[2]), "r"(b.w[3]));
    // row 2: lo(a2 b1..b3) -> 3..5, carry -> 6; hi(a2 b0..b3) -> 3..6
    asm("mad.lo.cc.u32 %0, %4, %6, %0;\n\t"
        "madc.lo.cc.u32 %1, %4, %7, %1;\n\t"
        "madc.lo.cc.u32 %2, %4, %8, %2;\n\t"
        "addc.u32 %3, 0, 0;\n\t"
        "mad.hi.cc.u32 %0, %4, %5, %0;\n\t"
        "madc.hi.cc.u32 %1, %4, %6, %1;\n\t"
        "madc.hi.cc.u32 %2, %4, %7, %2;\n\t"
        "madc.hi.u32 %3, %4, %8, %3;"
        : "+r"(p3), "+r"(p4), "+r"(p5), "=&r"(p6)
        : "r"(a.w[2]), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]), "r"(b.w[3]));
    // row 3: lo(a3 b0..b3) -> 3..6, carry -> 7; hi(a3 b0..b3) -> 4..7
    asm("mad.lo.cc.u32 %0, %5, %6, %0;\n\t"
        "madc.lo.cc.u32 %1, %5, %7, %1;\n\t"
        "madc.lo.cc.u32 %2, %5, %8, %2;\n\t"
        "madc.lo.cc.u32 %3, %5, %9, %3;\n\t"
        "addc.u32 %4, 0, 0;\n\t"
        "mad.hi.cc.u32 %1, %5, %6, %1;\n\t"
        "madc.hi.cc.u32 %2, %5, %7, %2;\n\t"
        "madc.hi.cc.u32 %3, %5, %8, %3;\n\t"
        "madc.hi.u32 %4, %5, %9, %4;"
        : "+r"(p3), "+r"(p4), "+r"(p5), "+r"(p6), "=&r"(p7)
        : "r"(a.w[3]), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]), "r"(b.w[3]));
}

// bits 112..239 of the product held in limbs 3..7
__device__ __forceinline__ fx fx_shift_out(uint32_t p3, uint32_t p4, uint32_t p5, uint32_t p6, uint32_t p7) {
    fx r;
    r.w[0] = __funnelshift_r(p3, p4, 16);
    r.w[1] = __funnelshift_r(p4, p5, 16);
    r.w[2] = __funnelshift_r(p5, p6, 16);
    r.w[3] = __funnelshift_r(p6, p7, 16);
    return r;
}
// p4..p7 -= m & x  (the two's-complement correction 2^128 x [sign] of a signed factor)
__device__ __forceinline__ void fx_sub_masked(uint32_t &p4, uint32_t &p5, uint32_t &p6, uint32_t &p7,
                                              const fx &x, uint32_t m) {
    asm("sub.cc.u32 %0, %0, %4;\n\t"
        "subc.cc.u32 %1, %1, %5;\n\t"
        "subc.cc.u32 %2, %2, %6;\n\t"
        "subc.u32 %3, %3, %7;"
        : "+r"(p4), "+r"(p5), "+r"(p6), "+r"(p7)
        : "r"(x.w[0] & m), "r"(x.w[1] & m), "r"(x.w[2] & m), "r"(x.w[3] & m));
}
__device__ __forceinline__ uint32_t fx_sign_mask(const fx &a) { return (uint32_t)((int32_t)a.w[3] >> 31); }

// a * b for a, b >= 0
__device__ __forceinline__ fx fx_mul_uu(const fx &a, const fx &b) {
    uint32_t p3, p4, p5, p6, p7;
    fx_mul_upper(a, b, p3, p4, p5, p6, p7);
    return fx_shift_out(p3, p4, p5, p6, p7);
}
// a * b for b >= 0, a of either sign: the unsigned product minus 2^128 b [a < 0], bits 112..239
__device__ __forceinline__ fx fx_mul_su(const fx &a, const fx &b) {
    uint32_t p3, p4, p5, p6, p7;
    fx_mul_upper(a, b, p3, p4, p5, p6, p7);
    fx_sub_masked(p4, p5, p6, p7, b, fx_sign_mask(a));
    return fx_shift_out(p3, p4, p5, p6, p7);
}

__device__ __forceinline__ fx fx_from_i128(__int128 v) {
    fx r;
    r.w[0] = (uint32_t)v;
    r.w[1] = (uint32_t)(v >> 32);
    r.w[2] = (uint32_t)(v >> 64);
    r.w[3] = (uint32_t)(v >> 96);
    return r;
}
// exact for |d| < 2^15 down to 2^-112 (lower bits truncated toward zero); zero outside
__device__ __forceinline__ fx fx_from_double(double d) {
    const unsigned long long bits = (unsigned long long)__double_as_longlong(d);
    const int ex = (int)((bits >> 52) & 0x7ff);
    if (ex == 0) return fx_zero();
    const unsigned long long mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const int s = ex - 963;  // d * 2^112 = mant * 2^(ex - 1075 + 112)
    if (s > 74) return fx_zero();  // |d| >= 2^15 (or not finite): outside the format
    unsigned __int128 v;
    if (s >= 0) v = (unsigned __int128)mant << s;
    else v = s > -64 ? (unsigned __int128)(mant >> (-s)) : (unsigned __int128)0;
    __int128 x = (__int128)v;
    if (bits >> 63) x = -x;
    return fx_from_i128(x);
}
// nearest-double leading part of a
__device__ __forceinline__ double fx_to_double(const fx &a) {
    const long long hi = (long long)(((unsigned long long)a.w[3] << 32) | a.w[2]);
    return (double)hi * 0x1p-48;
}
// a as a double-double (the top 64 bits rounded to a double, the remainder below)
__device__ __forceinline__ dd fx_to_dd(const fx &a) {
    const long long hi = (long long)(((unsigned long long)a.w[3] << 32) | a.w[2]);
    const unsigned long long lo = ((unsigned long long)a.w[1] << 32) | a.w[0];
    const double h = (double)hi;
    const long long rem = hi - (long long)h;  // |rem| <= 2^10: exact
    const double l = (double)rem + (double)lo * 0x1p-64;
    const dd s = dd_quick_two_sum(h, l);
    return dd(s.hi * 0x1p-48, s.lo * 0x1p-48);
}


// x^{-1/2} in Q16.112 for a packed x with ulp 2^-(127 - h0) (h0 = 15: Q16.112; h0 = 13: ulp
// 2^-114) in [2^-11, 2^11); pivots that pass the checks lie in [2^-10.4, 25].
//  * x = m 4^h', m in [1/2, 2): an odd shift s of X (m = 1 for the powers of four, which stay exact);
//  * an FP32 estimate r0 of r = m^{-1/2} (relative error below 2^-22), 24 bits, scale 30;
//  * one step of third order on the top 64 bits W of m: with e = 1 - m r0^2, r = r0 (1 + e/2 +
//    3/8 e^2) leaves 5/16 e^3 < 2^-64, so one step stands for the two Newton steps a quadratic
//    iteration needs: R = r 2^62 to 2^-61;
//  * one Newton step against the whole of x: with |e| < 2^-59 known, only the bits of m R^2 below
//    2^-59 are formed (columns 3, 4 and the low half of 5 of X R^2: nine products instead of two
//    full 128 x 64 ones), E = e 2^121, and y += y e / 2.
// The result is within one unit of 2^-112 (a big-integer emulation over the whole range, the FP32 estimate off
// by up to two units); exact for powers of four.  Inputs outside the range (checked by the callers) give a finite, meaningless
// result.
static __device__ __noinline__ fx fx_rsqrt_at(fx x, int h0) {
    int lz = __clz((int)x.w[3]);
    lz = lz < 3 ? 3 : (lz > 31 ? 31 : lz);
    const int s = (lz - 1) | 1;
    const int h = (h0 - s) >> 1;
    const unsigned long long W = ((unsigned long long)__funnelshift_l(x.w[2], x.w[3], s) << 32) |
                                 __funnelshift_l(x.w[1], x.w[2], s);
    const int sx = s - 2;
    const uint32_t x0 = x.w[0] << sx, x1 = __funnelshift_l(x.w[0], x.w[1], sx),
                   x2 = __funnelshift_l(x.w[1], x.w[2], sx), x3 = __funnelshift_l(x.w[2], x.w[3], sx);
    const uint32_t fb = __float_as_uint(rsqrtf(__uint2float_rn((uint32_t)(W >> 32)) * 0x1p-31f));
    const uint32_t r0 = ((fb & 0x7fffffu) | 0x800000u) << (((fb >> 23) - 120u) & 7u);
    const unsigned long long P = __umul64hi(W, ((unsigned long long)r0 * r0) << 2);  // m r0^2 2^61
    const long long E0 = (long long)((1ull << 61) - P);
    const int e32 = (int)(E0 >> 11);
    const int t = (int)(((long long)e32 * e32) >> 32);  // e^2 2^68
    const long long D = E0 + ((3 * t) >> 9);            // (e/2 + 3/8 e^2) 2^62
    const unsigned long long R = ((unsigned long long)r0 << 32) +
                                 (((unsigned long long)((long long)(int)r0 * (int)(D >> 32))) << 2) +
                                 (((unsigned long long)r0 * (uint32_t)D) >> 30);
    // Q = R^2, 128 bits
    const uint32_t ra = (uint32_t)R, rb = (uint32_t)(R >> 32);
    const unsigned long long aa = (unsigned long long)ra * ra, ab = (unsigned long long)ra * rb,
                             bb = (unsigned long long)rb * rb;
    const unsigned long long mid = (ab << 1) + (aa >> 32);  // ab < 2^63: no carry lost
    const unsigned long long top = bb + (mid >> 32) + ((mid < (aa >> 32)) ? (1ull << 32) : 0ull);
    const uint32_t q0 = (uint32_t)aa, q1 = (uint32_t)mid, q2 = (uint32_t)top, q3 = (uint32_t)(top >> 32);
    const unsigned long long S = ((unsigned long long)__umulhi(x0, q3) + __umulhi(x1, q2)) +
                                 ((unsigned long long)__umulhi(x2, q1) + __umulhi(x3, q0)) +
                                 (unsigned long long)x1 * q3 + (unsigned long long)x2 * q2 +
                                 (unsigned long long)x3 * q1 + ((unsigned long long)(x2 * q3 + x3 * q2) << 32);
    const long long E = -(long long)S;  // e 2^121 modulo 2^64
    // y = r 2^-h in Q16.112: R 2^(50 - h), plus R E 2^(-72 - h)
    int s2 = 18 - h;
    s2 = s2 > 26 ? 26 : s2;
    const long long dlt = __mul64hi((long long)R, E) >> (8 + h);
    const uint32_t ext = (uint32_t)(dlt >> 63);
    return fx{{0u, ra << s2, __funnelshift_l(ra, rb, s2), rb >> (32 - s2)}} +
           fx{{(uint32_t)dlt, (uint32_t)((unsigned long long)dlt >> 32), ext, ext}};
}
__device__ __forceinline__ fx fx_rsqrt(const fx &x) { return fx_rsqrt_at(x, 15); }

// Symmetric form of the 2x2 block elimination used by the fixed-point sweeps.  With
// the pivot block P = R R^T (R lower triangular, 1/r00 = a, r10, 1/r11 = b), the
// Schur update C - B P^{-1} B^T equals C - U U^T, U = B R^{-T}: row i of U is
// u0 = b_i0 a, u1 = (b_i1 - r10 u0) b = b_i1 b - u0 c with c = r10 b = p01 det^{-1/2}
// (two products side by side), and |u_ik| <= sqrt(c_ii).  a = p00^{-1/2} and rs = det^{-1/2}
// are independent, so the two rsqrts need not wait for each other: b = rs sqrt(p00) = rs p00 a.

// a >> k for 0 <= k <= 31 (arithmetic)
__device__ __forceinline__ fx fx_shr_small(const fx &a, int k) {
    fx r;
    r.w[0] = __funnelshift_r(a.w[0], a.w[1], k);
    r.w[1] = __funnelshift_r(a.w[1], a.w[2], k);
    r.w[2] = __funnelshift_r(a.w[2], a.w[3], k);
    r.w[3] = (uint32_t)((int32_t)a.w[3] >> k);
    return r;
}
// a >> s for any s >= 0 (arithmetic; s >= 127 leaves the sign)
__device__ __forceinline__ fx fx_shr(const fx &a, int s) {
    const uint32_t sg = (uint32_t)((int32_t)a.w[3] >> 31);
    if (s > 127) s = 127;
    const int q = s >> 5, b = s & 31;
    // limb shift by q (selects, no indexed local memory), then the bit shift
    const uint32_t w0 = q == 0 ? a.w[0] : q == 1 ? a.w[1] : q == 2 ? a.w[2] : a.w[3];
    const uint32_t w1 = q == 0 ? a.w[1] : q == 1 ? a.w[2] : q == 2 ? a.w[3] : sg;
    const uint32_t w2 = q == 0 ? a.w[2] : q == 1 ? a.w[3] : sg;
    const uint32_t w3 = q == 0 ? a.w[3] : sg;
    return fx_shr_small(fx{{w0, w1, w2, w3}}, b);
}
__device__ __forceinline__ fx fx_shfl_xor(const fx &a, int mask) {
    fx r;
#pragma unroll
    for (int k = 0; k < 4; ++k) r.w[k] = __shfl_xor_sync(0xffffffffu, a.w[k], mask);
    return r;
}
__device__ __forceinline__ fx fx_neg_if(const fx &a, bool neg) { return neg ? -a : a; }
