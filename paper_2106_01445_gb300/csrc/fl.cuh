// Limb form of the 128-bit fixed point: four 30-bit limbs, value = sum_i w[i] 2^(30 i) 2^-s,
// w[0..2] in [0, 2^30), w[3] signed.  The breadth-first levels and the register bottom of the
// fixed-point sweep keep their matrices in it.
//
// Why limbs of 30 bits.  A product of two packed 128-bit numbers is one long carry chain: 23
// IMADs that each wait for the carry of the one before, four funnel shifts to realign, and sign
// corrections.  With 30-bit limbs a partial product is below 2^60, so a column of a product (of
// two products side by side, for an update) is summed in a 64-bit register with no carry at all:
// each partial product is one IMAD.WIDE, the columns are independent chains, signed numbers need
// no correction, and one carry pass of five instructions a limb ends the whole entry.  The scales
// are chosen so that every product needs whole limbs only (no shifts):
//   matrix entries C, B, P     s = 114  (|x| < 32; a Schur complement of A <= 5 I stays below 5)
//   rows U = B R^-T            s = 117  (|u| <= sqrt(c_ii) < 4)
//   1/r00 and 1/r11 (a, b)     s = 123, five limbs     r10/(r00 r11) (c)     s = 120, five limbs
// with u u at 234 = 114 + 4 limbs and entry x a, u x c at 237 = 117 + 4 limbs.  Columns below
// the one that feeds the carry are dropped from u u: an entry update is high by at most 7 units of
// 2^-114 (the packed form: 2 units of 2^-112, i.e. 8 of these).
//
// Top limbs are cut to 32 bits, so the bounds above have to hold.  They do for every subset if A = I - O on
// the pattern's modes is positive definite (u_i u_i <= c_ii <= 5: the gather admits |O| <= 4), and that
// is what the chain of includes of all modes, one of the pattern's 2^n, tells: on it every row is checked
// before the cut (|u| < 4) and no diagonal entry may become negative, which keeps the others below
// 9 as well.  (Checked on every row of every subset the sweep was 2 to 5% slower, so it is 1%.)
//
// Measured on a GB300 at 128 threads x 4 CTAs per SM, independent updates: 0.77 SM clocks an
// entry against 1.18 for the packed form; IMAD.WIDE runs at 27 lanes per SM clock (plain IMAD at
// 59), so the 20 of an update take 0.73: the loop is at the multiplier's limit.  The 24-mode
// batch (2.42e8 subsets) went from 37.8 to 29.7 ms, with the same outputs bit for bit.
#pragma once
#include <stdint.h>

#include "fx.cuh"

struct __align__(16) fl {
    int32_t w[4];
};
struct fl5 {
    int32_t w[5];
};

constexpr int32_t kLimbMask = 0x3fffffff;

__device__ __forceinline__ int64_t fl_mw(int32_t a, int32_t b) { return (int64_t)a * (int64_t)b; }


// Q16.112 -> scale 114 (|x| < 128)
__device__ __forceinline__ fl fl_from_fx(const fx &a) {
    fl r;
    r.w[0] = (int32_t)((a.w[0] << 2) & (uint32_t)kLimbMask);
    r.w[1] = (int32_t)(__funnelshift_r(a.w[0], a.w[1], 28) & (uint32_t)kLimbMask);
    r.w[2] = (int32_t)(__funnelshift_r(a.w[1], a.w[2], 26) & (uint32_t)kLimbMask);
    r.w[3] = (int32_t)__funnelshift_r(a.w[2], a.w[3], 24);
    return r;
}
// scale 114 -> packed two's complement with ulp 2^-114
__device__ __forceinline__ fx fl_pack(const fl &a) {
    const uint32_t w0 = (uint32_t)a.w[0], w1 = (uint32_t)a.w[1], w2 = (uint32_t)a.w[2], w3 = (uint32_t)a.w[3];
    return fx{{w0 | (w1 << 30), (w1 >> 2) | (w2 << 28), (w2 >> 4) | (w3 << 26), (uint32_t)(a.w[3] >> 6)}};
}
// a positive Q16.112 number below 2^7 at scale 123 and at scale 126, five limbs
__device__ __forceinline__ fl5 fl5_at123(const fx &y) {
    const uint32_t m = (uint32_t)kLimbMask;
    return fl5{{(int32_t)((y.w[0] << 11) & m), (int32_t)(__funnelshift_r(y.w[0], y.w[1], 19) & m),
                (int32_t)(__funnelshift_r(y.w[1], y.w[2], 17) & m), (int32_t)(__funnelshift_r(y.w[2], y.w[3], 15) & m),
                (int32_t)(y.w[3] >> 13)}};
}
__device__ __forceinline__ fl5 fl5_at126(const fx &y) {
    const uint32_t m = (uint32_t)kLimbMask;
    return fl5{{(int32_t)((y.w[0] << 14) & m), (int32_t)(__funnelshift_r(y.w[0], y.w[1], 16) & m),
                (int32_t)(__funnelshift_r(y.w[1], y.w[2], 14) & m), (int32_t)(__funnelshift_r(y.w[2], y.w[3], 12) & m),
                (int32_t)(y.w[3] >> 10)}};
}

// columns 3..7 of a (four limbs) times b (five limbs), added to p
__device__ __forceinline__ void fl_mac45(int64_t p[5], const fl &a, const fl5 &b) {
    p[0] += fl_mw(a.w[0], b.w[3]) + fl_mw(a.w[1], b.w[2]) + fl_mw(a.w[2], b.w[1]) + fl_mw(a.w[3], b.w[0]);
    p[1] += fl_mw(a.w[0], b.w[4]) + fl_mw(a.w[1], b.w[3]) + fl_mw(a.w[2], b.w[2]) + fl_mw(a.w[3], b.w[1]);
    p[2] += fl_mw(a.w[1], b.w[4]) + fl_mw(a.w[2], b.w[3]) + fl_mw(a.w[3], b.w[2]);
    p[3] += fl_mw(a.w[2], b.w[4]) + fl_mw(a.w[3], b.w[3]);
    p[4] += fl_mw(a.w[3], b.w[4]);
}
// limbs of columns 4..7 with the carry of column 3: x2^-120; top: the last one before it is cut to 32 bits
__device__ __forceinline__ fl fl_carry(const int64_t p[5], int64_t &top) {
    fl r;
    int64_t x = p[1] + (p[0] >> 30);
    r.w[0] = (int32_t)x & kLimbMask;
    x = p[2] + (x >> 30);
    r.w[1] = (int32_t)x & kLimbMask;
    x = p[3] + (x >> 30);
    r.w[2] = (int32_t)x & kLimbMask;
    top = p[4] + (x >> 30);
    r.w[3] = (int32_t)top;
    return r;
}
__device__ __forceinline__ fl fl_carry(const int64_t p[5]) {
    int64_t top;
    return fl_carry(p, top);
}
__device__ __forceinline__ fl5 fl5_carry(const int64_t p[5]) {
    fl5 r;
    int64_t x = p[1] + (p[0] >> 30);
    r.w[0] = (int32_t)x & kLimbMask;
    x = p[2] + (x >> 30);
    r.w[1] = (int32_t)x & kLimbMask;
    x = p[3] + (x >> 30);
    r.w[2] = (int32_t)x & kLimbMask;
    x = p[4] + (x >> 30);
    r.w[3] = (int32_t)x & kLimbMask;
    r.w[4] = (int32_t)(x >> 30);
    return r;
}

// p00 p11 - p01^2 (scale 228) as a packed number with ulp 2^-114; columns 0 and 1 dropped
__device__ __forceinline__ fx fl_det2(const fl &a, const fl &c, const fl &b) {
    const int32_t d0 = 2 * c.w[0], d1 = 2 * c.w[1], d2 = 2 * c.w[2];
    int64_t p2 = fl_mw(a.w[0], b.w[2]) + fl_mw(a.w[1], b.w[1]) + fl_mw(a.w[2], b.w[0]) - fl_mw(d0, c.w[2]) -
                 fl_mw(c.w[1], c.w[1]);
    int64_t p3 = fl_mw(a.w[0], b.w[3]) + fl_mw(a.w[1], b.w[2]) + fl_mw(a.w[2], b.w[1]) + fl_mw(a.w[3], b.w[0]) -
                 fl_mw(d0, c.w[3]) - fl_mw(d1, c.w[2]);
    int64_t p4 = fl_mw(a.w[1], b.w[3]) + fl_mw(a.w[2], b.w[2]) + fl_mw(a.w[3], b.w[1]) - fl_mw(d1, c.w[3]) -
                 fl_mw(c.w[2], c.w[2]);
    int64_t p5 = fl_mw(a.w[2], b.w[3]) + fl_mw(a.w[3], b.w[2]) - fl_mw(d2, c.w[3]);
    int64_t p6 = fl_mw(a.w[3], b.w[3]) - fl_mw(c.w[3], c.w[3]);
    p3 += p2 >> 30;
    p4 += p3 >> 30;
    p5 += p4 >> 30;
    p6 += p5 >> 30;
    const uint32_t m = (uint32_t)kLimbMask;
    const uint32_t l3 = (uint32_t)p3 & m, l4 = (uint32_t)p4 & m, l5 = (uint32_t)p5 & m, l6 = (uint32_t)p6 & m;
    return fx{{(l3 >> 24) | (l4 << 6), (l4 >> 26) | (l5 << 4), (l5 >> 28) | (l6 << 2), (uint32_t)(p6 >> 30)}};
}

// flags of a unit: 1 a pivot was not positive; 2 beyond the range on the chain of all includes; kFlLost the
// arithmetic left its range (an entry of O beyond 4, a determinant below 2^-8): what the unit finds besides,
// 1 included, may be noise, and it reports 2 alone
constexpr int kFlLost = 4;
__device__ __forceinline__ int fl_unit_flags(int f) { return f & kFlLost ? 2 : f; }
// pivot check of a determinant with ulp 2^-114: 0 fine, 1 not positive, kFlLost below 2^-8
__device__ __forceinline__ int fl_pivot_bad(const fx &det) {
    if (!fx_positive(det)) return 1;
    return (int32_t)det.w[3] < 1024 ? kFlLost : 0;
}
__device__ __forceinline__ bool fl_positive(const fl &a) {
    return a.w[3] > 0 || (a.w[3] == 0 && (a.w[2] | a.w[1] | a.w[0]) != 0);
}
__device__ __forceinline__ int fl_chol_bad(const fl &p00, const fx &det) {
    if (!fl_positive(p00)) return 1;
    return fl_pivot_bad(det);
}
__device__ __forceinline__ fx fl_rsqrt(const fx &x) { return fx_rsqrt_at(x, 13); }  // ulp 2^-114

// the 2x2 block elimination's quantities (see fx.cuh): a = p00^{-1/2}, b = det^{-1/2} p00^{1/2},
// c = p01 det^{-1/2}, from a and rs = det^{-1/2} (packed Q16.112)
struct fl_piv {
    fl5 a, b, c;
};
__device__ __forceinline__ fl_piv fl_pivot_from(const fl &p00, const fl &p01, const fx &ya, const fx &rs) {
    fl_piv v;
    v.a = fl5_at123(ya);
    const fl5 r = fl5_at126(rs);
    int64_t pc[5] = {0, 0, 0, 0, 0}, pq[5] = {0, 0, 0, 0, 0}, pb[5] = {0, 0, 0, 0, 0};
    fl_mac45(pc, p01, r);  // 114 + 126 = 120 + 120
    v.c = fl5_carry(pc);
    fl_mac45(pq, p00, v.a);  // sqrt(p00), scale 117
    fl_mac45(pb, fl_carry(pq), r);  // 117 + 126 = 123 + 120
    v.b = fl5_carry(pb);
    return v;
}
// row (u0, u1) of U = B R^{-T}: u0 = b0 a, u1 = b1 b - u0 c; bits of `out` are set if it is outside [-4, 4)
__device__ __forceinline__ void fl_urow(const fl5 &a, const fl5 &b, const fl5 &c, const fl &b0, const fl &b1, fl &u0,
                                        fl &u1, uint32_t &out) {
    int64_t p[5] = {0, 0, 0, 0, 0}, q[5] = {0, 0, 0, 0, 0}, top0, top1;
    fl_mac45(p, b0, a);
    fl_mac45(q, b1, b);
    u0 = fl_carry(p, top0);
    const fl n{{-u0.w[0], -u0.w[1], -u0.w[2], -u0.w[3]}};
    fl_mac45(q, n, c);
    u1 = fl_carry(q, top1);
    constexpr int64_t four = 1ll << 29;
    const uint64_t v = (uint64_t)((top0 + four) | (top1 + four));
    out |= (uint32_t)(v >> 32) | ((uint32_t)v & ~(uint32_t)kLimbMask);
}
__device__ __forceinline__ void fl_urow(const fl5 &a, const fl5 &b, const fl5 &c, const fl &b0, const fl &b1, fl &u0,
                                        fl &u1) {
    uint32_t out = 0;
    fl_urow(a, b, c, b0, b1, u0, u1, out);
}
__device__ __forceinline__ uint32_t fl_negative(const fl &a) { return (uint32_t)a.w[3] & 0x80000000u; }
// c - u_i . u_j
__device__ __forceinline__ fl fl_sym_update(const fl &c, const fl &a0, const fl &a1, const fl &b0, const fl &b1) {
    const int64_t p3 = fl_mw(a0.w[0], b0.w[3]) + fl_mw(a0.w[1], b0.w[2]) + fl_mw(a0.w[2], b0.w[1]) +
                       fl_mw(a0.w[3], b0.w[0]) + fl_mw(a1.w[0], b1.w[3]) + fl_mw(a1.w[1], b1.w[2]) +
                       fl_mw(a1.w[2], b1.w[1]) + fl_mw(a1.w[3], b1.w[0]);
    const int64_t p4 = fl_mw(a0.w[1], b0.w[3]) + fl_mw(a0.w[2], b0.w[2]) + fl_mw(a0.w[3], b0.w[1]) +
                       fl_mw(a1.w[1], b1.w[3]) + fl_mw(a1.w[2], b1.w[2]) + fl_mw(a1.w[3], b1.w[1]);
    const int64_t p5 = fl_mw(a0.w[2], b0.w[3]) + fl_mw(a0.w[3], b0.w[2]) + fl_mw(a1.w[2], b1.w[3]) +
                       fl_mw(a1.w[3], b1.w[2]);
    const int64_t p6 = fl_mw(a0.w[3], b0.w[3]) + fl_mw(a1.w[3], b1.w[3]);
    fl r;
    int64_t x = (int64_t)c.w[0] - p4 - (p3 >> 30);
    r.w[0] = (int32_t)x & kLimbMask;
    x = (int64_t)c.w[1] - p5 + (x >> 30);
    r.w[1] = (int32_t)x & kLimbMask;
    x = (int64_t)c.w[2] - p6 + (x >> 30);
    r.w[2] = (int32_t)x & kLimbMask;
    r.w[3] = c.w[3] + (int32_t)(x >> 30);
    return r;
}
