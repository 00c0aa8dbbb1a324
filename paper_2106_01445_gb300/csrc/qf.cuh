// Software floating point with a 110-bit significand on the integer pipes, for the double-double
// paths.  The FP64 pipe of this GPU issues two lanes a clock and SM (a double-double multiply-
// subtract c - a0 b0 - a1 b1 is 27 of its instructions, 216 clocks of an SM a warp); the same
// operation here is about 130 integer instructions, 33 to 40 clocks, on 110 bits.
//
// A number is M 2^-110 4^e: M a signed 112-bit integer in three 30-bit limbs and a signed 22-bit top
// limb, normalised to 2^109 <= |M| <= 2^111 (zero: M = 0), e in [-512, 511] (the range of a double), in
// 16 bytes: w[0..2] the limbs, w[3] = top limb 2^10 + e + 512.  Results are truncated: a product below 2^-109
// of itself, a sum below 2^-108 of the larger operand.  The fused forms shift the factor of a smaller
// product in the product's place, which loses up to 2^-107 of the largest term a factor shifted: below
// 2^-106 of it for two terms (dot2, fma), 2^-105 for three (fms2), k 2^-107 for k (dot).  (Against a 192-bit sum
// the sweep's results are off by less than 2^-117 kappa, double-double's by 2^-112: truncations average out.)
// Limbs of 30 bits let every partial product of a column accumulate in 64 bits without a carry (fl.cuh);
// the exponent's base 4 keeps the normalising shift even, so that reciprocal square roots need no odd
// case of their own.
// Overflow saturates the exponent (a saturated number converts to NaN), underflow gives zero.
#pragma once
#include <stdint.h>

#include "fx.cuh"

struct __align__(16) qf {
    uint32_t w[4];
};

namespace qfn {

constexpr int32_t kM = 0x3fffffff;
#define QF_FN __host__ __device__ __forceinline__

struct reg {  // unpacked
    int32_t l[4];
    int e;
};
QF_FN reg unpack(const qf &a) {
    return reg{{(int32_t)a.w[0], (int32_t)a.w[1], (int32_t)a.w[2], (int32_t)a.w[3] >> 10}, (int)(a.w[3] & 0x3ffu) - 512};
}
QF_FN int64_t mw(int32_t a, int32_t b) { return (int64_t)a * (int64_t)b; }
QF_FN int lead(int64_t a) {  // floor(log2 a) for a > 0
#ifdef __CUDA_ARCH__
    return 63 - __clzll(a);
#else
    return 63 - __builtin_clzll((unsigned long long)a);
#endif
}
// l >> bits (arithmetic; bits >= 0)
QF_FN void shr(int32_t l[4], int bits) {
    if (bits >= 30) {  // whole limbs, by selects
        const int32_t sg = l[3] >> 31;
        bits = bits > 119 ? 119 : bits;
        const bool c2 = bits >= 60;
        l[0] = c2 ? l[2] : l[0];
        l[1] = c2 ? l[3] & kM : l[1];
        l[2] = c2 ? sg & kM : l[2];
        l[3] = c2 ? sg : l[3];
        bits -= c2 ? 60 : 0;
        const bool c1 = bits >= 30;
        l[0] = c1 ? l[1] : l[0];
        l[1] = c1 ? l[2] : l[1];
        l[2] = c1 ? l[3] & kM : l[2];
        l[3] = c1 ? sg : l[3];
        bits -= c1 ? 30 : 0;
    }
    const int u = 30 - bits;
    l[0] = (int32_t)(((uint32_t)l[0] >> bits) | ((uint32_t)l[1] << u)) & kM;
    l[1] = (int32_t)(((uint32_t)l[1] >> bits) | ((uint32_t)l[2] << u)) & kM;
    l[2] = (int32_t)(((uint32_t)l[2] >> bits) | ((uint32_t)l[3] << u)) & kM;
    l[3] >>= bits;
}
// columns p[0..3] (weights 2^(30 k), any sign) to limbs r[0..3] and a signed r4
QF_FN void carry(const int64_t p[4], int32_t r[5]) {
    int64_t x = p[0];
    r[0] = (int32_t)x & kM;
    x = p[1] + (x >> 30);
    r[1] = (int32_t)x & kM;
    x = p[2] + (x >> 30);
    r[2] = (int32_t)x & kM;
    x = p[3] + (x >> 30);
    r[3] = (int32_t)x & kM;
    r[4] = (int32_t)(x >> 30);
}
QF_FN qf pack(const int32_t l[4], int e) {
    if (e < -512) return qf{{0u, 0u, 0u, 0u}};
    e = e > 511 ? 511 : e;
    return qf{{(uint32_t)l[0], (uint32_t)l[1], (uint32_t)l[2], ((uint32_t)l[3] << 10) | (uint32_t)(e + 512)}};
}
// sum_k r[k] 2^(30 k) times 2^-S 4^e (S even), normalised, for sizes below 2^139.  The operations
// below form their results around 2^130, so that cancellations of up to 20 bits take no branch.
QF_FN qf normal(int32_t r[5], int S, int e) {
    int64_t hi = ((int64_t)r[4] << 30) + r[3];
    for (int k = 0; (hi ^ (hi >> 63)) == 0; ++k) {  // only the sign is left on top: move a limb up
        if (k == 3) {
            if (hi >= 0) return qf{{0u, 0u, 0u, 0u}};  // zero
            break;
        }
        r[3] = r[2];
        r[2] = r[1];
        r[1] = r[0];
        r[0] = 0;
        hi = ((int64_t)(int32_t)(hi >> 63) << 30) + r[3];
        r[4] = (int32_t)(hi >> 30);
        S += 30;
    }
    const int64_t m = hi ^ (hi >> 63);
    const int L = m ? lead(m) + 91 : 90;  // bits of the magnitude
    int s = (L - 110) & ~1;
    e += (s - S + 110) >> 1;
    if (s < 0) {  // L < 110: at most 20 bits to the left; one limb up and the rest back
        r[4] = (int32_t)hi;  // = r4 2^30 + r3, below 2^20 in size
        r[3] = r[2];
        r[2] = r[1];
        r[1] = r[0];
        r[0] = 0;
        s += 30;
    }
    const int u = 30 - s;
    int32_t l[4];
    l[0] = (int32_t)(((uint32_t)r[0] >> s) | ((uint32_t)r[1] << u)) & kM;
    l[1] = (int32_t)(((uint32_t)r[1] >> s) | ((uint32_t)r[2] << u)) & kM;
    l[2] = (int32_t)(((uint32_t)r[2] >> s) | ((uint32_t)r[3] << u)) & kM;
    l[3] = (int32_t)(((uint32_t)r[3] >> s) | ((uint32_t)r[4] << u));
    return pack(l, e);
}
// columns 3..6 of a b added to p, column 2 to p2 (columns 0 and 1 are below 2^-126 of the product)
QF_FN void mac(int64_t &p2, int64_t p[4], const int32_t a[4], const int32_t b[4]) {
    p2 += mw(a[0], b[2]) + mw(a[1], b[1]) + mw(a[2], b[0]);
    p[0] += mw(a[0], b[3]) + mw(a[1], b[2]) + mw(a[2], b[1]) + mw(a[3], b[0]);
    p[1] += mw(a[1], b[3]) + mw(a[2], b[2]) + mw(a[3], b[1]);
    p[2] += mw(a[2], b[3]) + mw(a[3], b[2]);
    p[3] += mw(a[3], b[3]);
}
// the columns of a product: value = columns 2^-130 4^(ea + eb)
constexpr int kS = 130;

}  // namespace qfn

QF_FN qf qf_zero() { return qf{{0u, 0u, 0u, 0u}}; }
QF_FN qf qf_one() { return qf{{0u, 0u, 0u, (1u << 30) | 512u}}; }  // M = 2^110
// x y, or -x y
template <bool NEG> QF_FN qf qf_mul(const qf &x, const qf &y) {
    using namespace qfn;
    reg a = unpack(x);
    const reg b = unpack(y);
    if (NEG)
        for (int k = 0; k < 4; ++k) a.l[k] = -a.l[k];
    int64_t p2 = 0, p[4] = {0, 0, 0, 0};
    mac(p2, p, a.l, b.l);
    p[0] += p2 >> 30;
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, a.e + b.e);
}
QF_FN qf operator*(const qf &x, const qf &y) { return qf_mul<false>(x, y); }
// x + y, or x - y
template <bool NEG> QF_FN qf qf_sum(const qf &x, const qf &y) {
    using namespace qfn;
    reg a = unpack(x), b = unpack(y);
    const int e = a.e > b.e ? a.e : b.e;
    int32_t big[4], sml[4];
    const bool af = a.e >= b.e;
    for (int k = 0; k < 4; ++k) {
        big[k] = af ? a.l[k] : (NEG ? -b.l[k] : b.l[k]);
        sml[k] = af ? b.l[k] : a.l[k];
    }
    shr(sml, 2 * (af ? a.e - b.e : b.e - a.e));
    int64_t p[4];
    for (int k = 0; k < 4; ++k) p[k] = (int64_t)(big[k] + (af && NEG ? -sml[k] : sml[k])) * (1 << 20);
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, e);
}
QF_FN qf operator+(const qf &x, const qf &y) { return qf_sum<false>(x, y); }
QF_FN qf operator-(const qf &x, const qf &y) { return qf_sum<true>(x, y); }
QF_FN qf operator-(const qf &x) { return qf_zero() - x; }
// x / 2 (truncated by at most one unit of M)
QF_FN qf qf_half(const qf &x) {
    using namespace qfn;
    const reg a = unpack(x);
    int64_t p[4];
    for (int k = 0; k < 4; ++k) p[k] = 2 * (int64_t)a.l[k];
    int32_t r[5];
    carry(p, r);
    return normal(r, 110, a.e - 1);
}
// sg0 a0 b0 + sg1 a1 b1
template <bool NEG0, bool NEG1> QF_FN qf qf_dot2(const qf &xa0, const qf &xb0, const qf &xa1, const qf &xb1) {
    using namespace qfn;
    reg a0 = unpack(xa0), a1 = unpack(xa1);
    const reg b0 = unpack(xb0), b1 = unpack(xb1);
    const int e0 = a0.e + b0.e, e1 = a1.e + b1.e, e = e0 > e1 ? e0 : e1;
    // the smaller product's factor is shifted in place of the product
    int32_t u[4], v[4];
    const bool f0 = e0 >= e1;
    for (int k = 0; k < 4; ++k) u[k] = f0 ? a1.l[k] : a0.l[k];
    shr(u, 2 * (f0 ? e0 - e1 : e1 - e0));
    for (int k = 0; k < 4; ++k) {
        v[k] = f0 ? (NEG0 ? -a0.l[k] : a0.l[k]) : (NEG0 ? -u[k] : u[k]);
        u[k] = f0 ? (NEG1 ? -u[k] : u[k]) : (NEG1 ? -a1.l[k] : a1.l[k]);
    }
    int64_t p2 = 0, p[4] = {0, 0, 0, 0};
    mac(p2, p, v, b0.l);
    mac(p2, p, u, b1.l);
    p[0] += p2 >> 30;
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, e);
}
// c + a b, with either sign
template <bool NEG, bool NEGC = false> QF_FN qf qf_fma(const qf &xc, const qf &xa, const qf &xb) {
    using namespace qfn;
    reg a = unpack(xa), c = unpack(xc);
    const reg b = unpack(xb);
    const int ep = a.e + b.e, e = ep > c.e ? ep : c.e;
    const bool pf = ep >= c.e;
    int32_t u[4];
    for (int k = 0; k < 4; ++k) u[k] = pf ? c.l[k] : a.l[k];
    shr(u, 2 * (pf ? ep - c.e : c.e - ep));
    int64_t p2 = 0, p[4];
    int32_t v[4];
    for (int k = 0; k < 4; ++k) {
        const int32_t g = pf ? u[k] : c.l[k], f = pf ? a.l[k] : u[k];
        p[k] = (int64_t)(NEGC ? -g : g) * (1 << 20);
        v[k] = NEG ? -f : f;
    }
    mac(p2, p, v, b.l);
    p[0] += p2 >> 30;
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, e);
}
// c - a0 b0 - a1 b1
QF_FN qf qf_fms2(const qf &xc, const qf &xa0, const qf &xb0, const qf &xa1, const qf &xb1) {
    using namespace qfn;
    reg a0 = unpack(xa0), a1 = unpack(xa1), c = unpack(xc);
    const reg b0 = unpack(xb0), b1 = unpack(xb1);
    const int e0 = a0.e + b0.e, e1 = a1.e + b1.e;
    const int em = e0 > e1 ? e0 : e1, e = em > c.e ? em : c.e;
    // of the three terms one keeps its place; shifts of zero bits cost the same as others
    shr(a0.l, 2 * (e - e0));
    shr(a1.l, 2 * (e - e1));
    shr(c.l, 2 * (e - c.e));
    int64_t p2 = 0, p[4];
    for (int k = 0; k < 4; ++k) {
        a0.l[k] = -a0.l[k];
        a1.l[k] = -a1.l[k];
        p[k] = (int64_t)c.l[k] * (1 << 20);
    }
    mac(p2, p, a0.l, b0.l);
    mac(p2, p, a1.l, b1.l);
    p[0] += p2 >> 30;
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, e);
}
// (-1)^neg0 a0 b0 + (-1)^neg1 a1 b1
QF_FN qf qf_dot2s(bool neg0, const qf &xa0, const qf &xb0, bool neg1, const qf &xa1, const qf &xb1) {
    using namespace qfn;
    reg a0 = unpack(xa0), a1 = unpack(xa1);
    const reg b0 = unpack(xb0), b1 = unpack(xb1);
    const int e0 = a0.e + b0.e, e1 = a1.e + b1.e, e = e0 > e1 ? e0 : e1;
    shr(a0.l, 2 * (e - e0));
    shr(a1.l, 2 * (e - e1));
    const int32_t m0 = -(int32_t)neg0, m1 = -(int32_t)neg1;
    for (int k = 0; k < 4; ++k) {
        a0.l[k] = (a0.l[k] ^ m0) - m0;
        a1.l[k] = (a1.l[k] ^ m1) - m1;
    }
    int64_t p2 = 0, p[4] = {0, 0, 0, 0};
    mac(p2, p, a0.l, b0.l);
    mac(p2, p, a1.l, b1.l);
    p[0] += p2 >> 30;
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, e);
}
// sum over i = i0, i0 + step, .. < n of a(i) b(i): one alignment to the largest exponent and one
// normalisation for the whole sum (n <= 64); a and b return pointers
template <typename FA, typename FB> QF_FN qf qf_dot(int i0, int step, int n, FA a, FB b) {
    using namespace qfn;
    int e = -100000;
    for (int i = i0; i < n; i += step) {
        const int et = (int)(a(i)->w[3] & 0x3ffu) + (int)(b(i)->w[3] & 0x3ffu);
        e = et > e ? et : e;
    }
    int64_t p2 = 0, p[4] = {0, 0, 0, 0};
    for (int i = i0; i < n; i += step) {
        reg x = unpack(*a(i));
        const reg y = unpack(*b(i));
        shr(x.l, 2 * (e - (x.e + y.e + 1024)));
        mac(p2, p, x.l, y.l);
        // keep the columns below 2^63
        p[0] += p2 >> 30;
        p2 &= kM;
        p[1] += p[0] >> 30;
        p[0] &= kM;
        p[2] += p[1] >> 30;
        p[1] &= kM;
    }
    int32_t r[5];
    carry(p, r);
    return normal(r, kS, e - 1024);
}
QF_FN bool qf_positive(const qf &a) {
    const int32_t t = (int32_t)a.w[3] >> 10;
    return t > 0 || (t == 0 && (a.w[0] | a.w[1] | a.w[2]) != 0u);
}
// overflowed, or from a double that is not finite
QF_FN bool qf_saturated(const qf &a) { return (a.w[3] & 0x3ffu) == 1023u; }
// exact (53 bits fit)
QF_FN qf qf_from_double(double d) {
    using namespace qfn;
    if (d == 0.0) return qf_zero();
    union { double f; unsigned long long u; } v;
    v.f = d;
    int ex = (int)((v.u >> 52) & 0x7ff);
    unsigned long long mant = v.u & ((1ull << 52) - 1);
    if (ex) mant |= 1ull << 52;
    else ex = 1;
    if (ex == 0x7ff) return qf{{0u, 0u, 0u, (uint32_t)((1 << 30) | 1023)}};  // saturated
    // d = mant 2^(ex - 1075)
    const int64_t sm = (v.u >> 63) ? -(int64_t)mant : (int64_t)mant;
    const int sh = (ex - 1075) & 1;
    const int64_t p[4] = {0, 0, (sm << sh), 0};  // weight 2^60
    int32_t r[5];
    carry(p, r);
    return normal(r, 60, (ex - 1075 - sh) / 2);
}
#ifdef __CUDACC__
// as a double-double (error below 2^-105); a saturated number is NaN
__device__ __forceinline__ dd qf_to_dd(const qf &x) {
    const qfn::reg a = qfn::unpack(x);
    const long long hi = ((long long)a.l[3] << 41) + ((long long)a.l[2] << 11) + (a.l[1] >> 19);  // M 2^-49
    const long long lo = ((long long)(a.l[1] & 0x7ffff) << 30) + a.l[0];
    const double h = (double)hi;
    const double l = (double)(hi - (long long)h) + (double)lo * 0x1p-49;
    const dd s = dd_quick_two_sum(h, l);
    if (a.e >= 511) return dd(__longlong_as_double(0x7ff8000000000000ll), 0.0);
    const double sc = ldexp(1.0, 2 * a.e - 61);
    return dd(s.hi * sc, s.lo * sc);
}
// 20 leading bits
__device__ __forceinline__ double qf_approx(const qf &x) {
    const int e = (int)(x.w[3] & 0x3ffu) - 512;
    return e < -500 ? 0.0 : (double)((int32_t)x.w[3] >> 10) * __hiloint2double((1003 + 2 * e) << 20, 0);
}
// x^{-1/2} for x > 0 (a finite, meaningless number otherwise): M 2^-110 4^(e mod 2) in [1/2, 8)
// through fx_rsqrt_at
__device__ __forceinline__ qf qf_rsqrt(const qf &x) {
    const qfn::reg a = qfn::unpack(x);
    const uint32_t w0 = (uint32_t)a.l[0], w1 = (uint32_t)a.l[1], w2 = (uint32_t)a.l[2], w3 = (uint32_t)a.l[3];
    const fx pk{{w0 | (w1 << 30), (w1 >> 2) | (w2 << 28), (w2 >> 4) | (w3 << 26), (uint32_t)(a.l[3] >> 6)}};
    const int odd = a.e & 1;
    const fx y = fx_rsqrt_at(pk, odd ? 19 : 17);  // Q16.112
    const uint32_t m = (uint32_t)qfn::kM;
    int32_t r[5] = {(int32_t)(y.w[0] & m), (int32_t)(__funnelshift_r(y.w[0], y.w[1], 30) & m),
                    (int32_t)(__funnelshift_r(y.w[1], y.w[2], 28) & m), (int32_t)(__funnelshift_r(y.w[2], y.w[3], 26) & m),
                    (int32_t)(y.w[3] >> 24)};
    return qfn::normal(r, 112, -((a.e - odd) >> 1));
}
#endif
