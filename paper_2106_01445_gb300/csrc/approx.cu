// The paper's moment approximation (Methods, "Partition function", "Moments
// calculation", "Approximation method") for click patterns S of n detectors:
//
//  1. sectors: Z_Z(t) = det(I - t O_Z)^{-1/2} = sum_k c_k[Z] t^k, where
//     c_k[Z] det(sigma_Q)^{-1/2} = P(k photons in Z, vacuum elsewhere).  The
//     coefficients are extracted by a discrete Fourier transform over
//     t_l = e^{i nu_l}, nu_l = 2 pi l / L (the paper's sum over nu);
//  2. moments: the minors with w <= j detectors removed give the factorial
//     moments of the vacuum count v in every sector,
//        D_w(t) = sum_{|W| = w} Z_{S \ W}(t),  D_w^(k) = sum_v C(v, w) q_k(v);
//     by Jacobi's identity Z_{S \ W}(t) = Z_S(t) det(G_WW)^{-1/2}, G = (I - t O_S)^{-1};
//  3. inverse moment problem: q_k(v) ~ exp(-f(v)), deg f <= j, moments 0..j
//     matched (convex maximum-entropy dual, damped Newton);
//  4. P(S) ~ det(sigma_Q)^{-1/2} sum_k exp(-f_k(0)).
//
// The circle |t| = rho is tilted to the Chernoff saddle of sector n so that the
// sectors carrying the all-clicked point (far in the upper tail for improbable
// patterns) sit near the peak of c_k rho^k and keep their relative precision.
// Kernels: approx_plan (per pattern: rho, and a rigorous bound K on the sector
// index with tilted tail < 1e-14 Z_S(rho) from Chernoff's inequality; DFT length
// L = K + 1), approx_minors (one CTA per (pattern, nu_l), l <= L/2 by conjugate
// symmetry), approx_fit (one CTA per pattern: inverse DFT, fits, sum).
#include <cooperative_groups.h>
#include <type_traits>
#include <math.h>

#include "ff.cuh"
#include "gbs_internal.cuh"

namespace cg = cooperative_groups;

#ifndef GBS_FF_FMS_INLINE
#define GBS_FF_FMS_INLINE __noinline__
#endif

namespace {

constexpr int kMaxOrder = 4;
constexpr int kMinorThreads = 256;
constexpr int kWideThreads = 512;   // of a minors CTA that has its SM to itself, orders 1 and 2
constexpr int kDftThreads = 128;
constexpr int kSecThreads = 256;   // one warp per sector
constexpr int kFitThreads = 128;   // a warp on several sectors
constexpr int kSumThreads = 128;   // one warp per pattern
constexpr int kPlanThreads = 256, kLogdetThreads = 128;
constexpr double kTailEps = 1e-14;
constexpr double kFlagShare = 1e-4;     // fallback reported when such sectors carry this share of P
constexpr int kNumRho = 15;
__constant__ double kRhos[kNumRho] = {1.0, 1.02, 1.05, 1.1, 1.15, 1.2, 1.25, 1.3, 1.4, 1.5, 1.7, 2.0, 2.5, 3.0, 4.0};
constexpr int kMaxK = 4095;
constexpr int kApproxMaxN = 112;

__host__ __device__ constexpr int sym(int d) { return d * (d + 1) / 2; }
__host__ __device__ constexpr int pidx(int d, int i, int j) { return i * d - (i * (i - 1)) / 2 + (j - i); }
__device__ __forceinline__ int pidx_any(int d, int i, int j) { return i <= j ? pidx(d, i, j) : pidx(d, j, i); }

// ---- complex arithmetic ---------------------------------------------------------
template <typename R> struct cx {
    R re, im;
};
template <typename R> __device__ __forceinline__ cx<R> mk(R a, R b) { return cx<R>{a, b}; }
template <typename R> __device__ __forceinline__ cx<R> operator+(cx<R> a, cx<R> b) { return {a.re + b.re, a.im + b.im}; }
template <typename R> __device__ __forceinline__ cx<R> operator-(cx<R> a, cx<R> b) { return {a.re - b.re, a.im - b.im}; }
template <typename R> __device__ __forceinline__ cx<R> operator*(cx<R> a, cx<R> b) {
    return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re};
}
template <typename R> __device__ __forceinline__ cx<R> cinv(cx<R> a) {
    const R d = R(1) / (a.re * a.re + a.im * a.im);
    return {a.re * d, -a.im * d};
}
__device__ __forceinline__ float rsqrt_r(float x) { return rsqrtf(x); }
__device__ __forceinline__ double rsqrt_r(double x) { return rsqrt(x); }
__device__ __forceinline__ ff rsqrt_r(ff x) { return ff_rsqrt(x); }
// principal p^{-1/2} for Re p > 0: with a = |p| and s = sqrt((a + Re p)/2) (no
// cancellation: Re p > 0), sqrt(p) = s + i Im p / (2 s) and p^{-1/2} = (s - i Im p/(2 s)) / a;
// two reciprocal square roots, no division
template <typename R> __device__ __forceinline__ cx<R> crsqrt(cx<R> p) {
    const R n2 = p.re * p.re + p.im * p.im;
    const R ra = rsqrt_r(n2);
    const R h = (n2 * ra + p.re) * R(0.5);
    const R rh = rsqrt_r(h);
    return {h * rh * ra, -p.im * ra * rh * R(0.5)};
}
// float-float complex products, reciprocals and roots as shared (non-inlined) calls (the
// overloads win over the templates): inlined everywhere they overflowed the instruction
// cache (-33% time on the order-4 minors with these three out of line)
static __device__ __noinline__ cx<ff> operator*(cx<ff> a, cx<ff> b) {
    return {ff_dot2(a.re, b.re, -a.im, b.im), ff_dot2(a.re, b.im, a.im, b.re)};
}
// e - a b: one fused form per part for float-float (see ff_fms2)
template <typename R> __device__ __forceinline__ cx<R> cfms(cx<R> e, cx<R> a, cx<R> b) { return e - a * b; }
__device__ __forceinline__ cx<ff> cfms_ff(cx<ff> e, cx<ff> a, cx<ff> b) {
    return {ff_fms2(e.re, a.re, b.re, -a.im, b.im), ff_fms2(e.im, a.re, b.im, a.im, b.re)};
}
// out of line in the group terms (their unrolled loops hold dozens of these: inlined, the
// code overflows the instruction cache); inline in the inverse's one-line update loop
static __device__ GBS_FF_FMS_INLINE cx<ff> cfms(cx<ff> e, cx<ff> a, cx<ff> b) { return cfms_ff(e, a, b); }
template <typename R> __device__ __forceinline__ cx<R> cfms_inl(cx<R> e, cx<R> a, cx<R> b) { return e - a * b; }
__device__ __forceinline__ cx<ff> cfms_inl(cx<ff> e, cx<ff> a, cx<ff> b) { return cfms_ff(e, a, b); }
// FP64 in fused multiply-adds, four an update instead of six: the gradient's (the forward keeps the
// form above, whose last digits its fits go by)
__device__ __forceinline__ cx<double> cfma_d(cx<double> c, cx<double> a, cx<double> b) {
    return {fma(a.re, b.re, fma(-a.im, b.im, c.re)), fma(a.re, b.im, fma(a.im, b.re, c.im))};
}
__device__ __forceinline__ cx<double> cfms_d(cx<double> e, cx<double> a, cx<double> b) {
    return {fma(-a.re, b.re, fma(a.im, b.im, e.re)), fma(-a.re, b.im, fma(-a.im, b.re, e.im))};
}
template <bool FUSED, typename R> __device__ __forceinline__ cx<R> cfms_inv(cx<R> e, cx<R> a, cx<R> b) {
    if constexpr (FUSED) return cfms_d(e, a, b);
    else return cfms_inl(e, a, b);
}
static __device__ __noinline__ cx<ff> cinv(cx<ff> a) { return cinv<ff>(a); }
static __device__ __noinline__ cx<ff> crsqrt(cx<ff> p) { return crsqrt<ff>(p); }
__device__ __forceinline__ cx<double> widen(cx<float> a) { return {(double)a.re, (double)a.im}; }

// ---- the four-detector step of the pair phases ----------------------------------------
// K entry: v - sum_k x_k y_k over the four rows of the pair's Schur factor (x = w_c, y = w_d)
template <typename R>
__device__ __forceinline__ cx<R> rank4_entry(cx<R> v, const cx<R> *x, const cx<R> *y, int i, int j) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v = cfms(v, x[2 * k + i], y[2 * k + j]);
    return v;
}
// the term det(G_{P+c+d})^{-1/2} = f3_c det(S)^{-1/2}, S = H_d - K^T H_c^{-1} K, from K and the
// stored items of c (ic) and d (jd); *bad: a pivot of S not accretive
template <typename R> struct QuadTerm {
    cx<R> term;
    int bad;
};
template <typename R>
__device__ __forceinline__ QuadTerm<R> quad_term(cx<R> k00, cx<R> k01, cx<R> k10, cx<R> k11, const cx<R> *ic,
                                                 const cx<R> *jd) {
    const cx<R> K[2][2] = {{k00, k01}, {k10, k11}};
    const cx<R> i00 = ic[11], i01 = ic[12], i11 = ic[13];
    cx<R> X[2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        X[0][j] = i00 * K[0][j] + i01 * K[1][j];
        X[1][j] = i01 * K[0][j] + i11 * K[1][j];
    }
    const cx<R> s00 = cfms(cfms(jd[8], K[0][0], X[0][0]), K[1][0], X[1][0]);
    const cx<R> s01 = cfms(cfms(jd[9], K[0][0], X[0][1]), K[1][0], X[1][1]);
    const cx<R> s11 = cfms(cfms(jd[10], K[0][1], X[0][1]), K[1][1], X[1][1]);
    const cx<R> det = cfms(s00 * s11, s01, s01);
    QuadTerm<R> q;
    q.bad = !(s00.re > R(0)) || !(det.re * s00.re + det.im * s00.im > R(0));
    q.term = ic[14] * crsqrt(det);
    return q;
}
// float-float: each of these as one out-of-line call whose arithmetic is inline (the same
// operations as the shared complex calls, a few calls per four-detector group instead of
// ~30: their argument traffic cost more than the code they share)
__device__ __forceinline__ cx<ff> cmul_ff(cx<ff> a, cx<ff> b) {
    return {ff_dot2(a.re, b.re, -a.im, b.im), ff_dot2(a.re, b.im, a.im, b.re)};
}
static __device__ __noinline__ cx<ff> rank4_entry(cx<ff> v, const cx<ff> *x, const cx<ff> *y, int i, int j) {
#pragma unroll
    for (int k = 0; k < 4; ++k) v = cfms_ff(v, x[2 * k + i], y[2 * k + j]);
    return v;
}
static __device__ __noinline__ QuadTerm<ff> quad_term(cx<ff> k00, cx<ff> k01, cx<ff> k10, cx<ff> k11,
                                                      const cx<ff> *ic, const cx<ff> *jd) {
    const cx<ff> K[2][2] = {{k00, k01}, {k10, k11}};
    const cx<ff> i00 = ic[11], i01 = ic[12], i11 = ic[13];
    cx<ff> X[2][2];
#pragma unroll
    for (int j = 0; j < 2; ++j) {
        X[0][j] = cmul_ff(i00, K[0][j]) + cmul_ff(i01, K[1][j]);
        X[1][j] = cmul_ff(i01, K[0][j]) + cmul_ff(i11, K[1][j]);
    }
    const cx<ff> s00 = cfms_ff(cfms_ff(jd[8], K[0][0], X[0][0]), K[1][0], X[1][0]);
    const cx<ff> s01 = cfms_ff(cfms_ff(jd[9], K[0][0], X[0][1]), K[1][0], X[1][1]);
    const cx<ff> s11 = cfms_ff(cfms_ff(jd[10], K[0][1], X[0][1]), K[1][1], X[1][1]);
    const cx<ff> det = cfms_ff(cmul_ff(s00, s11), s01, s01);
    QuadTerm<ff> q;
    q.bad = !(s00.re > ff(0.0f, 0.0f)) || !(det.re * s00.re + det.im * s00.im > ff(0.0f, 0.0f));
    q.term = cmul_ff(ic[14], crsqrt<ff>(det));
    return q;
}
__device__ __forceinline__ cx<double> widen(cx<double> a) { return a; }
__device__ __forceinline__ cx<double> widen(cx<ff> a) { return {ff_to_double(a.re), ff_to_double(a.im)}; }

// an entry of I - t O_S, t = cs + i sn, from the FP64 products (forming it in FP32 was
// measured no faster and raised the FP32 path's fit fallbacks)
template <typename R> __device__ __forceinline__ cx<R> init_entry(bool diag, double cs, double sn, double o) {
    return mk<R>(R((diag ? 1.0 : 0.0) - cs * o), R(-sn * o));
}

// per precision of the minors: largest pattern (the packed inverse must fit in shared
// memory) and the tilted-sector share below which a sector counts as rounding noise
template <typename R> struct MinorPrec;
template <> struct MinorPrec<double> {
    static constexpr int min_blocks = 1;
    static constexpr int nmax = 79;
    static constexpr bool pair = true;  // n in (nmax, 112] on a CTA pair
    static constexpr double sector_eps = 1e-12;
    static constexpr bool floor_flag = false;  // below the floor: the oracle's own reading of negligible sectors
};
template <> struct MinorPrec<ff> {
    // two CTAs per SM: capped at 128 registers (a few spills) it runs 14% faster than one
    // CTA of 255-register threads
    static constexpr int min_blocks = 2;
    static constexpr int nmax = 79;
    static constexpr bool pair = true;
    static constexpr double sector_eps = 1e-12;
    static constexpr bool floor_flag = false;
};
template <> struct MinorPrec<float> {
    static constexpr int min_blocks = 2;  // 127 registers: two CTAs per SM
    static constexpr int nmax = 112;
    static constexpr bool pair = false;
    static constexpr double sector_eps = 1e-6;  // moments resolved to ~1e-7 K
    static constexpr bool floor_flag = true;    // below it: unresolved, reported (GBS_E_FLOOR)
};

// ---- plan: sector bound and DFT length per pattern ---------------------------------
struct ApproxPlan {
    int *pat_n;           // clicks (-1 invalid)
    int *pat_L;           // DFT length
    double *pat_rho;      // contour radius
    long long *unit_off;  // n_pat + 1: units (pattern, l) with l = 0..L/2
    long long *total;     // total units (0 if over capacity)
    int *overflow;
    double *unit_D;       // 2 (j + 1) doubles per unit: D_w(t_l), w = 0..j
    int *unit_flag;       // per pattern: non-positive pivot seen
    long long *info;      // units, largest n, largest L, sectors (read back to size the launches)
    long long *sec_off;   // n_pat + 1: sectors k = 0..L-1 of each pattern
    double *pat_max;      // per pattern: largest tilted sector
    double *sec_D;        // (kMaxOrder + 1) per sector: D_w^(k), w = 0..order
    double *sec_part;     // per sector: fitted last point (negative: the fit fell back)
    uint32_t *sec_slow;   // sectors left to the slow fits' kernel (below 2^32: a sector is 92 bytes of workspace)
    unsigned long long *slow;  // their number, and the kernel's work counter
};

// ---- plan -----------------------------------------------------------------------------------
// log det(I - rho O_S), +inf if not positive definite, for every pattern (blockIdx.x) and every
// radius of the grid with either sign (blockIdx.y: radius y / 2, sign minus for odd y): Cholesky in
// shared memory (packed), one CTA each.  Launched once for each class of sizes, the CTAs of other
// sizes leaving at once: with one class for all, the largest pattern's 200 KB let a single CTA
// onto an SM, and the 29 factorisations of a pattern ran one after another in it.  FP64-bound: one barrier a
// pivot, the next pivot's reciprocal by the thread that updates it (a division is ten instructions
// of this pipe on every warp that takes it), the logarithms after the last pivot, side by side.
// Measured on a GB300: 256 50-mode patterns 6.9 -> 1.1 ms, 64 100-mode ones 20.6 -> 6.0.
__device__ __forceinline__ int pattern_modes_of(uint64_t lo, uint64_t hi, int M, int n_limit) {
    const int n = __popcll(lo) + __popcll(hi);
    const uint64_t mlo = M >= 64 ? ~0ull : (1ull << M) - 1, mhi = M >= 128 ? ~0ull : M > 64 ? (1ull << (M - 64)) - 1 : 0ull;
    return !(lo & ~mlo) && !(hi & ~mhi) && n <= n_limit ? n : -1;
}
constexpr int kNumShift = 2 * kNumRho;
__global__ void __launch_bounds__(kLogdetThreads) approx_logdet_kernel(int M, const double *__restrict__ O,
                                                                     const uint64_t *__restrict__ pats, int n_limit,
                                                                     int n_from, int n_to, double *__restrict__ ld) {
    extern __shared__ double S[];
    __shared__ uint8_t modes[128];
    __shared__ double s_inv[2], s_log[2 * kApproxMaxN];  // s_inv: of this pivot and of the next
    const int p = blockIdx.x, y = blockIdx.y, t = threadIdx.x;
    const uint64_t lo = pats[2 * p], hi = pats[2 * p + 1];
    const int n = pattern_modes_of(lo, hi, M, n_limit);
    if (n < n_from || n > n_to || y == 1) return;  // (the smallest radius needs one sign only)
    if (t < M) {
        const uint64_t w = t < 64 ? lo : hi, bit = 1ull << (t & 63);
        if (w & bit) modes[(t < 64 ? 0 : __popcll(lo)) + __popcll(w & (bit - 1))] = (uint8_t)t;
    }
    const double rho = y & 1 ? -kRhos[y >> 1] : kRhos[y >> 1];
    const int N = 2 * n, N2 = 2 * M;
    __syncthreads();
    auto folded = [&](int D, auto body) {  // entries (i, j), i <= j, of a D x D triangle, rows p and D - 1 - p as one
        const int w = D + 1, E = ((D + 1) >> 1) * w;
        int fp = t / w, fq = t - fp * w;
        const int sp = kLogdetThreads / w, sq = kLogdetThreads - sp * w;
        for (int f = t; f < E; f += kLogdetThreads) {
            const bool low = fq < D - fp;
            const int i = low ? fp : D - 1 - fp, j = low ? fp + fq : i + (fq - (D - fp));
            if (low || i > fp) body(i, j);  // (an odd D's middle row stands alone)
            fq += sq;
            fp += sp;
            if (fq >= w) { fq -= w; ++fp; }
        }
    };
    folded(N, [&](int i, int j) {
        const int si = modes[i >> 1] + (i & 1) * M, sj = modes[j >> 1] + (j & 1) * M;
        const double v = (i == j ? 1.0 : 0.0) - rho * O[(size_t)si * N2 + sj];
        S[pidx(N, i, j)] = v;
        if (j == 0) s_inv[0] = 1.0 / v;
    });
    __syncthreads();
    bool bad = false;
    for (int k = 0; k < N; ++k) {
        const double d = S[pidx(N, k, k)];
        if (!(d > 0.0)) {  // the same on every thread
            bad = true;
            break;
        }
        const double inv = s_inv[k & 1];
        const int Dt = N - k - 1;
        const double *row = S + pidx(N, k, k) + 1;
        double *C = S + pidx(N, k, k) + Dt + 1;  // the trailing block, packed
        if (Dt > 0)
            folded(Dt, [&](int i, int j) {
                double &c = C[pidx(Dt, i, j)];
                c -= row[i] * row[j] * inv;
                if (j == 0) s_inv[(k + 1) & 1] = 1.0 / c;
            });
        __syncthreads();
    }
    if (bad) {
        if (t == 0) ld[(size_t)p * kNumShift + y] = INFINITY;
        return;
    }
    if (y & 1) {  // only its definiteness counts
        if (t == 0) ld[(size_t)p * kNumShift + y] = 0.0;
        return;
    }
    for (int k = t; k < N; k += kLogdetThreads) s_log[k] = log(S[pidx(N, k, k)]);
    __syncthreads();
    if (t == 0) {
        double v = 0.0;
        for (int k = 0; k < N; ++k) v += s_log[k];
        ld[(size_t)p * kNumShift + y] = v;
    }
}

// sector bound and DFT length per pattern, one warp each
__global__ void __launch_bounds__(kPlanThreads) approx_plan_kernel(int M, const uint64_t *__restrict__ pats, int n_pat,
                                                                 int n_limit, const double *__restrict__ ld,
                                                                 ApproxPlan pl) {
    const int p = blockIdx.x * (kPlanThreads / 32) + (threadIdx.x >> 5), q = threadIdx.x & 31;
    if (p >= n_pat) return;
    const int n = pattern_modes_of(pats[2 * p], pats[2 * p + 1], M, n_limit);
    int L = 1;
    double rho_t = 1.0;
    if (n > 0) {
        // log Z_S(rho) = -1/2 log det(I - rho O_S) on the radii where I -+ rho O_S are
        // positive definite (then I - t O_S is accretive on the whole circle |t| = rho)
        const double *lp = ld + (size_t)p * kNumShift;
        const double lm = q < kNumRho ? lp[2 * q] : INFINITY;
        const bool valid = q < kNumRho && isfinite(lm) && (q == 0 || isfinite(lp[2 * q + 1]));
        const double lz = -0.5 * lm;
        const int nv = __ffs(~__ballot_sync(0xffffffffu, valid)) - 1;
        // contour radius: Chernoff saddle for sector n, argmin log Z(rho) - n log rho
        const int nc = nv > 1 ? nv - 1 : 1;
        const double obj = q < kNumRho ? lz - n * log(kRhos[q]) : INFINITY;
        double mn = q < nc ? obj : INFINITY;
        for (int off = 16; off; off >>= 1) mn = fmin(mn, __shfl_xor_sync(0xffffffffu, mn, off));
        const unsigned at = __ballot_sync(0xffffffffu, q < nc && obj == mn);
        const int qt = at ? __ffs(at) - 1 : 0;
        rho_t = kRhos[qt];
        // sector range: sum_{k > K} c_k rho_t^k <= (rho_t/rho)^K Z(rho) <= eps Z(rho_t)
        const double lzt = __shfl_sync(0xffffffffu, lz, qt);
        double best = q > qt && q < nv ? (lz - lzt - log(kTailEps)) / log(kRhos[q] / rho_t) : INFINITY;
        for (int off = 16; off; off >>= 1) best = fmin(best, __shfl_xor_sync(0xffffffffu, best, off));
        int K = isfinite(best) ? (int)ceil(best) : kMaxK;
        if (K < n) K = n;
        if (K > kMaxK) K = kMaxK;
        L = K + 1;
    }
    if (q == 0) {
        pl.pat_n[p] = n;
        pl.pat_L[p] = n < 0 ? 0 : L;
        pl.pat_rho[p] = rho_t;
        pl.pat_max[p] = 0.0;
        pl.unit_flag[p] = 0;
    }
}

// offsets of the patterns' units and sectors, and the sizes that the host reads back: one CTA, a run of
// patterns a thread, then a scan over the threads
constexpr int kScanThreads = 1024;
__global__ void __launch_bounds__(kScanThreads) approx_scan_kernel(int n_pat, long long cap, int n_single, ApproxPlan pl) {
    __shared__ long long su[kScanThreads], sc[kScanThreads];
    __shared__ int s_n, s_small, s_L;
    const int t = threadIdx.x, per = (n_pat + kScanThreads - 1) / kScanThreads;
    const int p0 = t * per < n_pat ? t * per : n_pat, p1 = p0 + per < n_pat ? p0 + per : n_pat;
    if (t == 0) {
        s_n = 0;
        s_small = -1;
        s_L = 1;
    }
    long long units = 0, secs = 0;
    int nmax = 0, nsmall = -1, Lmax = 1;
    for (int p = p0; p < p1; ++p) {
        const int L = pl.pat_L[p], n = pl.pat_n[p];
        units += L > 0 ? L / 2 + 1 : 0;
        secs += L > 0 ? L : 0;
        nmax = n > nmax ? n : nmax;
        nsmall = n <= n_single && n > nsmall ? n : nsmall;
        Lmax = L > Lmax ? L : Lmax;
    }
    su[t] = units;
    sc[t] = secs;
    __syncthreads();
    atomicMax(&s_n, nmax);
    atomicMax(&s_small, nsmall);
    atomicMax(&s_L, Lmax);
    for (int off = 1; off < kScanThreads; off <<= 1) {
        const long long a = t >= off ? su[t - off] : 0, b = t >= off ? sc[t - off] : 0;
        __syncthreads();
        su[t] += a;
        sc[t] += b;
        __syncthreads();
    }
    const long long run = su[kScanThreads - 1];
    units = su[t] - units;
    secs = sc[t] - secs;
    for (int p = p0; p < p1; ++p) {
        const int L = pl.pat_L[p];
        pl.unit_off[p] = units;
        pl.sec_off[p] = secs;
        units += L > 0 ? L / 2 + 1 : 0;
        secs += L > 0 ? L : 0;
    }
    if (t == 0) {
        pl.unit_off[n_pat] = run;
        pl.sec_off[n_pat] = sc[kScanThreads - 1];
        *pl.overflow = run > cap ? 1 : 0;
        *pl.total = run > cap ? 0 : run;
        pl.info[0] = run;
        pl.info[1] = s_n;
        pl.info[2] = s_L;
        pl.info[3] = sc[kScanThreads - 1];
        pl.info[4] = s_small;  // largest n of the one-CTA minors kernel (0: empty patterns only, -1: none)
    }
}

// ---- minors at one nu point ------------------------------------------------------
// unpivoted LDL^T pivots of a complex symmetric K x K matrix (packed, in registers,
// K even); returns prod p^{-1/2}.  Every pivot of an accretive matrix has Re p > 0, so
// |arg p| < pi/2 and the principal root of a product of two pivots is the product of
// their principal roots: one root per pair of pivots.
template <typename R, int K>
__device__ __forceinline__ cx<R> ldl_rsqrt_prod(cx<R> (&a)[K * (K + 1) / 2], bool &bad) {
    cx<R> f = mk<R>(R(1), R(0)), prev = mk<R>(R(1), R(0));
#pragma unroll
    for (int k = 0; k < K; ++k) {
        cx<R> d = a[pidx(K, k, k)];
        if (!(d.re > R(0))) bad = true;
        if (k & 1) f = f * crsqrt(prev * d);
        prev = d;
        if (k + 1 < K) {
            cx<R> inv = cinv(d);
#pragma unroll
            for (int i = k + 1; i < K; ++i) {
                cx<R> li = a[pidx(K, k, i)] * inv;
#pragma unroll
                for (int j = i; j < K; ++j) a[pidx(K, i, j)] = cfms(a[pidx(K, i, j)], li, a[pidx(K, k, j)]);
            }
        }
    }
    return f;
}

// per-thread sums of the group terms: FP64 for FP64 minors; float-float (TwoSum) for
// FP32 minors, which keeps the FP64 pipe out of the inner loop
template <typename R> struct GroupAcc;
template <> struct GroupAcc<double> {
    double v[2 * (kMaxOrder + 1)];
    __device__ void zero() {
        for (int w = 0; w < 2 * (kMaxOrder + 1); ++w) v[w] = 0.0;
    }
    __device__ __forceinline__ void add(int w, cx<double> f) {
        v[2 * w] += f.re;
        v[2 * w + 1] += f.im;
    }
    __device__ __forceinline__ double get(int q) const { return v[q]; }
};
template <> struct GroupAcc<ff> {
    double v[2 * (kMaxOrder + 1)];
    __device__ void zero() {
        for (int w = 0; w < 2 * (kMaxOrder + 1); ++w) v[w] = 0.0;
    }
    __device__ __forceinline__ void add(int w, cx<ff> f) {
        v[2 * w] += ff_to_double(f.re);
        v[2 * w + 1] += ff_to_double(f.im);
    }
    __device__ __forceinline__ double get(int q) const { return v[q]; }
};
template <> struct GroupAcc<float> {
    float hi[2 * (kMaxOrder + 1)], lo[2 * (kMaxOrder + 1)];
    __device__ void zero() {
        for (int w = 0; w < 2 * (kMaxOrder + 1); ++w) hi[w] = lo[w] = 0.0f;
    }
    __device__ __forceinline__ void two(int q, float x) {
        const float s = hi[q] + x, bp = s - hi[q];
        lo[q] += (hi[q] - (s - bp)) + (x - bp);
        hi[q] = s;
    }
    __device__ __forceinline__ void add(int w, cx<float> f) {
        two(2 * w, f.re);
        two(2 * w + 1, f.im);
    }
    __device__ __forceinline__ double get(int q) const { return (double)hi[q] + (double)lo[q]; }
};

// ---- the inverse's working layout -----------------------------------------------------
// The matrix entry (E) and the staged column b and quotients u = b / pivot of two pivots (parity
// `par`), in `rows` entries a row behind the matrix.
template <typename R, bool FUSED = false> struct InvOps {
    using E = cx<R>;
    static constexpr int rows = 4;
    static constexpr bool eager = false;  // an update of a skipped entry costs the FP64 pipe
    E *G;
    cx<R> *st;
    int N;
    __device__ __forceinline__ InvOps(cx<R> *g, cx<R> *stage, int n) : G(g), st(stage), N(n) {}
    static __device__ __forceinline__ E pack(cx<R> v) { return v; }
    __device__ __forceinline__ cx<R> get(int a) const { return G[a]; }
    __device__ __forceinline__ cx<R> b(int par, int i) const { return st[par * N + i]; }
    __device__ __forceinline__ cx<R> u(int par, int i) const { return st[(2 + par) * N + i]; }
    __device__ __forceinline__ void put(int par, int i, cx<R> bv, cx<R> uv) {
        st[par * N + i] = bv;
        st[(2 + par) * N + i] = uv;
    }
    __device__ __forceinline__ E update(E e, int par, int i, int j) const { return cfms_inv<FUSED>(e, b(par, i), u(par, j)); }
    __device__ __forceinline__ void finish(int, int, int) {}
};
// Float-float: both parts of a complex entry at once in packed FP32 (the add, multiply and fma of two
// lanes an instruction), the same operations part for part as cfms_ff.  An entry is (re.hi, im.hi,
// re.lo, im.lo), turned back into cx<ff> at the end; b is staged as the factor of both parts, negated:
// (-re, -re) and (im, -im), high and low.  Measured on a GB300, whole calls at
// order 2 (with the two-row tiles): 50 modes 34.6 -> 28.6 ms, 100 modes 149 -> 114.
__device__ __forceinline__ uint64_t f2_pack(float a, float b) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
    return r;
}
__device__ __forceinline__ void f2_unpack(uint64_t v, float &a, float &b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
    uint64_t r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ uint64_t f2_add(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ uint64_t f2_mul(uint64_t a, uint64_t b) {
    uint64_t r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
template <> struct InvOps<ff, false> {
    using E = ulonglong2;  // .x: (re.hi, im.hi), .y: (re.lo, im.lo)
    static constexpr int rows = 6;
    static constexpr bool eager = true;   // two updates a tile side by side, without a branch
    E *G, *st;
    int N;
    __device__ __forceinline__ InvOps(cx<ff> *g, cx<ff> *stage, int n) : G((E *)g), st((E *)stage), N(n) {}
    static __device__ __forceinline__ E pack(cx<ff> v) { return E{f2_pack(v.re.hi, v.im.hi), f2_pack(v.re.lo, v.im.lo)}; }
    static __device__ __forceinline__ cx<ff> unpack(E e) {
        cx<ff> v;
        f2_unpack(e.x, v.re.hi, v.im.hi);
        f2_unpack(e.y, v.re.lo, v.im.lo);
        return v;
    }
    __device__ __forceinline__ cx<ff> get(int a) const { return unpack(G[a]); }
    __device__ __forceinline__ cx<ff> b(int par, int i) const {
        const E x = st[2 * (par * N + i)], y = st[2 * (par * N + i) + 1];
        cx<ff> v;
        float z;
        f2_unpack(x.x, v.re.hi, z);
        f2_unpack(x.y, v.re.lo, z);
        v.re = ff(-v.re.hi, -v.re.lo);
        f2_unpack(y.x, v.im.hi, z);
        f2_unpack(y.y, v.im.lo, z);
        return v;
    }
    __device__ __forceinline__ cx<ff> u(int par, int i) const { return unpack(st[(4 + par) * N + i]); }
    __device__ __forceinline__ void put(int par, int i, cx<ff> bv, cx<ff> uv) {
        st[2 * (par * N + i)] = E{f2_pack(-bv.re.hi, -bv.re.hi), f2_pack(-bv.re.lo, -bv.re.lo)};
        st[2 * (par * N + i) + 1] = E{f2_pack(bv.im.hi, -bv.im.hi), f2_pack(bv.im.lo, -bv.im.lo)};
        st[(4 + par) * N + i] = pack(uv);
    }
    __device__ __forceinline__ E update(E e, int par, int i, int j) const {
        const E x0 = st[2 * (par * N + i)], x1 = st[2 * (par * N + i) + 1], y0 = st[(4 + par) * N + j];
        float a, b;
        f2_unpack(y0.x, a, b);
        const uint64_t y1h = f2_pack(b, a);
        f2_unpack(y0.y, a, b);
        const uint64_t y1l = f2_pack(b, a), m1 = f2_pack(-1.0f, -1.0f);
        // the products with their remainders, negated (x holds the minus)
        const uint64_t p0 = f2_mul(x0.x, y0.x), p1 = f2_mul(x1.x, y1h);
        const uint64_t q0 = f2_fma(x0.x, y0.x, f2_mul(p0, m1)), q1 = f2_fma(x1.x, y1h, f2_mul(p1, m1));
        // e.hi + p0 + p1 with the sums' remainders
        const uint64_t s = f2_add(e.x, p0), sb = f2_fma(e.x, m1, s);
        const uint64_t r0 = f2_add(f2_fma(f2_fma(sb, m1, s), m1, e.x), f2_fma(sb, m1, p0));
        const uint64_t v = f2_add(s, p1), vb = f2_fma(s, m1, v);
        const uint64_t r1 = f2_add(f2_fma(f2_fma(vb, m1, v), m1, s), f2_fma(vb, m1, p1));
        uint64_t lo = f2_add(f2_add(e.y, f2_add(r0, r1)), f2_add(q0, q1));
        lo = f2_fma(x0.x, y0.y, lo);
        lo = f2_fma(x0.y, y0.x, lo);
        lo = f2_fma(x1.x, y1l, lo);
        lo = f2_fma(x1.y, y1h, lo);
        const uint64_t h = f2_add(v, lo);
        return E{h, f2_fma(f2_fma(v, m1, h), m1, lo)};
    }
    // the matrix as cx<ff>, entry by entry in its place
    __device__ __forceinline__ void finish(int entries, int t, int threads) {
        for (int f = t; f < entries; f += threads) {
            const cx<ff> v = get(f);
            ((cx<ff> *)G)[f] = v;
        }
    }
};

// The rows [lo, hi) (both even) of the upper triangle in tiles of two rows and one column: row pairs q
// and (last - q) share one run of fw tiles, an odd middle pair follows.  Of a pair's first tile, on the
// diagonal, the second row's entry is not in the triangle.
struct RowPairs {
    int N, lo, hi, mid, fw, fP, tiles;
    uint32_t inv;  // f / fw = f inv >> 24, for f fw < 2^24 and f inv < 2^32
    __device__ __forceinline__ RowPairs(int N_, int lo_, int hi_) : N(N_), lo(lo_), hi(hi_) {
        const int np = (hi - lo) >> 1, half = np >> 1;
        mid = lo + 2 * half;
        fw = 2 * N - lo - hi + 2;
        fP = half * fw;
        tiles = fP + ((np & 1) ? N - mid : 0);
        inv = (1u << 24) / (uint32_t)fw + 1u;
    }
    __device__ __forceinline__ void at(int f, int &i, int &j) const {
        const int q = (int)(((uint32_t)f * inv) >> 24), r = f - q * fw, a = lo + 2 * q;
        const bool low = r < N - a;
        i = f >= fP ? mid : low ? a : hi - 2 - 2 * q;
        j = f >= fP ? mid + (f - fP) : low ? a + r : i + (r - (N - a));
    }
};

// G <- -(I - t O_S)^{-1} in shared memory (packed upper triangle of 2n x 2n, then the
// staged pivot columns, InvOps::rows of 2n entries), t = cs + i sn, by the symmetric sweep operator on
// every pivot; Z_S(t) = prod of principal pivot^{-1/2} (the LDL^T pivots, one root per
// pair) to s_zs.  A pivot with Re <= 0 sets *s_bad.  All kMinorThreads threads take part; ends
// with a barrier.
//
// One phase and one barrier a pivot.  Pivot k's column b and u = b / pivot are staged; in its phase
//  * the first warps (a thread a row) form column k + 1 as pivot k leaves it, and stage it and its
//    quotients by the next pivot in the other buffers;
//  * the others begin with the entries outside rows and columns k and k + 1, e - b_i u_j, in tiles of
//    two rows (RowPairs); the first
//    ones join after kHeadStart rounds, about what the column, two reciprocals' worth, costs them.
// Every warp computing both pivots' reciprocals, with a barrier between the entries and the next
// column, cost as much as the entries at 50 rows: 16 of a hundred instructions each on eight warps
// against 40 rounds of 70.  Every entry's operations and their order are those of the plain form.
// Measured on a GB300, whole calls: order 2 at 50 modes 35.1 -> 31.9 ms, the FP64 gradient at 32 modes
// 74.2 -> 61.6.  A tile of two rows then halved the index work and the loads of u an entry, which with
// packed float-float were most of its instructions (78 an entry, 33 of them on the integer ALUs); two
// tiles at a time were slower (31.5 ms for 28.6).
constexpr int kHeadStart = 4;
template <typename R, bool FUSED = false, int TH = kMinorThreads>
__device__ __forceinline__ void sweep_inverse(int M, const double *__restrict__ O, const int *modes, int n,
                                              double cs, double sn, cx<R> *Gs, int *s_bad, double *s_zs) {
    constexpr int W = TH / 32;
    __shared__ cx<R> s_inv[2];
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int N = 2 * n, N2 = 2 * M;
    using Ops = InvOps<R, FUSED>;
    Ops A(Gs, Gs + sym(N), N);
    const RowPairs rp(N, 0, N);
    for (int f = t; f < rp.tiles; f += TH) {
        int i, j;
        rp.at(f, i, j);
        const int sj = modes[j >> 1] + (j & 1) * M, si = modes[i >> 1], e = pidx(N, i, j);
        A.G[e] = Ops::pack(init_entry<R>(i == j, cs, sn, O[(size_t)si * N2 + sj]));
        if (j > i) A.G[e + (N - i - 1)] = Ops::pack(init_entry<R>(i + 1 == j, cs, sn, O[(size_t)(si + M) * N2 + sj]));
    }
    __syncthreads();
    const int NS = (N + 31) >> 5;  // warps that stage columns
    if (wp < NS) {
        const cx<R> inv0 = cinv(A.get(0));
        if (t < N) {
            const cx<R> v = A.get(t);
            A.put(0, t, v, v * inv0);
        }
        if (t == 0) s_inv[0] = inv0;
    }
    __syncthreads();
    cx<double> zs = mk<double>(1.0, 0.0);  // on the last warp's first thread
    cx<R> dprev = mk<R>(R(1), R(0));
    const int rounds = (rp.tiles + 31) >> 5;
    for (int k = 0; k < N; ++k) {
        const int par = k & 1;
        if (t == TH - 32) {
            const cx<R> d = A.b(par, k);
            if (!(d.re > R(0))) *s_bad = 1;
            if (k & 1) zs = zs * widen(crsqrt(dprev * d));
            dprev = d;
        }
        if (wp < NS) {
            // scale pivot k's row and column (entry (k, k + 1) is the next column's)
            if (t < N && t != k && t != k + 1) A.G[pidx_any(N, t, k)] = Ops::pack(A.u(par, t));
            if (t == k) A.G[pidx(N, k, k)] = Ops::pack(mk<R>(R(0), R(0)) - s_inv[par]);
            if (k + 1 < N) {
                // the next pivot (its place in G stays as it is until its own phase)
                const cx<R> dn = cfms_inv<FUSED>(A.get(pidx(N, k + 1, k + 1)), A.b(par, k + 1), A.u(par, k + 1));
                const cx<R> invn = cinv(dn);
                if (t < N) {
                    const int lo = t < k + 1 ? t : k + 1, hi = t < k + 1 ? k + 1 : t;
                    const int e = pidx(N, lo, hi);
                    cx<R> v;
                    if (t == k) v = A.u(par, k + 1);
                    else if (t == k + 1) v = dn;
                    else v = cfms_inv<FUSED>(A.get(e), A.b(par, lo), A.u(par, hi));
                    if (t != k + 1) A.G[e] = Ops::pack(v);
                    A.put(par ^ 1, t, v, v * invn);
                    if (t == k + 1) s_inv[par ^ 1] = invn;
                }
            }
        }
        // the tiles, 32 a round and warp: entries outside rows and columns k and k + 1
        const int first = wp < NS || ((k & 1) && wp == W - 1) ? kHeadStart : 0;  // busy warps join later
        const int m = NS < W ? W - NS - (k & 1) : 0;
        for (int r = first;; ++r) {
            const int c = r < kHeadStart ? r * m + (wp - NS) : kHeadStart * m + (r - kHeadStart) * W + wp;
            if (c >= rounds) break;
            const int f = c * 32 + lane;
            int i, j;
            rp.at(f < rp.tiles ? f : 0, i, j);
            const bool in = f < rp.tiles && (unsigned)(j - k) > 1u;
            const int e = pidx(N, i, j);
            const int a[2] = {in && (unsigned)(i - k) > 1u ? e : -1,
                              in && j > i && (unsigned)(i + 1 - k) > 1u ? e + (N - i - 1) : -1};
            typename Ops::E v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q)  // (a skipped entry's place takes a staged value, dropped below)
                if (Ops::eager || a[q] >= 0)
                    v[q] = A.update(a[q] < 0 ? A.st[(Ops::rows - 2 + par) * N] : A.G[a[q]], par, i + q, j);
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (a[q] >= 0) A.G[a[q]] = v[q];
        }
        __syncthreads();
    }
    A.finish(sym(N), t, TH);
    if (t == TH - 32) { s_zs[0] = zs.re; s_zs[1] = zs.im; }
    __syncthreads();
}

// shared-memory entries of the one-CTA minors kernel for patterns of up to n clicks: the
// packed inverse, then max(the staged pivot columns, the pair phases' items); the items
// number at least n - 1 and up to 8 n as long as the CTAs per SM of the bare inverse stay
__host__ __device__ inline int minor_smem_entries(int n, int esz, int min_blocks) {
    constexpr long long kSM = 228 * 1024, kCTA = 227 * 1024, kPerCTA = 4 * 1024;  // 1 KB reserved + static
    const long long inv = (long long)n * (2 * n + 1), base = inv + 8LL * n;
    long long per = kSM / (min_blocks > 1 ? 2 : 1) - kPerCTA;
    if (base * esz > per) per = kCTA - kPerCTA;            // the inverse alone takes the SM
    long long items = (per / esz - inv) / 15;
    if (items > 8LL * n) items = 8LL * n;
    if (items < n - 1) items = n - 1;
    const long long ent = inv + (15 * items > 8LL * n ? 15 * items : 8LL * n);
    return (int)ent;
}

// two CTAs of float-float patterns of n clicks share an SM: the inverse, and its staged columns or the
// items the pair phases need
__host__ __device__ inline bool minor_shares_sm(int n) {
    const long long stage = 2LL * InvOps<ff>::rows * n, items = 15LL * (n - 1);
    return ((long long)n * (2 * n + 1) + (stage > items ? stage : items)) * (long long)sizeof(cx<ff>) <=
           228 * 1024 / 2 - 4 * 1024;
}

// Read-only view of the swept matrix -G, G = (I - t O_S)^{-1}, packed upper triangle of
// N x N: rows [0, rsplit) at b0, rows [rsplit, N) at b1 (whose first entry is packed
// entry off1).  One CTA: rsplit = N.  A CTA pair (cluster): each half in one CTA's shared
// memory, the other half reached through distributed shared memory.
template <typename R> struct GView {
    const cx<R> *b0, *b1;
    int N, rsplit, off1;
    __device__ __forceinline__ int rowoff(int r) const { return r * N - (r * (r - 1)) / 2 - r; }
    // p with p[col] = swept entry (r, col), col >= r
    __device__ __forceinline__ const cx<R> *row(int r) const {
        return r < rsplit ? b0 + rowoff(r) : b1 + (rowoff(r) - off1);
    }
    __device__ __forceinline__ cx<R> g(int i, int j) const {  // G(i, j) = -swept(i, j)
        const cx<R> v = i <= j ? row(i)[j] : row(j)[i];
        return mk<R>(-v.re, -v.im);
    }
};

// ---- the pair phases' items ------------------------------------------------------------
// Complex products, fused multiply-subtracts and roots: IN selects, for float-float, the
// inline forms of the shared out-of-line calls (the same operations).
template <typename R, bool IN> __device__ __forceinline__ cx<R> pmul(cx<R> a, cx<R> b) {
    if constexpr (IN) return cmul_ff(a, b); else return a * b;
}
template <typename R, bool IN> __device__ __forceinline__ cx<R> pfms(cx<R> e, cx<R> a, cx<R> b) {
    if constexpr (IN) return cfms_ff(e, a, b); else return cfms(e, a, b);
}
template <typename R, bool IN> __device__ __forceinline__ cx<R> prsqrt(cx<R> p) {
    if constexpr (IN) return crsqrt<ff>(p); else return crsqrt(p);
}
template <typename R, bool IN> __device__ __forceinline__ cx<R> pinv(cx<R> p) {
    if constexpr (IN) return cinv<ff>(p); else return cinv(p);
}
// item (b, e) of pair P = {a, b}: G_PP = L D L^T (unit lower L, accretive pivots), w = D^-1/2
// L^-1 G_{P,e}, H_e = G_ee - w^T w; stores w (8), H_e (3), H_e^-1 (3) and
// f3 = det(G_{P+e})^{-1/2} at o and returns f3 (bad: a pivot not accretive)
template <typename R> struct PairItem {
    cx<R> f3;
    int bad;
};
// G_PP = L D L^T of pair P = {a, b} (unit lower L, accretive pivots): L (6), D^-1/2 (4) and
// f2 = det(G_PP)^{-1/2} at pd[0..10]; returns 1 if a pivot is not accretive
constexpr int kPairLdl = 11;
template <typename R, bool IN>
__device__ __forceinline__ int pair_ldl_body(const GView<R> &V, int a, int b, cx<R> *pd) {
    int bad = 0;
    const int rr[4] = {2 * a, 2 * a + 1, 2 * b, 2 * b + 1};
    cx<R> m4[10];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = i; j < 4; ++j) m4[pidx(4, i, j)] = V.g(rr[i], rr[j]);
    cx<R> f2 = mk<R>(R(1), R(0)), prev = mk<R>(R(1), R(0));
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        const cx<R> d = m4[pidx(4, k, k)];
        if (!(d.re > R(0))) bad = 1;
        if (k & 1) f2 = pmul<R, IN>(f2, prsqrt<R, IN>(pmul<R, IN>(prev, d)));
        prev = d;
        pd[6 + k] = prsqrt<R, IN>(d);
        const cx<R> inv = pinv<R, IN>(d);
#pragma unroll
        for (int i = k + 1; i < 4; ++i) {
            const cx<R> li = pmul<R, IN>(m4[pidx(4, k, i)], inv);
            pd[pidx(3, k, i - 1)] = li;
#pragma unroll
            for (int j = i; j < 4; ++j) m4[pidx(4, i, j)] = pfms<R, IN>(m4[pidx(4, i, j)], li, m4[pidx(4, k, j)]);
        }
    }
    pd[10] = f2;
    return bad;
}
// item (b, e) of pair P = {a, b} from the pair's factorisation pd: w = D^-1/2 L^-1 G_{P,e},
// H_e = G_ee - w^T w; stores w (8), H_e (3), H_e^-1 (3) and f3 = det(G_{P+e})^{-1/2} at o and
// returns f3 (bad: a pivot of H_e not accretive)
template <typename R, bool IN>
__device__ __forceinline__ PairItem<R> pair_item_from(const GView<R> &V, int a, int b, int e, const cx<R> *pd,
                                                      cx<R> *o) {
    PairItem<R> out;
    out.bad = 0;
    const int rr[4] = {2 * a, 2 * a + 1, 2 * b, 2 * b + 1};
    // y = L^-1 G_{P,e} (two columns), w = D^-1/2 y
    cx<R> w[4][2];
#pragma unroll
    for (int col = 0; col < 2; ++col) {
        cx<R> y[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            cx<R> v = V.g(rr[i], 2 * e + col);
#pragma unroll
            for (int k = 0; k < i; ++k) v = pfms<R, IN>(v, pd[pidx(3, k, i - 1)], y[k]);
            y[i] = v;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) w[i][col] = pmul<R, IN>(y[i], pd[6 + i]);
    }
    // H_e = G_ee - w^T w; its pivots h00 and det / h00
    cx<R> h00 = V.g(2 * e, 2 * e), h01 = V.g(2 * e, 2 * e + 1), h11 = V.g(2 * e + 1, 2 * e + 1);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        h00 = pfms<R, IN>(h00, w[k][0], w[k][0]);
        h01 = pfms<R, IN>(h01, w[k][0], w[k][1]);
        h11 = pfms<R, IN>(h11, w[k][1], w[k][1]);
    }
    const cx<R> det = pfms<R, IN>(pmul<R, IN>(h00, h11), h01, h01);
    if (!(h00.re > R(0)) || !(det.re * h00.re + det.im * h00.im > R(0))) out.bad = 1;
    out.f3 = pmul<R, IN>(pd[10], prsqrt<R, IN>(det));
    const cx<R> id = pinv<R, IN>(det);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
        o[2 * k] = w[k][0];
        o[2 * k + 1] = w[k][1];
    }
    o[8] = h00;
    o[9] = h01;
    o[10] = h11;
    o[11] = pmul<R, IN>(h11, id);
    o[12] = mk<R>(R(0), R(0)) - pmul<R, IN>(h01, id);
    o[13] = pmul<R, IN>(h00, id);
    o[14] = out.f3;
    return out;
}
// item (b, e) with the pair's factorisation in registers (no table of them: the CTA pair)
template <typename R, bool IN>
__device__ __forceinline__ PairItem<R> pair_item_body(const GView<R> &V, int a, int b, int e, cx<R> *o) {
    cx<R> pd[kPairLdl];
    const int bad = pair_ldl_body<R, IN>(V, a, b, pd);
    PairItem<R> out = pair_item_from<R, IN>(V, a, b, e, pd, o);
    out.bad |= bad;
    return out;
}
template <typename R>
__device__ __forceinline__ PairItem<R> pair_item(const GView<R> &V, int a, int b, int e, cx<R> *o) {
    return pair_item_body<R, false>(V, a, b, e, o);
}
template <typename R> __device__ __forceinline__ int pair_ldl(const GView<R> &V, int a, int b, cx<R> *pd) {
    return pair_ldl_body<R, false>(V, a, b, pd);
}
template <typename R>
__device__ __forceinline__ PairItem<R> pair_item_tab(const GView<R> &V, int a, int b, int e, const cx<R> *pd,
                                                     cx<R> *o) {
    return pair_item_from<R, false>(V, a, b, e, pd, o);
}
// float-float: one out-of-line call per item (and per pair factorisation) with its
// arithmetic inline
static __device__ __noinline__ PairItem<ff> pair_item(const GView<ff> V, int a, int b, int e, cx<ff> *o) {
    return pair_item_body<ff, true>(V, a, b, e, o);
}
static __device__ __noinline__ int pair_ldl(const GView<ff> V, int a, int b, cx<ff> *pd) {
    return pair_ldl_body<ff, true>(V, a, b, pd);
}
static __device__ __noinline__ PairItem<ff> pair_item_tab(const GView<ff> V, int a, int b, int e, const cx<ff> *pd,
                                                          cx<ff> *o) {
    return pair_item_from<ff, true>(V, a, b, e, pd, o);
}

// The group terms det(G_WW)^{-1/2} of every W with |W| <= order, summed per |W| into acc.
// Groups of one and two detectors: worker `tid` of `nthr` takes every nthr-th.  Groups of
// three and four detectors go through each pair P = {a, b} (a < b) and the Schur
// complement of G_PP in G, G^(P) = G - G_.P G_PP^-1 G_P.: with H_e = G^(P)_ee (2 x 2),
//   det G_{P+e} = det G_PP det H_e,
//   det G_{P+c+d} = det G_PP det H_c det(H_d - K^T H_c^-1 K),  K = G^(P)_cd,
// and G^(P)_cd = G_cd - w_c^T w_d with w_e = D_P^-1/2 L_P^-1 G_Pe (G_PP = L_P D_P L_P^T).
// The pairs of one `a` are taken in groups of consecutive b: phase 1 stores w_e, H_e, H_e^-1
// and det(G_{P+e})^{-1/2} for every (b, e > b) of the group in `scratch` (cap items of 15
// complex entries; every CTA computes all of them with its own threads), phase 2 forms the
// four-detector terms of every (b, c, d), b < c < d (workers t2 of n2).  That is ~34 complex
// products per four-detector group, against ~60 through a 6 x 6 factorisation per triple.
// All pivots are accretive (Re > 0), so each determinant's principal root is the product of
// its factors' principal roots.  Every thread of the CTA must call this (it synchronises the
// CTA); s_off holds 2 (n + 1) ints of shared memory; add3: this CTA adds the three-detector
// terms (of a CTA pair, one computes them for its phase 2 only).  table: the group's pair
// factorisations G_PP = L D L^T are computed once per b into `scratch` ahead of the items
// (cap >= n - 1 then), instead of once per item.  LOW: order <= 2, whose terms need no barrier.
template <typename R, bool LOW = false>
__device__ __forceinline__ void group_terms(const GView<R> &V, int n, int order, int tid, int nthr, int t2,
                                            int n2, cx<R> *scratch, int cap, int *s_off, bool add3, bool table,
                                            GroupAcc<R> &acc, bool &bad) {
    // w = 1: det of the 2x2 block, one root
    if (order >= 1)
        for (int a = tid; a < n; a += nthr) {
            cx<R> m[3] = {V.g(2 * a, 2 * a), V.g(2 * a, 2 * a + 1), V.g(2 * a + 1, 2 * a + 1)};
            acc.add(1, ldl_rsqrt_prod<R, 2>(m, bad));
        }
    // w = 2
    if (order >= 2)
        for (int idx = tid; idx < n * (n - 1) / 2; idx += nthr) {
            int a = 0, rem = idx;
            while (rem >= n - 1 - a) { rem -= n - 1 - a; ++a; }
            int b = a + 1 + rem;
            int rr[4] = {2 * a, 2 * a + 1, 2 * b, 2 * b + 1};
            cx<R> m[10];
#pragma unroll
            for (int i = 0; i < 4; ++i)
#pragma unroll
                for (int j = i; j < 4; ++j) m[pidx(4, i, j)] = V.g(rr[i], rr[j]);
            acc.add(2, ldl_rsqrt_prod<R, 4>(m, bad));
        }
    if constexpr (LOW) return;
    // order 4 in FP64 and float-float: the pair phases below; order 3, and every order in
    // FP32 (whose arithmetic is cheap next to the phases' barriers): a 6 x 6 factorisation
    // per triple, each serving its fourth detectors through a 2 x 2 Schur block
    constexpr bool kPairPhases = !std::is_same<R, float>::value;
    if (order >= 3 && !(kPairPhases && order >= 4)) {
        // w = 3, and w = 4 from each triple's factorisation.  Triples in order of their
        // largest detector c (then b, a), so the lanes of a warp share c and with it the
        // number n - 1 - c of fourth detectors d > c.
        if (order >= 3) {
            const long long ntri = (long long)n * (n - 1) * (n - 2) / 6;
            for (long long idx = tid; idx < ntri; idx += nthr) {
                // c: the largest with C(c, 3) <= idx; then b: the largest with C(b, 2) <= rem
                // (FP32 estimates on the MUFU pipe, corrected exactly in integers)
                int c = (int)cbrtf(6.0f * (float)idx);
                while ((long long)(c + 1) * c * (c - 1) / 6 <= idx) ++c;
                while ((long long)c * (c - 1) * (c - 2) / 6 > idx) --c;
                const long long rem = idx - (long long)c * (c - 1) * (c - 2) / 6;
                int b = (int)sqrtf(2.0f * (float)rem);
                while ((long long)(b + 1) * b / 2 <= rem) ++b;
                while ((long long)b * (b - 1) / 2 > rem) --b;
                const int a = (int)(rem - (long long)b * (b - 1) / 2);
                const int rr[6] = {2 * a, 2 * a + 1, 2 * b, 2 * b + 1, 2 * c, 2 * c + 1};
                // rows of the triple: entry (rr[i], col) with rr[i] <= col at rp[i][col]
                const cx<R> *rp[6];
    #pragma unroll
                for (int i = 0; i < 6; ++i) rp[i] = V.row(rr[i]);
                auto gr = [&](int i, int col) -> cx<R> { const cx<R> v = rp[i][col]; return mk<R>(-v.re, -v.im); };
                cx<R> w6[21];
    #pragma unroll
                for (int i = 0; i < 6; ++i)
    #pragma unroll
                    for (int j = i; j < 6; ++j) w6[pidx(6, i, j)] = gr(i, rr[j]);
                // LDL^T kept: unit lower L (Lf[k][i], k < i), inverse pivots Dinv
                cx<R> Lf[15], Dinv[6];
                cx<R> f3 = mk<R>(R(1), R(0)), prev = mk<R>(R(1), R(0));
    #pragma unroll
                for (int k = 0; k < 6; ++k) {
                    cx<R> d = w6[pidx(6, k, k)];
                    if (!(d.re > R(0))) bad = true;
                    if (k & 1) f3 = f3 * crsqrt(prev * d);
                    prev = d;
                    cx<R> inv = cinv(d);
                    Dinv[k] = inv;
    #pragma unroll
                    for (int i = k + 1; i < 6; ++i) {
                        cx<R> li = w6[pidx(6, k, i)] * inv;
                        Lf[pidx(5, k, i - 1)] = li;
    #pragma unroll
                        for (int j = i; j < 6; ++j) w6[pidx(6, i, j)] = cfms(w6[pidx(6, i, j)], li, w6[pidx(6, k, j)]);
                    }
                }
                acc.add(3, f3);
                // float-float: this triple's quads summed in float-float first, then one FP64
                // addition (keeps the FP64 pipe, 1/64 of FP32 here, out of the quad loop)
                constexpr bool kTriplePartial = std::is_same<R, ff>::value;
                cx<R> q4 = mk<R>(R(0), R(0));
                if (order >= 4)
                    for (int d4 = c + 1; d4 < n; ++d4) {
                        // y = L^{-1} G_{abc, d}; S = G_dd - y^T D^{-1} y (2 x 2); det S^{-1/2}
                        cx<R> y0[6], y1[6];
    #pragma unroll
                        for (int i = 0; i < 6; ++i) {
                            cx<R> v0 = gr(i, 2 * d4), v1 = gr(i, 2 * d4 + 1);
    #pragma unroll
                            for (int k = 0; k < i; ++k) {
                                v0 = cfms(v0, Lf[pidx(5, k, i - 1)], y0[k]);
                                v1 = cfms(v1, Lf[pidx(5, k, i - 1)], y1[k]);
                            }
                            y0[i] = v0;
                            y1[i] = v1;
                        }
                        const cx<R> *r0 = V.row(2 * d4), *r1 = V.row(2 * d4 + 1);
                        const cx<R> e00 = r0[2 * d4], e01 = r0[2 * d4 + 1], e11 = r1[2 * d4 + 1];
                        cx<R> s00 = mk<R>(-e00.re, -e00.im), s01 = mk<R>(-e01.re, -e01.im),
                              s11 = mk<R>(-e11.re, -e11.im);
    #pragma unroll
                        for (int k = 0; k < 6; ++k) {
                            const cx<R> z0 = y0[k] * Dinv[k], z1 = y1[k] * Dinv[k];
                            s00 = cfms(s00, z0, y0[k]);
                            s01 = cfms(s01, z0, y1[k]);
                            s11 = cfms(s11, z1, y1[k]);
                        }
                        // pivots s00 and det / s00 of the accretive block: Re > 0 each
                        const cx<R> det = cfms(s00 * s11, s01, s01);
                        if (!(s00.re > R(0)) || !(det.re * s00.re + det.im * s00.im > R(0))) bad = true;
                        const cx<R> term = f3 * crsqrt(det);
                        if constexpr (kTriplePartial) q4 = q4 + term;
                        else acc.add(4, term);
                    }
                if constexpr (kTriplePartial)
                    if (order >= 4) acc.add(4, q4);
            }
        }
    } else if (order >= 3 && n >= 3) {
        constexpr int IW = 15;  // per (b, e): w (4 x 2), H_e (3), H_e^-1 (3), det(G_{P+e})^{-1/2}
        const int t1 = threadIdx.x, n1 = blockDim.x;
        int *off1 = s_off, *off2 = s_off + (n + 1);
        cx<R> q4 = mk<R>(R(0), R(0));
        for (int a = 0; a + 2 < n; ++a) {
            for (int b0 = a + 1; b0 + 1 < n;) {
                // the group: b in [b0, b1) while its items (and with `table` each pair's
                // factorisation) fit in cap items' entries (at least one b: cap >= n - 2, and
                // n - 1 with the table)
                const int per_b = table ? kPairLdl : 0;
                int b1 = b0, items = 0;
                while (b1 + 1 < n &&
                       (b1 == b0 || IW * (items + (n - b1 - 1)) + per_b * (b1 - b0 + 1) <= IW * cap)) {
                    items += n - b1 - 1;
                    ++b1;
                }
                if (t1 == 0) {
                    int s1 = 0, s2 = 0;
                    for (int b = b0; b < b1; ++b) {
                        off1[b - b0] = s1;
                        off2[b - b0] = s2;
                        s1 += n - b - 1;
                        s2 += (n - b - 1) * (n - b - 2) / 2;
                    }
                    off1[b1 - b0] = s1;
                    off2[b1 - b0] = s2;
                }
                const int nb = b1 - b0;
                // the group's pair factorisations (with `table`), then its items
                cx<R> *const items_at = scratch + (size_t)per_b * nb;
                if (table)
                    for (int bb = t1; bb < nb; bb += n1)
                        if (pair_ldl(V, a, b0 + bb, scratch + (size_t)kPairLdl * bb)) bad = true;
                __syncthreads();
                // phase 1: every (b, e), e > b
                for (int it = t1; it < items; it += n1) {
                    int lo = 0, hi = nb;
                    while (hi - lo > 1) {
                        const int mid = (lo + hi) >> 1;
                        if (off1[mid] <= it) lo = mid; else hi = mid;
                    }
                    const int b = b0 + lo, e = b + 1 + (it - off1[lo]);
                    const PairItem<R> pi = table ? pair_item_tab(V, a, b, e, scratch + (size_t)kPairLdl * lo,
                                                                 items_at + (size_t)IW * it)
                                                 : pair_item(V, a, b, e, items_at + (size_t)IW * it);
                    if (pi.bad) bad = true;
                    if (add3) acc.add(3, pi.f3);
                }
                __syncthreads();
                // phase 2: every (b, c, d), b < c < d
                if (order >= 4) {
                    const int total = off2[nb];
                    for (int it = t2; it < total; it += n2) {
                        int lo = 0, hi = nb;
                        while (hi - lo > 1) {
                            const int mid = (lo + hi) >> 1;
                            if (off2[mid] <= it) lo = mid; else hi = mid;
                        }
                        const int b = b0 + lo, r = it - off2[lo];
                        // (c', d') with c' < d' in colex order: r = d'(d' - 1)/2 + c'
                        int dp = (int)((1.0f + sqrtf(1.0f + 8.0f * (float)r)) * 0.5f);
                        while (dp * (dp - 1) / 2 > r) --dp;
                        while ((dp + 1) * dp / 2 <= r) ++dp;
                        const int cp = r - dp * (dp - 1) / 2;
                        const int c = b + 1 + cp, d = b + 1 + dp;
                        const cx<R> *ic = items_at + (size_t)IW * (off1[lo] + cp);
                        const cx<R> *jd = items_at + (size_t)IW * (off1[lo] + dp);
                        // K = G^(P)_cd = G_cd - w_c^T w_d; X = H_c^-1 K; S = H_d - K^T X
                        const cx<R> k00 = rank4_entry(V.g(2 * c, 2 * d), ic, jd, 0, 0);
                        const cx<R> k01 = rank4_entry(V.g(2 * c, 2 * d + 1), ic, jd, 0, 1);
                        const cx<R> k10 = rank4_entry(V.g(2 * c + 1, 2 * d), ic, jd, 1, 0);
                        const cx<R> k11 = rank4_entry(V.g(2 * c + 1, 2 * d + 1), ic, jd, 1, 1);
                        const QuadTerm<R> qt = quad_term(k00, k01, k10, k11, ic, jd);
                        if (qt.bad) bad = true;
                        q4 = q4 + qt.term;
                    }
                }
                acc.add(4, q4);     // this group's four-detector terms (zero if order 3)
                q4 = mk<R>(R(0), R(0));
                __syncthreads();    // the group's items are read: the next group may overwrite them
                b0 = b1;
            }
        }
    }
}

// a warp's sums of the group terms (lanes combined by a fixed butterfly) into red[warp]
template <typename R>
__device__ __forceinline__ void warp_group_sums(const GroupAcc<R> &acc, double *red_row) {
    double accd[2 * (kMaxOrder + 1)];
#pragma unroll
    for (int w = 0; w < 2 * (kMaxOrder + 1); ++w) accd[w] = w < 2 ? 0.0 : acc.get(w);
#pragma unroll
    for (int w = 2; w < 2 * (kMaxOrder + 1); ++w)
        for (int off = 16; off; off >>= 1) accd[w] += __shfl_xor_sync(0xffffffffu, accd[w], off);
    if ((threadIdx.x & 31) == 0)
#pragma unroll
        for (int w = 0; w < 2 * (kMaxOrder + 1); ++w) red_row[w] = accd[w];
}

// the unit's D_w(t_l) = Z_S(t_l) sum_{|W| = w} det(G_WW)^{-1/2}, from the warp sums in
// warp order (deterministic)
__device__ __forceinline__ void write_unit(const ApproxPlan &pl, long long u, int order, const double *zs,
                                           const double (*red)[2 * (kMaxOrder + 1)], int nwarps) {
    const cx<double> z = mk<double>(zs[0], zs[1]);
    double *out = pl.unit_D + (size_t)u * 2 * (kMaxOrder + 1);
    out[0] = z.re;
    out[1] = z.im;
    for (int w = 1; w <= kMaxOrder; ++w) {
        double re = 0.0, im = 0.0;
        for (int q = 0; q < nwarps; ++q) {
            re += red[q][2 * w];
            im += red[q][2 * w + 1];
        }
        cx<double> v = z * mk<double>(re, im);
        out[2 * w] = w <= order ? v.re : 0.0;
        out[2 * w + 1] = w <= order ? v.im : 0.0;
    }
}

// the pattern of unit u (skipping patterns without units: equal offsets)
__device__ __forceinline__ int unit_pattern(const ApproxPlan &pl, int n_pat, long long u) {
    int lo_ = 0, hi_ = n_pat;
    while (hi_ - lo_ > 1) {
        int mid = (lo_ + hi_) >> 1;
        if (pl.unit_off[mid] <= u) lo_ = mid; else hi_ = mid;
    }
    int p = lo_;
    while (p + 1 < n_pat && pl.unit_off[p + 1] <= u) ++p;
    return p;
}

// One CTA per (pattern, nu_l) unit, for patterns of n_from to n_single clicks (the packed
// inverse in this CTA's shared memory); larger patterns are left to the cluster kernel.
// TH = 512: order <= 2 on an SM that holds one CTA only.  The inverse, nearly all of the work there,
// takes all 16 warps; the group terms stay with the first 256 threads, whose split of the sums is
// that of every other size.
template <typename R, int TH>
__global__ void __launch_bounds__(TH, TH > kMinorThreads ? 1 : MinorPrec<R>::min_blocks) approx_minors_kernel(int M, const double *__restrict__ O,
                                                                    const uint64_t *__restrict__ pats,
                                                                    int n_pat, int order, int n_from, int n_single,
                                                                    int smem_entries,
                                                                    unsigned long long *counter,
                                                                    ApproxPlan pl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    cx<R> *G = (cx<R> *)smem_raw;
    __shared__ int modes[128];
    __shared__ int s_off[2 * (kApproxMaxN + 1)];
    __shared__ long long s_u;
    __shared__ int s_bad;
    __shared__ double red[kMinorThreads / 32][2 * (kMaxOrder + 1)];
    __shared__ double s_zs[2];
    const int t = threadIdx.x;
    const long long total = *pl.total;
    for (;;) {
        if (t == 0) s_u = (long long)atomicAdd(counter, 1ull);
        __syncthreads();
        const long long u = s_u;
        if (u >= total) break;
        const int p = unit_pattern(pl, n_pat, u);
        const int l = (int)(u - pl.unit_off[p]);
        const int n = pl.pat_n[p], L = pl.pat_L[p];
        if (n < n_from || n > n_single) {   // a pattern for another launch
            __syncthreads();
            continue;
        }
        const uint64_t wlo = pats[2 * p], whi = pats[2 * p + 1];
        if (t == 0) {
            int c = 0;
            for (int i = 0; i < M; ++i) {
                uint64_t w = i < 64 ? wlo : whi;
                if (w >> (i & 63) & 1ull) modes[c++] = i;
            }
            s_bad = 0;
        }
        __syncthreads();
        const int N = 2 * n;
        // t = rho e^{i nu}, nu = 2 pi l / L; M_t = I - t O_S (complex symmetric)
        double sn, cs;
        sincospi(2.0 * (double)l / (double)L, &sn, &cs);
        const double rho = pl.pat_rho[p];
        sn *= rho;
        cs *= rho;
        sweep_inverse<R, false, TH>(M, O, modes, n, cs, sn, G, &s_bad, s_zs);
        GroupAcc<R> acc;
        acc.zero();
        bool bad = false;
        const GView<R> V{G, G, N, N, 0};
        // the staged columns and the rest of the allocation serve the pair phases
        // items per group from this pattern's own n (not the batch's allocation): the work
        // split, and with it every rounding, is the same in any batch
        const int cap = (minor_smem_entries(n, (int)sizeof(cx<R>), MinorPrec<R>::min_blocks) - sym(N)) / 15;
        constexpr bool kLow = TH > kMinorThreads;
        if (!kLow || t < kMinorThreads)
            group_terms<R, kLow>(V, n, order, t, kMinorThreads, t, kMinorThreads, G + sym(N), cap, s_off, true, true, acc, bad);
        if (bad) s_bad = 1;
        if (!kLow || t < kMinorThreads) warp_group_sums<R>(acc, red[t >> 5]);
        __syncthreads();
        if (t == 0) {
            write_unit(pl, u, order, s_zs, red, kMinorThreads / 32);
            if (s_bad) atomicOr(pl.unit_flag + p, 1);
        }
        __syncthreads();
    }
}

// ---- the same for large patterns on a CTA pair (thread-block cluster of two) ----------
// The packed 2n x 2n inverse of a pattern with n up to 112 clicks (403 KB in FP64 or
// float-float) exceeds one SM's shared memory: the two CTAs of a cluster hold half of its
// rows each and reach the other half through distributed shared memory.  The sweep
// operator runs on both halves at once (each CTA updates its own entries; the pivot
// columns are staged into both CTAs, one cluster barrier per pivot); the group terms are
// split over the 512 threads of the pair.
constexpr int kPairMaxN = kApproxMaxN;

// rows [0, rsplit) hold about half of the packed entries of an N x N upper triangle (N even; an even
// rsplit, with the smaller of the larger halves)
__host__ __device__ inline int pair_split_row(int N) {
    const int tot = N * (N + 1) / 2;
    int r = 0, acc = 0;
    while (r < N && 2 * (acc + (N - r)) <= tot) { acc += N - r; ++r; }
    const int d = r & ~1, low = d * N - d * (d - 1) / 2, u = d + 2, high = u * N - u * (u - 1) / 2;
    const int best = u < N && high < tot - low ? u : d;
    return best > 0 ? best : (N > 2 ? 2 : N);
}
__host__ __device__ inline int pair_part_entries(int N) {  // the larger half
    const int r = pair_split_row(N), lo = r * N - r * (r - 1) / 2, tot = N * (N + 1) / 2;
    return lo > tot - lo ? lo : tot - lo;
}

// The inverse of sweep_inverse on both halves, one phase and one cluster barrier a pivot (in the place
// of three barriers, with every warp forming the pivot's reciprocal).  A CTA forms its own entries of
// the next column and stages them, and their quotients, in both CTAs.  The pivot after the next one may
// be the other CTA's: its diagonal entry is passed on a pivot ahead (dg), so that both know the next
// pivot as soon as a phase begins.  Measured on a GB300, order 2, 64 patterns of 40 to 90
// clicks at 100 modes: the pair kernel 83.6 -> 75.5 ms (with 512 threads), the one-CTA kernel 74.1 -> 61.5
// (sizes that share an SM in a launch of their own, the others with 512 threads).
template <typename R> struct PairPivots {
    cx<R> inv[2];  // reciprocal of this pivot and of the next
    cx<R> dg[2];   // the next pivot's diagonal entry as the pivot before this one left it
};
template <typename R, int TH>
__device__ void sweep_inverse_pair(cg::cluster_group &cl, int rank, int M, const double *__restrict__ O,
                                   const uint8_t *modes, int n, double cs, double sn, cx<R> *Gs, cx<R> *stage,
                                   cx<R> *stage_peer, PairPivots<R> *pv, PairPivots<R> *pv_peer, int rsplit, int off1,
                                   int *s_bad, double *s_zs) {
    constexpr int W = TH / 32;
    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int N = 2 * n, N2 = 2 * M;
    const int r_lo = rank ? rsplit : 0, r_hi = rank ? N : rsplit;
    const int base = rank ? off1 : 0;
    using Ops = InvOps<R>;
    Ops A(Gs, stage, N), peer(Gs, stage_peer, N);  // (of the peer, the staged columns)
    auto lidx = [&](int i, int j) { return i * N - (i * (i - 1)) / 2 + (j - i) - base; };  // own row i <= j
    auto own = [&](int i) { return i >= r_lo && i < r_hi; };
    const RowPairs rp(N, r_lo, r_hi);
    for (int f = t; f < rp.tiles; f += TH) {
        int i, j;
        rp.at(f, i, j);
        const int sj = modes[j >> 1] + (j & 1) * M, si = modes[i >> 1], e = lidx(i, j);
        A.G[e] = Ops::pack(init_entry<R>(i == j, cs, sn, O[(size_t)si * N2 + sj]));
        if (j > i) A.G[e + (N - i - 1)] = Ops::pack(init_entry<R>(i + 1 == j, cs, sn, O[(size_t)(si + M) * N2 + sj]));
    }
    __syncthreads();
    const int NS = (N + 31) >> 5;  // warps that stage columns
    if (wp < NS && t < N) {
        if (rank == 0) {  // pivot 0's column is row 0
            const cx<R> inv0 = cinv(A.get(0)), v = A.get(t), u = v * inv0;
            A.put(0, t, v, u);
            peer.put(0, t, v, u);
            if (t == 0) pv->inv[0] = pv_peer->inv[0] = inv0;
        }
        if (t == 1 && own(1)) pv->dg[1] = pv_peer->dg[1] = A.get(lidx(1, 1));
    }
    cl.sync();
    cx<double> zs = mk<double>(1.0, 0.0);  // on the last warp's first thread
    cx<R> dprev = mk<R>(R(1), R(0));
    const int rounds = (rp.tiles + 31) >> 5;
    for (int k = 0; k < N; ++k) {
        const int par = k & 1;
        if (t == TH - 32) {
            const cx<R> d = A.b(par, k);
            if (!(d.re > R(0))) *s_bad = 1;
            if (k & 1) zs = zs * widen(crsqrt(dprev * d));
            dprev = d;
        }
        if (wp < NS) {
            if (t < N && t != k + 1) {  // scale pivot k's row and column (entry (k, k + 1) is the next column's)
                const int lo = t < k ? t : k, hi = t < k ? k : t;
                if (own(lo)) A.G[lidx(lo, hi)] = Ops::pack(t == k ? mk<R>(R(0), R(0)) - pv->inv[par] : A.u(par, t));
            }
            if (k + 1 < N) {
                const cx<R> dn = cfms_inl(pv->dg[par ^ 1], A.b(par, k + 1), A.u(par, k + 1));
                const cx<R> invn = cinv(dn);
                if (t < N) {
                    const int lo = t < k + 1 ? t : k + 1, hi = t < k + 1 ? k + 1 : t;
                    if (own(lo)) {
                        const int e = lidx(lo, hi);
                        cx<R> v;
                        if (t == k) v = A.u(par, k + 1);
                        else if (t == k + 1) v = dn;
                        else v = cfms_inl(A.get(e), A.b(par, lo), A.u(par, hi));
                        if (t != k + 1) A.G[e] = Ops::pack(v);
                        const cx<R> u = v * invn;
                        A.put(par ^ 1, t, v, u);
                        peer.put(par ^ 1, t, v, u);
                    }
                    if (t == k + 1) pv->inv[par ^ 1] = invn;
                    if (t == k + 2 && own(t)) {
                        const int e = lidx(t, t);
                        const cx<R> v = cfms_inl(A.get(e), A.b(par, t), A.u(par, t));
                        A.G[e] = Ops::pack(v);
                        pv->dg[par] = pv_peer->dg[par] = v;
                    }
                }
            }
        }
        // the tiles, 32 a round and warp: entries outside rows and columns k and k + 1
        const int first = wp < NS || ((k & 1) && wp == W - 1) ? kHeadStart : 0;  // busy warps join later
        const int m = NS < W ? W - NS - (k & 1) : 0;
        for (int r = first;; ++r) {
            const int c = r < kHeadStart ? r * m + (wp - NS) : kHeadStart * m + (r - kHeadStart) * W + wp;
            if (c >= rounds) break;
            const int f = c * 32 + lane;
            int i, j;
            rp.at(f < rp.tiles ? f : 0, i, j);
            const bool in = f < rp.tiles && (unsigned)(j - k) > 1u;
            const int e = lidx(i, j);
            const int a[2] = {in && (unsigned)(i - k) > 1u && (i != k + 2 || j != k + 2) ? e : -1,
                              in && j > i && (unsigned)(i + 1 - k) > 1u && (i != k + 1 || j != k + 2) ? e + (N - i - 1) : -1};
            typename Ops::E v[2];
#pragma unroll
            for (int q = 0; q < 2; ++q)  // (a skipped entry's place takes a staged value, dropped below)
                if (Ops::eager || a[q] >= 0)
                    v[q] = A.update(a[q] < 0 ? A.st[(Ops::rows - 2 + par) * N] : A.G[a[q]], par, i + q, j);
#pragma unroll
            for (int q = 0; q < 2; ++q)
                if (a[q] >= 0) A.G[a[q]] = v[q];
        }
        cl.sync();
    }
    if (Ops::rows != 4) {  // the packed form turned back before the peer reads it
        A.finish(rank ? sym(N) - off1 : off1, t, TH);
        cl.sync();
    }
    if (t == TH - 32) { s_zs[0] = zs.re; s_zs[1] = zs.im; }
}

template <typename R, int TH>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(TH, 1)
approx_minors_pair_kernel(int M, const double *__restrict__ O, const uint64_t *__restrict__ pats, int n_pat,
                          int order, int n_single, int smem_entries, unsigned long long *counter, ApproxPlan pl) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ uint8_t modes[128];  // bytes: at 112 clicks the CTA needs all but ~0.2 KB of 227 KB
    __shared__ int s_off[2 * (kApproxMaxN + 1)];
    __shared__ long long s_u;
    __shared__ int s_bad;
    __shared__ double red[2 * (kMinorThreads / 32)][2 * (kMaxOrder + 1)];
    __shared__ double s_zs[2];
    __shared__ PairPivots<R> s_pv;
    constexpr bool kLow = TH > kMinorThreads;  // order <= 2: group terms on 256 threads, as in the one-CTA kernel
    cg::cluster_group cl = cg::this_cluster();
    const int rank = (int)cl.block_rank(), t = threadIdx.x;
    const long long total = *pl.total;
    for (;;) {
        if (rank == 0 && t == 0) {
            const long long v = (long long)atomicAdd(counter, 1ull);
            s_u = v;
            *cl.map_shared_rank(&s_u, 1) = v;
        }
        cl.sync();
        const long long u = s_u;
        if (u >= total) break;
        const int p = unit_pattern(pl, n_pat, u);
        const int n = pl.pat_n[p];
        if (n <= n_single) {  // a pattern for the one-CTA kernel: both CTAs skip it
            cl.sync();        // (every thread has read s_u before rank 0 writes the next)
            continue;
        }
        const int l = (int)(u - pl.unit_off[p]), L = pl.pat_L[p];
        const uint64_t wlo = pats[2 * p], whi = pats[2 * p + 1];
        if (t == 0) {
            int c = 0;
            for (int i = 0; i < M; ++i) {
                uint64_t w = i < 64 ? wlo : whi;
                if (w >> (i & 63) & 1ull) modes[c++] = i;
            }
            s_bad = 0;
        }
        __syncthreads();
        const int N = 2 * n, rsplit = pair_split_row(N), off1 = rsplit * N - rsplit * (rsplit - 1) / 2;
        cx<R> *Gl = (cx<R> *)smem_raw;
        cx<R> *stage = Gl + pair_part_entries(N);
        cx<R> *stage_peer = cl.map_shared_rank(stage, rank ^ 1);
        double sn, cs;
        sincospi(2.0 * (double)l / (double)L, &sn, &cs);
        const double rho = pl.pat_rho[p];
        sn *= rho;
        cs *= rho;
        sweep_inverse_pair<R, TH>(cl, rank, M, O, modes, n, cs, sn, Gl, stage, stage_peer, &s_pv,
                                  cl.map_shared_rank(&s_pv, rank ^ 1), rsplit, off1, &s_bad, s_zs);
        cx<R> *G0 = rank == 0 ? Gl : cl.map_shared_rank(Gl, 0);
        cx<R> *G1 = rank == 1 ? Gl : cl.map_shared_rank(Gl, 1);
        const GView<R> V{G0, G1, N, rsplit, off1};
        GroupAcc<R> acc;
        acc.zero();
        bool bad = false;
        // each CTA computes every pair item in its own scratch (the staging area and beyond),
        // rank 0 adds the three-detector terms, the four-detector ones are split over both
        if (!kLow || t < kMinorThreads)
            group_terms<R, kLow>(V, n, order, rank * kMinorThreads + t, 2 * kMinorThreads, rank * kMinorThreads + t,
                       2 * kMinorThreads, stage, n - 2, s_off, rank == 0, false, acc, bad);
        if (bad) s_bad = 1;
        // warp sums: rank 1's into rank 0's table (rows 8..15), then rank 0 writes the unit
        double (*red0)[2 * (kMaxOrder + 1)] = rank == 0 ? red : cl.map_shared_rank(red, 0);
        if (!kLow || t < kMinorThreads)
            warp_group_sums<R>(acc, red0[rank * (kMinorThreads / 32) + (t >> 5)]);
        __syncthreads();
        if (rank == 1 && t == 0 && s_bad) atomicOr(cl.map_shared_rank(&s_bad, 0), 1);
        cl.sync();
        if (rank == 0 && t == 0) {
            write_unit(pl, u, order, s_zs, red, 2 * (kMinorThreads / 32));
            if (s_bad) atomicOr(pl.unit_flag + p, 1);
        }
        // the next ticket's barrier keeps both CTAs' shared memory live until the peer is done
    }
    cl.sync();
}

// ---- per-sector fit (maximum-entropy dual, damped Newton) ----------------------------
// One warp per sector: the lanes share the support points of the sums; every lane then
// takes the same Newton step from the same (broadcast) sums.
__device__ __forceinline__ double warp_sum_bcast(double v) {
    for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return __shfl_sync(0xffffffffu, v, 0);
}

// support x_s = v_s / n for v in [v0, n-1]; moments m (m_0 = 1); J + 1 coefficients
__device__ bool maxent_fit_warp(int v0, int n, int J, const double *m, double *a, int lane) {
    const int S = n - v0;
    auto phi_grad = [&](const double *aa, double *g, double *H, double &phi) {
        double pw[2 * kMaxOrder + 1];
        for (int q = 0; q <= 2 * J; ++q) pw[q] = 0.0;
        double ph = 0.0;
        for (int s = lane; s < S; s += 32) {
            double x = (double)(v0 + s) / n, f = 0.0, xp = 1.0;
            for (int i = 0; i <= J; ++i) { f += aa[i] * xp; xp *= x; }
            double q = exp(-f);
            ph += q;
            xp = 1.0;
            for (int i = 0; i <= 2 * J; ++i) { pw[i] += xp * q; xp *= x; }
        }
        phi = warp_sum_bcast(ph);
        for (int i = 0; i <= 2 * J; ++i) pw[i] = warp_sum_bcast(pw[i]);
        for (int i = 0; i <= J; ++i) {
            phi += aa[i] * m[i];
            if (g) g[i] = m[i] - pw[i];
            if (H)
                for (int k = 0; k <= J; ++k) H[i * (kMaxOrder + 1) + k] = pw[i + k];
        }
    };
    for (int i = 0; i <= J; ++i) a[i] = 0.0;
    a[0] = log((double)S);
    double g[kMaxOrder + 1], H[(kMaxOrder + 1) * (kMaxOrder + 1)], phi;
    phi_grad(a, g, H, phi);
    for (int it = 0; it < 200; ++it) {
        double gmax = 0.0;
        for (int i = 0; i <= J; ++i) gmax = fmax(gmax, fabs(g[i]));
        // H step = g by Gaussian elimination with partial pivoting (the Hessian is
        // positive definite but can be numerically singular for exact fits)
        double Ab[(kMaxOrder + 1) * (kMaxOrder + 2)], st[kMaxOrder + 1];
        const int W = kMaxOrder + 2;
        for (int i = 0; i <= J; ++i) {
            for (int k = 0; k <= J; ++k) Ab[i * W + k] = H[i * (kMaxOrder + 1) + k];
            Ab[i * W + J + 1] = g[i];
        }
        bool singular = false;
        for (int c = 0; c <= J && !singular; ++c) {
            int piv = c;
            for (int i = c + 1; i <= J; ++i)
                if (fabs(Ab[i * W + c]) > fabs(Ab[piv * W + c])) piv = i;
            if (Ab[piv * W + c] == 0.0) { singular = true; break; }
            if (piv != c)
                for (int k = 0; k <= J + 1; ++k) {
                    double tmp = Ab[c * W + k];
                    Ab[c * W + k] = Ab[piv * W + k];
                    Ab[piv * W + k] = tmp;
                }
            for (int i = c + 1; i <= J; ++i) {
                double f = Ab[i * W + c] / Ab[c * W + c];
                for (int k = c; k <= J + 1; ++k) Ab[i * W + k] -= f * Ab[c * W + k];
            }
        }
        if (singular) return gmax <= 1e-13;
        for (int i = J; i >= 0; --i) {
            double v = Ab[i * W + J + 1];
            for (int q = i + 1; q <= J; ++q) v -= Ab[i * W + q] * st[q];
            st[i] = v / Ab[i * W + i];
        }
        if (gmax <= 1e-13) {
            // a last full Newton step: the parameters converge, not only the moments
            for (int i = 0; i <= J; ++i) a[i] -= st[i];
            return true;
        }
        double gst = 0.0;
        for (int i = 0; i <= J; ++i) gst += g[i] * st[i];
        double tstep = 1.0, an[kMaxOrder + 1], gn[kMaxOrder + 1], Hn[(kMaxOrder + 1) * (kMaxOrder + 1)], phin;
        for (;;) {
            for (int i = 0; i <= J; ++i) an[i] = a[i] - tstep * st[i];
            phi_grad(an, gn, Hn, phin);
            if (isfinite(phin) && phin <= phi - 1e-4 * tstep * gst) break;
            double gnmax = 0.0;
            for (int i = 0; i <= J; ++i) gnmax = fmax(gnmax, fabs(gn[i]));
            if (isfinite(phin) && phin <= phi + 1e-14 * fabs(phi) && gnmax <= 0.5 * gmax) break;
            tstep *= 0.5;
            // no further decrease: moments on the boundary of the moment cone up to
            // their rounding; the fit stands if the residual is at that level
            if (tstep < 1e-12) return gmax <= 1e-10;
        }
        for (int i = 0; i <= J; ++i) { a[i] = an[i]; g[i] = gn[i]; }
        for (int i = 0; i < (kMaxOrder + 1) * (kMaxOrder + 1); ++i) H[i] = Hn[i];
        phi = phin;
    }
    double gmax = 0.0;
    for (int i = 0; i <= J; ++i) gmax = fmax(gmax, fabs(g[i]));
    return gmax <= 1e-10;
}

// The same fit, a warp on up to 32 sectors: the sums over the support, the Newton step and every
// comparison in the order of maxent_fit_warp, so the results are its, bit for bit.  The FP64 pipe
// charges a warp instruction the same for one lane as for 32 (16 clocks of an SM), and a Newton step is a
// few hundred of them on the same numbers in every lane.  So here
//  * the sums of one sector after another are taken by the whole warp, its 2 J + 2 sums halved at each
//    step of the butterfly (each value still added in the butterfly's order; 12 additions for 10 values
//    instead of 50) and handed to the sector's lane;
//  * then every lane takes its own sector's step at once: those whose trial point is accepted solve for
//    the next one, the others halve theirs; finished sectors leave the loop over the sums.
template <int J>
__device__ __forceinline__ bool newton_step(const double *pw, const double *g, double *st) {
    double Ab[J + 1][J + 2];
#pragma unroll
    for (int i = 0; i <= J; ++i) {
#pragma unroll
        for (int k = 0; k <= J; ++k) Ab[i][k] = pw[i + k];
        Ab[i][J + 1] = g[i];
    }
    bool singular = false;
#pragma unroll
    for (int c = 0; c <= J; ++c) {
        int piv = c;
        double best = Ab[c][c];
#pragma unroll
        for (int i = c + 1; i <= J; ++i)
            if (fabs(Ab[i][c]) > fabs(best)) {
                piv = i;
                best = Ab[i][c];
            }
        singular = singular || best == 0.0;
#pragma unroll
        for (int i = c + 1; i <= J; ++i)
#pragma unroll
            for (int k = 0; k <= J + 1; ++k) {
                const double u = Ab[c][k], v = Ab[i][k];
                Ab[c][k] = piv == i ? v : u;
                Ab[i][k] = piv == i ? u : v;
            }
#pragma unroll
        for (int i = c + 1; i <= J; ++i) {
            const double f = Ab[i][c] / Ab[c][c];
#pragma unroll
            for (int k = c; k <= J + 1; ++k) Ab[i][k] -= f * Ab[c][k];
        }
    }
#pragma unroll
    for (int i = J; i >= 0; --i) {
        double v = Ab[i][J + 1];
#pragma unroll
        for (int q = i + 1; q <= J; ++q) v -= Ab[i][q] * st[q];
        st[i] = v / Ab[i][i];
    }
    return singular;
}

// sums over the warp of NV values a lane, in the order of a butterfly over offsets 16 .. 1: at each
// offset a lane keeps half of its values (the upper half where its bit is set).  Afterwards
// lane l holds the sum of value half_index<NV>(l).
template <int NV> __host__ __device__ constexpr int half_index(int l) {
    int at = 0, slots = NV, real = NV;  // real: the lane's own values among its slots (the rest is padding)
    for (int off = 16; off; off >>= 1) {
        if (slots == 1) break;
        const int h = (slots + 1) / 2;
        if (l & off) {
            at += h;
            real = real > h ? real - h : 0;
        } else {
            real = real < h ? real : h;
        }
        slots = h;
    }
    return real > 0 ? at : -1;
}
template <int NV> __host__ __device__ constexpr int half_owner(int v) {
    for (int l = 0; l < 32; ++l)
        if (half_index<NV>(l) == v) return l;
    return 0;
}
template <int CUR, int OFF> __device__ __forceinline__ void half_steps(double *v, int lane) {
    if constexpr (OFF > 0) {
        constexpr int H = (CUR + 1) / 2;
        if constexpr (CUR > 1) {
            const bool up = lane & OFF;
#pragma unroll
            for (int k = 0; k < H; ++k) {
                const double lo = v[k], hi = H + k < CUR ? v[H + k] : 0.0;
                v[k] = (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, OFF);
            }
        } else {
            v[0] += __shfl_xor_sync(0xffffffffu, v[0], OFF);
        }
        half_steps<(CUR > 1 ? H : 1), OFF / 2>(v, lane);
    }
}

// sums of x^i q, i <= 2 J, and of q (last) with q = exp(-f(x)) over the support x = s / S, s < S, by a
// warp: lane l ends with value half_index<2 J + 2>(l) in v[0].  xt: s / xn
template <int J>
__device__ __forceinline__ void fit_sums(const double *aa, int S, const double *xt, int xn, int lane, double *v) {
    constexpr int NP = 2 * J + 1, NV = NP + 1;
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = 0.0;
    for (int s = lane; s < S; s += 32) {
        const double xs = S == xn ? xt[s] : (double)s / S;
        double f = 0.0, xp = 1.0;
#pragma unroll
        for (int i = 0; i <= J; ++i) { f += aa[i] * xp; xp *= xs; }
        const double q = exp(-f);
        v[NP] += q;
        xp = 1.0;
#pragma unroll
        for (int i = 0; i < NP; ++i) { v[i] += xp * q; xp *= xs; }
    }
    half_steps<NV, 16>(v, lane);
}
// one trial point: its value of the dual, gradient, and whether the line search takes it
template <int J>
__device__ __forceinline__ bool trial(const double *an, const double *sum, const double *m, bool first, double phi,
                                      double gmax, double gst, double tstep, double &phin, double *gn, double &gnmax) {
    phin = sum[2 * J + 1];
    gnmax = 0.0;
#pragma unroll
    for (int i = 0; i <= J; ++i) {
        phin += an[i] * m[i];
        gn[i] = m[i] - sum[i];
        gnmax = fmax(gnmax, fabs(gn[i]));
    }
    return first || (isfinite(phin) && phin <= phi - 1e-4 * tstep * gst) ||
           (isfinite(phin) && phin <= phi + 1e-14 * fabs(phi) && gnmax <= 0.5 * gmax);
}

// the fits of the warp's sectors, lane i's with n clicks and moments m (act: it has one): 1 it stands
// (coefficients a), 0 it does not, -1 not decided after kFitRounds trial points.  x: s / xn
constexpr int kFitRounds = 40;
template <int J>
__device__ int maxent_fit_lanes(bool act, int n, const double *m, double *a, const double *x, int xn, int lane) {
    constexpr int NV = 2 * J + 2;
    double st[J + 1], phi = 0.0, gmax = 0.0, gst = 0.0, tstep = 1.0;
    int state = act ? 0 : 2, it = 0;  // 0: first point, 1: a trial point, 2: done
    int ok = act ? -1 : 0;
#pragma unroll
    for (int i = 0; i <= J; ++i) {
        a[i] = 0.0;
        st[i] = 0.0;
    }
    if (act) a[0] = log((double)n);
    unsigned left = __ballot_sync(0xffffffffu, state != 2);
    for (int round = 0; left && round < kFitRounds; ++round) {
        double an[J + 1], sum[NV];
#pragma unroll
        for (int i = 0; i <= J; ++i) an[i] = state == 1 ? a[i] - tstep * st[i] : a[i];
        for (unsigned todo = left; todo; todo &= todo - 1) {
            const int src = __ffs(todo) - 1, S = __shfl_sync(0xffffffffu, n, src);
            double aa[J + 1], v[NV];
#pragma unroll
            for (int i = 0; i <= J; ++i) aa[i] = __shfl_sync(0xffffffffu, an[i], src);
            fit_sums<J>(aa, S, x, xn, lane, v);
#pragma unroll
            for (int i = 0; i < NV; ++i) {
                const double u = __shfl_sync(0xffffffffu, v[0], half_owner<NV>(i));
                if (lane == src) sum[i] = u;
            }
        }
        if (state != 2) {
            double phin, gn[J + 1], gnmax;
            if (!trial<J>(an, sum, m, state == 0, phi, gmax, gst, tstep, phin, gn, gnmax)) {
                tstep *= 0.5;
                if (tstep < 1e-12) {
                    ok = gmax <= 1e-10;
                    state = 2;
                }
            } else {
                it += state;
                state = 1;
                phi = phin;
                gmax = gnmax;
                tstep = 1.0;
#pragma unroll
                for (int i = 0; i <= J; ++i) a[i] = an[i];
                if (it == 200) {
                    ok = gmax <= 1e-10;
                    state = 2;
                } else if (newton_step<J>(sum, gn, st)) {
                    ok = gmax <= 1e-13;
                    state = 2;
                } else if (gmax <= 1e-13) {
#pragma unroll
                    for (int i = 0; i <= J; ++i) a[i] -= st[i];
                    ok = 1;
                    state = 2;
                } else {
                    gst = 0.0;
#pragma unroll
                    for (int i = 0; i <= J; ++i) gst += gn[i] * st[i];
                }
            }
        }
        left = __ballot_sync(0xffffffffu, state != 2);
    }
    return ok;
}

// The same fit by a cluster of kSlowCtas CTAs of four warps: W = sixteen steps of a line search at once,
// 2^-Wr .. 2^-(Wr+W-1) in round r, of which the first accepted one counts.  A few fits in ten thousand
// (moments on the boundary of their cone) search 30 and more halvings in each of up to 200 iterations,
// and one of them on one warp (7,157 trial points, 66 ms) took longer than all others together.  The step is solved
// by one warp of each CTA (a CTA's four warps sit on the four quarters of its SM, each with an FP64 pipe of
// its own); every thread keeps the state.
// `one`: a CTA by itself, W = 4: where there are thousands of such fits the steps tried for nothing fill the pipes.
constexpr int kSlowCtas = 4, kSlowThreads = 128, kSlowWarps = kSlowCtas * kSlowThreads / 32;
struct SlowShared {
    double x[kApproxMaxN];
    double st[kMaxOrder + 1];
    double sum[2][kSlowThreads / 32][2 * kMaxOrder + 2];  // two rounds' trial sums
    int take[2][kSlowThreads / 32];
    int singular;
    long long job;
};
__device__ __forceinline__ void slow_sync(const cooperative_groups::cluster_group &cl, bool one) {
    if (one) __syncthreads();
    else cl.sync();
}
template <int J>
__device__ bool maxent_fit_cluster(const cooperative_groups::cluster_group &cl, bool one, SlowShared &sh, int n,
                                   const double *m, double *a) {
    constexpr int NV = 2 * J + 2;
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, rank = (int)cl.block_rank();
    const int W = one ? kSlowThreads / 32 : kSlowWarps, me = one ? wp : rank * 4 + wp;
    double st[J + 1], an[J + 1], sum[NV], v[NV], gn[J + 1], phi = 0.0, phin, gmax = 0.0, gnmax, gst = 0.0;
    int buf = 0;
#pragma unroll
    for (int i = 0; i <= J; ++i) a[i] = 0.0;
    a[0] = log((double)n);
    fit_sums<J>(a, n, sh.x, n, lane, v);
#pragma unroll
    for (int i = 0; i < NV; ++i) sum[i] = __shfl_sync(0xffffffffu, v[0], half_owner<NV>(i));
    trial<J>(a, sum, m, true, 0.0, 0.0, 0.0, 1.0, phi, gn, gmax);
    for (int it = 0; it < 200; ++it) {
        if (wp == 0) {
            const bool singular = newton_step<J>(sum, gn, st);
            if (lane == 0) {
#pragma unroll
                for (int i = 0; i <= J; ++i) sh.st[i] = st[i];
                sh.singular = singular;
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i <= J; ++i) st[i] = sh.st[i];
        const bool singular = sh.singular;
        if (singular) return gmax <= 1e-13;
        if (gmax <= 1e-13) {
#pragma unroll
            for (int i = 0; i <= J; ++i) a[i] -= st[i];
            return true;
        }
        gst = 0.0;
#pragma unroll
        for (int i = 0; i <= J; ++i) gst += gn[i] * st[i];
        double tround = 1.0;
        for (;;) {
            double t = tround;
            for (int c = 0; c < me; ++c) t *= 0.5;
#pragma unroll
            for (int i = 0; i <= J; ++i) an[i] = a[i] - t * st[i];
            fit_sums<J>(an, n, sh.x, n, lane, v);
#pragma unroll
            for (int i = 0; i < NV; ++i) sum[i] = __shfl_sync(0xffffffffu, v[0], half_owner<NV>(i));
            const bool take = t >= 1e-12 && trial<J>(an, sum, m, false, phi, gmax, gst, t, phin, gn, gnmax);
            if (lane == 0) {
                sh.take[buf][wp] = take;
#pragma unroll
                for (int i = 0; i < NV; ++i) sh.sum[buf][wp][i] = sum[i];
            }
            slow_sync(cl, one);  // this round's sums are in; the other buffer is free again after the next one
            int found = -1;
            for (int c = W - 1; c >= 0; --c)
                if ((one ? &sh : cl.map_shared_rank(&sh, c / 4))->take[buf][c & 3]) found = c;
            if (found >= 0) {
                const double *src = (one ? &sh : cl.map_shared_rank(&sh, found / 4))->sum[buf][found & 3];
#pragma unroll
                for (int i = 0; i < NV; ++i) sum[i] = src[i];
                t = tround;
                for (int c = 0; c < found; ++c) t *= 0.5;
#pragma unroll
                for (int i = 0; i <= J; ++i) a[i] -= t * st[i];
            }
            buf ^= 1;
            if (found >= 0) break;
            for (int c = 0; c < W; ++c) tround *= 0.5;
            if (tround < 1e-12) return gmax <= 1e-10;
        }
        trial<J>(a, sum, m, true, 0.0, 0.0, 0.0, 1.0, phi, gn, gmax);
    }
    return gmax <= 1e-10;
}

__device__ __forceinline__ double stirling2(int i, int w) {
    // S(i, w) for i, w <= 4
    const double tab[5][5] = {{1, 0, 0, 0, 0}, {0, 1, 0, 0, 0}, {0, 1, 1, 0, 0}, {0, 1, 3, 1, 0}, {0, 1, 7, 6, 1}};
    return tab[i][w];
}

// inverse DFT of one pattern's tables (real: O is real, so D(conj t) = conj D(t)):
//   D_w^(k) = (1/L) sum_l D_w(t_l) e^{-2 pi i k l / L}
// gridDim.y CTAs per pattern, about eight an SM in all: one each left most SMs without work on 64
// patterns and waited for the largest ones.  Measured on a GB300, order 2, 64
// patterns of 40 to 90 clicks: 1.95 -> 0.59 ms.
__global__ void __launch_bounds__(kDftThreads) approx_dft_kernel(int order, ApproxPlan pl) {
    extern __shared__ double tw[];  // cos, sin (2 pi m / L), m < L
    __shared__ double red[kDftThreads / 32];
    const int p = blockIdx.x, t = threadIdx.x;
    const int n = pl.pat_n[p], L = pl.pat_L[p];
    if (n < 0 || L <= 0 || *pl.overflow) return;
    const int H = L / 2;
    for (int m = t; m < L; m += kDftThreads) sincospi(2.0 * (double)m / (double)L, &tw[2 * m + 1], &tw[2 * m]);
    __syncthreads();
    const double *U = pl.unit_D + (size_t)pl.unit_off[p] * 2 * (kMaxOrder + 1);
    double *D = pl.sec_D + (size_t)pl.sec_off[p] * (kMaxOrder + 1);
    double mx = 0.0;
    for (int idx = blockIdx.y * kDftThreads + t; idx < (order + 1) * L; idx += gridDim.y * kDftThreads) {
        const int k = idx / (order + 1), w = idx - k * (order + 1);
        double s = U[2 * w];  // l = 0
        int m = 0;            // k l mod L
        for (int l = 1; l <= H; ++l) {
            m += k;
            if (m >= L) m -= L;
            const double re = U[(size_t)l * 2 * (kMaxOrder + 1) + 2 * w];
            const double im = U[(size_t)l * 2 * (kMaxOrder + 1) + 2 * w + 1];
            const double term = re * tw[2 * m] + im * tw[2 * m + 1];  // Re(D(t_l) e^{-i 2 pi k l / L})
            s += (2 * l == L) ? term : 2.0 * term;
        }
        D[(size_t)k * (kMaxOrder + 1) + w] = s / L;
        if (w == 0) mx = fmax(mx, s / L);
    }
    for (int off = 16; off; off >>= 1) mx = fmax(mx, __shfl_xor_sync(0xffffffffu, mx, off));
    if ((t & 31) == 0) red[t >> 5] = mx;
    __syncthreads();
    if (t == 0) {
        for (int w = 1; w < kDftThreads / 32; ++w) mx = fmax(mx, red[w]);
        if (mx > 0.0)  // (of the CTAs' maxima, none negative: as integers; the plan sets it to 0)
            atomicMax((unsigned long long *)pl.pat_max + p, (unsigned long long)__double_as_longlong(mx));
    }
}

// raw moments mu_i, i <= Jmax, of a sector from its factorial moments
__device__ __forceinline__ void raw_moments(const double *Dk, int Jmax, double *mu) {
    for (int i = 0; i <= Jmax; ++i) {
        double s = 0.0, fw = 1.0;
        for (int w = 0; w <= i; ++w) {
            s += stirling2(i, w) * fw * Dk[w];
            fw *= (w + 1);
        }
        mu[i] = s;
    }
}

// one warp per (pattern, sector k): factorial moments -> raw moments (Stirling numbers)
// -> maximum-entropy fit on the support v in [max(0, n - k), n - 1] -> the last point.
// curves (one pattern only, else null): every sector's fitted distribution over the
// clicks c = n - v, tilted, row k of curve_K + 1 rows of n + 1 (sectors with fewer photons
// than detectors are fitted too)
__global__ void __launch_bounds__(kSecThreads) approx_sector_fit_kernel(int n_pat, int order, double sector_eps,
                                                                      ApproxPlan pl, double *__restrict__ curves,
                                                                      int curve_K) {
    const int lane = threadIdx.x & 31;
    const long long nsec = pl.sec_off[n_pat];
    const long long nwarps = (long long)gridDim.x * (kSecThreads / 32);
    if (*pl.overflow) return;
    for (long long gs = (long long)blockIdx.x * (kSecThreads / 32) + (threadIdx.x >> 5); gs < nsec; gs += nwarps) {
        // the pattern whose sector range holds gs (the last with sec_off <= gs)
        int lo = 0, hi = n_pat;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pl.sec_off[mid] <= gs) lo = mid; else hi = mid;
        }
        const int p = lo, n = pl.pat_n[p];
        const int k = (int)(gs - pl.sec_off[p]);
        const double *Dk = pl.sec_D + (size_t)gs * (kMaxOrder + 1);
        const double D0 = Dk[0];
        double val = 0.0;
        bool fell = false;
        const bool curve = curves != nullptr && k <= curve_K;
        if (curve && k == 0 && D0 > 0.0 && lane == 0) curves[0] = D0;   // no photon: no click (c = 0)
        if (n == 0) {
            val = (k == 0) ? D0 : 0.0;
        } else if ((k >= n || (curve && k >= 1)) && D0 >= sector_eps * pl.pat_max[p] && D0 > 0.0) {
            const int v0 = n - k > 0 ? n - k : 0;
            const int S = n - v0;
            const int Jmax = order < S - 1 ? order : S - 1;
            double mu[kMaxOrder + 1];
            raw_moments(Dk, Jmax, mu);
            bool done = false;
            for (int J = Jmax; J >= 0 && !done; --J) {
                double m[kMaxOrder + 1], a[kMaxOrder + 1];
                double np = 1.0;
                for (int i = 0; i <= J; ++i) { m[i] = mu[i] / np / mu[0]; np *= n; }
                if (maxent_fit_warp(v0, n, J, m, a, lane)) {
                    val = k >= n ? mu[0] * exp(-a[0]) : 0.0;
                    done = true;
                    if (J != Jmax) fell = true;
                    if (curve)
                        for (int v = v0 + lane; v < n; v += 32) {
                            const double x = (double)v / n;
                            double f = a[J];
                            for (int i = J - 1; i >= 0; --i) f = f * x + a[i];
                            curves[(size_t)k * (n + 1) + (n - v)] = mu[0] * exp(-f);
                        }
                }
            }
            if (!done) fell = true;
        }
        if (lane == 0) pl.sec_part[gs] = fell ? -val : val;   // the sign marks a fallback
    }
}

// The fits of the warp's sectors whose own order (the batch's, or less where the support is small) is J or below,
// one order after the other: 1 it stands (val), else to be done by approx_fit_slow_kernel
template <int J>
__device__ __forceinline__ int fit_lane_orders(bool fit, int Jmax, int n, const double *Dk, const double *x, int xn,
                                              int lane, double &val) {
    int done = 0;
    const bool act = fit && Jmax == J;
    if (__any_sync(0xffffffffu, act)) {
        double m[J + 1], a[J + 1], mu[J + 1];
        if (act) {
            raw_moments(Dk, J, mu);
            double np = 1.0;
#pragma unroll
            for (int i = 0; i <= J; ++i) {
                m[i] = mu[i] / np / mu[0];
                np *= n;
            }
        }
        const int ok = maxent_fit_lanes<J>(act, n, m, a, x, xn, lane);
        if (act && ok == 1) {
            val = mu[0] * exp(-a[0]);
            done = 1;
        }
    }
    if constexpr (J > 0) done |= fit_lane_orders<J - 1>(fit, Jmax, n, Dk, x, xn, lane, val);
    return done;
}

// The same values, P consecutive sectors a warp (P <= 32), all of an order at once in maxent_fit_lanes; the
// fits that take many trial points or fail go to approx_fit_slow_kernel.  Both kernels together, GB300: 256
// 50-mode patterns at order 2 11.4 -> 5.2 ms, 96 at order 4 66 -> 14.8 ms (one warp a sector before).
// Patterns of no more clicks than the order have their lower order here too: on the clusters, 200
// patterns of 2 and 3 clicks at order 2 took 8.9 ms for 3.8.
template <int J>
__global__ void __launch_bounds__(kFitThreads, 3) approx_sector_fit_lanes_kernel(int n_pat, int P, double sector_eps,
                                                                                ApproxPlan pl) {
    __shared__ double s_x[kFitThreads / 32][kPairMaxN];
    const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
    double *x = s_x[wp];
    const long long nsec = pl.sec_off[n_pat];
    if (*pl.overflow) return;
    const long long g0 = ((long long)blockIdx.x * (kFitThreads / 32) + wp) * P, gs = g0 + lane;
    if (g0 >= nsec) return;
    const bool in = lane < P && gs < nsec;
    int lo = 0, hi = n_pat;  // the pattern whose sector range holds gs
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (pl.sec_off[mid] <= (in ? gs : g0)) lo = mid; else hi = mid;
    }
    const int p = lo, n = pl.pat_n[p];
    const int k = (int)(gs - pl.sec_off[p]);
    const int xn = __shfl_sync(0xffffffffu, n, 0);
    for (int v = lane; v < xn; v += 32) x[v] = (double)v / xn;
    __syncwarp();
    const double *Dk = pl.sec_D + (size_t)(in ? gs : g0) * (kMaxOrder + 1);
    const double D0 = Dk[0];
    double val = 0.0;
    const bool fit = in && n > 0 && k >= n && D0 >= sector_eps * pl.pat_max[p] && D0 > 0.0;
    if (in && n == 0) val = k == 0 ? D0 : 0.0;
    const int done = fit_lane_orders<J>(fit, J < n - 1 ? J : n - 1, n, Dk, x, xn, lane, val);
    if (in) pl.sec_part[gs] = val;
    if (fit && !done) pl.sec_slow[atomicAdd(pl.slow, 1ull)] = (uint32_t)gs;
}

// the sectors that approx_sector_fit_lanes_kernel left: fits that take many trial points, and fits that
// fail at their order and go on at lower ones
__global__ void __cluster_dims__(kSlowCtas, 1, 1) __launch_bounds__(kSlowThreads)
    approx_fit_slow_kernel(int n_pat, int order, ApproxPlan pl) {
    __shared__ SlowShared sh;
    const cooperative_groups::cluster_group cl = cooperative_groups::this_cluster();
    const int t = threadIdx.x;
    if (*pl.overflow) return;
    const long long jobs = (long long)pl.slow[0];
    // more than six a cluster: each CTA by itself (200 patterns of 2 and 3 clicks at order 2, 2121 such fits, whole
    // calls: 6.3 -> 3.7 ms; 200 of 5 and 6 clicks at order 4, 4569 of them: 50 -> 27 ms).  With fewer the longest
    // fit counts: of seven batches with 640 to 850 three were up to a third slower that way.
    const bool one = jobs > 6ll * (gridDim.x / kSlowCtas);
    const bool first = (one || cl.block_rank() == 0) && t == 0;
    for (;;) {
        if (first) sh.job = (long long)atomicAdd(pl.slow + 1, 1ull);
        slow_sync(cl, one);
        const long long job = (one ? &sh : cl.map_shared_rank(&sh, 0))->job;
        slow_sync(cl, one);  // read by all before the next one is drawn, and before a CTA exits
        if (job >= jobs) break;
        const long long gs = pl.sec_slow[job];
        int lo = 0, hi = n_pat;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pl.sec_off[mid] <= gs) lo = mid; else hi = mid;
        }
        const int n = pl.pat_n[lo];
        for (int v = t; v < n; v += kSlowThreads) sh.x[v] = (double)v / n;
        __syncthreads();
        const double *Dk = pl.sec_D + (size_t)gs * (kMaxOrder + 1);
        const int top = order < n - 1 ? order : n - 1;
        double m[kMaxOrder + 1], a[kMaxOrder + 1], mu[kMaxOrder + 1], val = 0.0;
        raw_moments(Dk, top, mu);
        bool done = false, fell = false;
        for (int j = top; j >= 0 && !done; --j) {
            double np = 1.0;
            for (int i = 0; i <= j; ++i) { m[i] = mu[i] / np / mu[0]; np *= n; }
            done = j == 4   ? maxent_fit_cluster<4>(cl, one, sh, n, m, a)
                   : j == 3 ? maxent_fit_cluster<3>(cl, one, sh, n, m, a)
                   : j == 2 ? maxent_fit_cluster<2>(cl, one, sh, n, m, a)
                   : j == 1 ? maxent_fit_cluster<1>(cl, one, sh, n, m, a)
                            : maxent_fit_cluster<0>(cl, one, sh, n, m, a);
            if (done) {
                val = mu[0] * exp(-a[0]);
                if (j != top) fell = true;
            }
            slow_sync(cl, one);  // the next fit writes its sums where a slower CTA may still read this one's
        }
        if (!done) fell = true;
        if (first) pl.sec_part[gs] = fell ? -val : val;   // the sign marks a fallback
    }
}
// P: as many sectors a warp as leave three warps for each quarter of an SM
template <int J> void launch_fit_lanes(gbs_ctx *ctx, long long secs, int n_pat, double eps, const ApproxPlan &pl) {
    int P = 1;
    while (P < 32 && secs >= 2ll * P * 12 * ctx->num_sms) P *= 2;
    const long long per = (long long)(kFitThreads / 32) * P;
    approx_sector_fit_lanes_kernel<J><<<(unsigned)((secs + per - 1) / per), kFitThreads, 0, ctx->stream>>>(n_pat, P, eps,
                                                                                                         pl);
}

// the curves untilted (rho^-k) and scaled by det(sigma_Q)^{-1/2}
__global__ void approx_curve_scale_kernel(int curve_K, int n, const double *__restrict__ logdet, ApproxPlan pl,
                                          double *__restrict__ curves) {
    const long long f = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (f >= (long long)(curve_K + 1) * (n + 1)) return;
    const int k = (int)(f / (n + 1));
    curves[f] = *pl.overflow ? nan("") : curves[f] * exp(-0.5 * (*logdet) - k * log(pl.pat_rho[0]));
}

// per pattern (one warp): sum_k part_k rho^{-k} in logs (the tables are tilted by rho^k)
// floor_eps > 0 (FP32 minors, whose moments resolve sectors only down to that share of the
// largest): a sector k >= n below the floor carries at most floor_eps * (largest) of tilted
// mass, so its all-clicked point at most that; when those bounds add up to kFlagShare of the
// estimate, the estimate may be missing what the precision cannot resolve: GBS_E_FLOOR
__global__ void __launch_bounds__(kSumThreads) approx_sum_kernel(int n_pat, const double *__restrict__ logdet,
                                                               double floor_eps,
                                                               ApproxPlan pl, double *__restrict__ logP,
                                                               double *__restrict__ kappa,
                                                               double *__restrict__ err_bound,
                                                               int32_t *__restrict__ status) {
    const int p = blockIdx.x * (kSumThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    if (p >= n_pat) return;
    const int n = pl.pat_n[p], L = pl.pat_L[p];
    if (n < 0 || *pl.overflow) {
        if (lane == 0) {
            logP[p] = nan("");
            if (kappa) kappa[p] = nan("");
            if (err_bound) err_bound[p] = nan("");
            if (status) status[p] = n < 0 ? GBS_E_INVALID : GBS_E_NOMEM;
        }
        return;
    }
    const double *part = pl.sec_part + pl.sec_off[p];
    const double lr = log(pl.pat_rho[p]);
    double top = -INFINITY;
    for (int k = lane; k < L; k += 32)
        if (part[k] != 0.0) top = fmax(top, log(fabs(part[k])) - k * lr);
    for (int off = 16; off; off >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, off));
    double s = 0.0, sf = 0.0, sd = 0.0;
    const double lfloor = floor_eps > 0.0 && pl.pat_max[p] > 0.0 ? log(floor_eps * pl.pat_max[p]) : -INFINITY;
    for (int k = lane; k < L; k += 32)
        if (part[k] != 0.0) {
            const double w = exp(log(fabs(part[k])) - k * lr - top);
            s += w;
            if (part[k] < 0.0) sf += w;
        } else if (k >= n && n > 0 && isfinite(lfloor)) {
            sd += exp(lfloor - k * lr - (isfinite(top) ? top : lfloor));
        }
    s = warp_sum_bcast(s);
    sf = warp_sum_bcast(sf);
    sd = warp_sum_bcast(sd);
    if (lane == 0) {
        logP[p] = s > 0.0 ? -0.5 * (*logdet) + top + log(s) : -INFINITY;
        if (kappa) kappa[p] = (double)(L - 1);
        if (err_bound) err_bound[p] = nan("");
        int st = GBS_OK;
        if (pl.unit_flag[p]) st = GBS_E_NOT_SPD;
        else if (sd > 0.0 && (!(s > 0.0) || sd >= kFlagShare * s)) st = GBS_E_FLOOR;
        else if (sf >= kFlagShare * s) st = GBS_E_FIT;
        if (status) status[p] = st;
    }
}

// ---- gradient of the approximation (not in the paper) ---------------------------------
// L = sum_p w_p log P_p; reverse mode through the steps above, per pattern:
//  * sum:     d log(sum_k part_k rho^-k) / d part_k = rho^-k / sum;
//  * fit:     implicit derivative of the moment conditions of the fitted exp(-f) on its
//             support, sum_s x_s^i F(x_s) = mu'_i with mu'_i = mu_i / n^i: at the solution
//             d part / d mu'_i = e^{-a_0} (Hn^-1)_0i, Hn_il = sum_s x_s^(i+l) e^{-f(x_s)} the
//             Newton matrix of the normalised fit;
//  * moments: mu'_i = sum_{w <= i} S(i, w) w! D_w^(k) / n^i;
//  * DFT:     D_w^(k) = (1/L) sum_{l <= L/2} c_l Re(D_w(t_l) e^{-2 pi i k l / L}), c_l = 1 for
//             l = 0 and l = L/2, else 2; the adjoint of D_w(t_l) as one complex number
//             (d/dRe - i d/dIm) is cbar_w(t_l) = (c_l / L) sum_k gamma_w^(k) e^{-2 pi i k l / L};
//  * minors:  with d det(X)^-1/2 = -1/2 det(X)^-1/2 tr(X^-1 dX) and I - t O = (1 - t) I + t A,
//             d Z_{S\W}(t) / dA_S = -1/2 t Z_{S\W}(t) [(I - t O_{S\W})^-1 embedded in S], and that
//             embedded inverse is G - G_{.W} G_WW^-1 G_{W.} (zero on the rows of W), so unit
//             (S, t_l) adds Re(-1/2 t (s G - G K G)) to dlog P / dA_S, with
//             s = sum_w cbar_w D_w(t) and K = sum_{W, |W| <= j} cbar_|W| Z_{S\W}(t) embed(G_WW^-1).
// K is built one 2 x 2 mode block (a, b) per warp (no atomics, a fixed summation order):
// every W holding a and b is V + {a, b} with V over the other modes; eliminating V first
// leaves on the rows of a and b the Schur complement of V in G_WW, whose inverse is the
// (a, b) block of G_WW^-1 and whose pivots complete det(G_WW).
constexpr int kGradApproxMaxN = 48;  // clicks per pattern on the approximation's gradient
constexpr int kPanel = 8;            // columns of K G per pass of the G K G product

__device__ __forceinline__ double factorial_small(int w) {
    const double tab[kMaxOrder + 1] = {1, 1, 2, 6, 24};
    return tab[w];
}

// y = Hn^-1 e_0 for the (J + 1) x (J + 1) Newton matrix Hn_il = pw[i + l] (Gaussian
// elimination with partial pivoting, as the fit's own step); false if singular
__device__ bool solve_e0(int J, const double *pw, double *y) {
    const int W = kMaxOrder + 2;
    double Ab[(kMaxOrder + 1) * (kMaxOrder + 2)];
    for (int i = 0; i <= J; ++i) {
        for (int k = 0; k <= J; ++k) Ab[i * W + k] = pw[i + k];
        Ab[i * W + J + 1] = i == 0 ? 1.0 : 0.0;
    }
    for (int c = 0; c <= J; ++c) {
        int piv = c;
        for (int i = c + 1; i <= J; ++i)
            if (fabs(Ab[i * W + c]) > fabs(Ab[piv * W + c])) piv = i;
        if (Ab[piv * W + c] == 0.0) return false;
        if (piv != c)
            for (int k = 0; k <= J + 1; ++k) {
                const double tmp = Ab[c * W + k];
                Ab[c * W + k] = Ab[piv * W + k];
                Ab[piv * W + k] = tmp;
            }
        for (int i = c + 1; i <= J; ++i) {
            const double f = Ab[i * W + c] / Ab[c * W + c];
            for (int k = c; k <= J + 1; ++k) Ab[i * W + k] -= f * Ab[c * W + k];
        }
    }
    for (int i = J; i >= 0; --i) {
        double v = Ab[i * W + J + 1];
        for (int q = i + 1; q <= J; ++q) v -= Ab[i * W + q] * y[q];
        y[i] = v / Ab[i * W + i];
    }
    return true;
}

// one warp per sector: the forward's fit again (same inputs and code, so the same order
// and coefficients), then beta_w = d part / d D_w^(k), w = 0..kMaxOrder (0 where unused)
__global__ void __launch_bounds__(kSecThreads) approx_fit_adjoint_kernel(int n_pat, int order, ApproxPlan pl,
                                                                       double *__restrict__ sec_B) {
    const int lane = threadIdx.x & 31;
    const long long nsec = pl.sec_off[n_pat];
    const long long nwarps = (long long)gridDim.x * (kSecThreads / 32);
    if (*pl.overflow) return;
    for (long long gs = (long long)blockIdx.x * (kSecThreads / 32) + (threadIdx.x >> 5); gs < nsec; gs += nwarps) {
        int lo = 0, hi = n_pat;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pl.sec_off[mid] <= gs) lo = mid; else hi = mid;
        }
        const int p = lo, n = pl.pat_n[p];
        const int k = (int)(gs - pl.sec_off[p]);
        const double *Dk = pl.sec_D + (size_t)gs * (kMaxOrder + 1);
        double beta[kMaxOrder + 1];
        for (int w = 0; w <= kMaxOrder; ++w) beta[w] = 0.0;
        // fitted sectors only (k >= n: the support is v = 0..n-1)
        if (n > 0 && k >= n && pl.sec_part[gs] != 0.0) {
            const int Jmax = order < n - 1 ? order : n - 1;
            double mu[kMaxOrder + 1];
            for (int i = 0; i <= Jmax; ++i) {
                double s = 0.0, fw = 1.0;
                for (int w = 0; w <= i; ++w) {
                    s += stirling2(i, w) * fw * Dk[w];
                    fw *= (w + 1);
                }
                mu[i] = s;
            }
            for (int J = Jmax; J >= 0; --J) {
                double m[kMaxOrder + 1], a[kMaxOrder + 1];
                double np = 1.0;
                for (int i = 0; i <= J; ++i) { m[i] = mu[i] / np / mu[0]; np *= n; }
                if (!maxent_fit_warp(0, n, J, m, a, lane)) continue;
                double pw[2 * kMaxOrder + 1];
                for (int q = 0; q <= 2 * J; ++q) pw[q] = 0.0;
                for (int sp = lane; sp < n; sp += 32) {
                    const double x = (double)sp / n;
                    double f = 0.0, xp = 1.0;
                    for (int i = 0; i <= J; ++i) { f += a[i] * xp; xp *= x; }
                    const double q = exp(-f);
                    xp = 1.0;
                    for (int i = 0; i <= 2 * J; ++i) { pw[i] += xp * q; xp *= x; }
                }
                for (int i = 0; i <= 2 * J; ++i) pw[i] = warp_sum_bcast(pw[i]);
                double y[kMaxOrder + 1];
                if (solve_e0(J, pw, y)) {
                    const double e = exp(-a[0]);
                    for (int w = 0; w <= J; ++w) {
                        double s = 0.0, ni = 1.0;
                        for (int i = 0; i <= J; ++i) {
                            if (i >= w) s += y[i] * stirling2(i, w) * factorial_small(w) / ni;
                            ni *= n;
                        }
                        beta[w] = e * s;
                    }
                }
                break;
            }
        }
        if (lane == 0)
            for (int w = 0; w <= kMaxOrder; ++w) sec_B[(size_t)gs * (kMaxOrder + 1) + w] = beta[w];
    }
}

// one CTA per pattern: gamma_w^(k) = beta_w^(k) rho^-k / sum (in place), then the DFT's
// adjoint to the units: cbar_w(t_l), l = 0..L/2, interleaved (re, im) like unit_D
__global__ void __launch_bounds__(kDftThreads) approx_dft_adjoint_kernel(int order, ApproxPlan pl,
                                                                       double *__restrict__ sec_B,
                                                                       double *__restrict__ unit_B) {
    extern __shared__ double tw[];  // cos, sin (2 pi m / L), m < L
    __shared__ double s_top, s_sum;
    const int p = blockIdx.x, t = threadIdx.x;
    const int n = pl.pat_n[p], L = pl.pat_L[p];
    if (n <= 0 || L <= 0 || *pl.overflow) return;
    const int H = L / 2;
    const double *part = pl.sec_part + pl.sec_off[p];
    const double lr = log(pl.pat_rho[p]);
    if (t < 32) {
        // the sum of the tilted last points in logs, as the forward's sum
        double top = -INFINITY;
        for (int k = t; k < L; k += 32)
            if (part[k] != 0.0) top = fmax(top, log(fabs(part[k])) - k * lr);
        for (int off = 16; off; off >>= 1) top = fmax(top, __shfl_xor_sync(0xffffffffu, top, off));
        double s = 0.0;
        for (int k = t; k < L; k += 32)
            if (part[k] != 0.0) s += exp(log(fabs(part[k])) - k * lr - top);
        s = warp_sum_bcast(s);
        if (t == 0) { s_top = top; s_sum = s; }
    }
    for (int m = t; m < L; m += kDftThreads) sincospi(2.0 * (double)m / (double)L, &tw[2 * m + 1], &tw[2 * m]);
    __syncthreads();
    const double top = s_top, ssum = s_sum;
    double *B = sec_B + (size_t)pl.sec_off[p] * (kMaxOrder + 1);
    for (int k = t; k < L; k += kDftThreads) {
        const double gk = (part[k] != 0.0 && ssum > 0.0) ? exp(-k * lr - top) / ssum : 0.0;
        for (int w = 0; w <= kMaxOrder; ++w) B[(size_t)k * (kMaxOrder + 1) + w] *= gk;
    }
    __syncthreads();
    double *Ub = unit_B + (size_t)pl.unit_off[p] * 2 * (kMaxOrder + 1);
    for (int idx = t; idx < (H + 1) * (kMaxOrder + 1); idx += kDftThreads) {
        const int l = idx / (kMaxOrder + 1), w = idx - l * (kMaxOrder + 1);
        double re = 0.0, im = 0.0;
        if (w <= order) {
            int m = 0;  // k l mod L
            for (int k = 0; k < L; ++k) {
                const double gm = B[(size_t)k * (kMaxOrder + 1) + w];
                re += gm * tw[2 * m];
                im -= gm * tw[2 * m + 1];
                m += l;
                if (m >= L) m -= L;
            }
        }
        const double c = (l == 0 || 2 * l == L) ? 1.0 : 2.0;
        Ub[(size_t)l * 2 * (kMaxOrder + 1) + 2 * w] = c * re / L;
        Ub[(size_t)l * 2 * (kMaxOrder + 1) + 2 * w + 1] = c * im / L;
    }
}

// The modes m[0..NV-1] (V) and then the NT tail modes of G_WW (local mode indices, rows
// 2m and 2m + 1 of G), from the swept matrix Gs (= -G, packed): eliminate V's 2 NV pivots
// (unpivoted LDL^T) and return det(G_VV)^-1/2 (principal roots of pivot pairs; Re > 0
// for every pivot of the accretive G) with the Schur complement of V on the tail rows
// in s (packed 2 NT x 2 NT).
template <int NV, int NT>
__device__ __forceinline__ cx<double> schur_tail(const cx<double> *__restrict__ Gs, int N, const int (&m)[NV + NT],
                                                 cx<double> (&s)[NT * (2 * NT + 1)], bool &bad) {
    constexpr int K = 2 * (NV + NT);
    cx<double> a[K * (K + 1) / 2];
    int rr[K];
#pragma unroll
    for (int i = 0; i < K; ++i) rr[i] = 2 * m[i >> 1] + (i & 1);
#pragma unroll
    for (int i = 0; i < K; ++i)
#pragma unroll
        for (int j = i; j < K; ++j) {
            const cx<double> v = Gs[pidx_any(N, rr[i], rr[j])];
            a[pidx(K, i, j)] = mk<double>(-v.re, -v.im);
        }
    cx<double> f = mk<double>(1.0, 0.0), prev = mk<double>(1.0, 0.0);
#pragma unroll
    for (int k = 0; k < 2 * NV; ++k) {
        const cx<double> d = a[pidx(K, k, k)];
        if (!(d.re > 0.0)) bad = true;
        if (k & 1) f = f * crsqrt(prev * d);
        prev = d;
        const cx<double> inv = cinv(d);
#pragma unroll
        for (int i = k + 1; i < K; ++i) {
            const cx<double> li = a[pidx(K, k, i)] * inv;
#pragma unroll
            for (int j = i; j < K; ++j) a[pidx(K, i, j)] = cfms_d(a[pidx(K, i, j)], li, a[pidx(K, k, j)]);
        }
    }
#pragma unroll
    for (int i = 0; i < 2 * NT; ++i)
#pragma unroll
        for (int j = i; j < 2 * NT; ++j) s[pidx(2 * NT, i, j)] = a[pidx(K, 2 * NV + i, 2 * NV + j)];
    return f;
}

// C(o, v) for v <= 3
__device__ __forceinline__ int binom_small(int o, int v) {
    return v == 0 ? 1 : v == 1 ? o : v == 2 ? o * (o - 1) / 2 : o * (o - 1) * (o - 2) / 6;
}
// the r-th pair i1 < i2 in colex order (i2 the largest with C(i2, 2) <= r); FP32 estimate,
// corrected exactly in integers
__device__ __forceinline__ void unrank_pair(int r, int &i1, int &i2) {
    int c = (int)sqrtf(2.0f * (float)r);
    while ((c + 1) * c / 2 <= r) ++c;
    while (c * (c - 1) / 2 > r) --c;
    i2 = c;
    i1 = r - c * (c - 1) / 2;
}
// the r-th triple i1 < i2 < i3 in colex order
__device__ __forceinline__ void unrank_triple(int r, int &i1, int &i2, int &i3) {
    int c = (int)cbrtf(6.0f * (float)r);
    while ((c + 1) * c * (c - 1) / 6 <= r) ++c;
    while (c * (c - 1) * (c - 2) / 6 > r) --c;
    i3 = c;
    unrank_pair(r - c * (c - 1) * (c - 2) / 6, i1, i2);
}

// W = V + {a}: adds wz Z-factor det(G_WW)^-1/2 [G_WW^-1]_aa to the diagonal block (k00, k01, k11)
template <int NV>
__device__ __forceinline__ void diag_leaf(const cx<double> *__restrict__ Gs, int N, const int (&m)[NV + 1],
                                          cx<double> wz, cx<double> &k00, cx<double> &k01, cx<double> &k11,
                                          bool &bad) {
    cx<double> s[3];
    const cx<double> f = schur_tail<NV, 1>(Gs, N, m, s, bad);
    const cx<double> det = cfms_d(s[0] * s[2], s[1], s[1]);
    if (!(s[0].re > 0.0) || !(det.re * s[0].re + det.im * s[0].im > 0.0)) bad = true;
    const cx<double> wgt = wz * f * crsqrt(det) * cinv(det);
    k00 = cfma_d(k00, wgt, s[2]);
    k01 = cfms_d(k01, wgt, s[1]);
    k11 = cfma_d(k11, wgt, s[0]);
}

// W = V + {a, b}, a < b: adds wz det(G_WW)^-1/2 [G_WW^-1]_ab to the off-diagonal block
// ko = (00, 01, 10, 11); with the tail S = [[P, Q], [Q^T, R]] (a's rows, b's rows),
// [S^-1]_ab = -P^-1 Q C^-1, C = R - Q^T P^-1 Q, det S = det P det C
template <int NV>
__device__ __forceinline__ void off_leaf(const cx<double> *__restrict__ Gs, int N, const int (&m)[NV + 2],
                                         cx<double> wz, cx<double> (&ko)[4], bool &bad) {
    cx<double> s[10];
    const cx<double> f = schur_tail<NV, 2>(Gs, N, m, s, bad);
    const cx<double> p00 = s[pidx(4, 0, 0)], p01 = s[pidx(4, 0, 1)], p11 = s[pidx(4, 1, 1)];
    const cx<double> q00 = s[pidx(4, 0, 2)], q01 = s[pidx(4, 0, 3)], q10 = s[pidx(4, 1, 2)], q11 = s[pidx(4, 1, 3)];
    const cx<double> r00 = s[pidx(4, 2, 2)], r01 = s[pidx(4, 2, 3)], r11 = s[pidx(4, 3, 3)];
    const cx<double> detP = cfms_d(p00 * p11, p01, p01);
    const cx<double> iP = cinv(detP);
    // X = P^-1 Q
    const cx<double> x00 = cfms_d(p11 * q00, p01, q10) * iP, x01 = cfms_d(p11 * q01, p01, q11) * iP;
    const cx<double> x10 = cfms_d(p00 * q10, p01, q00) * iP, x11 = cfms_d(p00 * q11, p01, q01) * iP;
    const cx<double> c00 = cfms_d(cfms_d(r00, q00, x00), q10, x10), c01 = cfms_d(cfms_d(r01, q00, x01), q10, x11),
                     c11 = cfms_d(cfms_d(r11, q01, x01), q11, x11);
    const cx<double> detC = cfms_d(c00 * c11, c01, c01);
    const cx<double> iC = cinv(detC);
    if (!(p00.re > 0.0) || !(detP.re * p00.re + detP.im * p00.im > 0.0) || !(c00.re > 0.0) ||
        !(detC.re * c00.re + detC.im * c00.im > 0.0))
        bad = true;
    const cx<double> ci00 = c11 * iC, ci01 = mk<double>(0.0, 0.0) - c01 * iC, ci11 = c00 * iC;
    const cx<double> wgt = wz * f * crsqrt(detP) * crsqrt(detC);
    ko[0] = cfms_d(ko[0], wgt, cfma_d(x00 * ci00, x01, ci01));
    ko[1] = cfms_d(ko[1], wgt, cfma_d(x00 * ci01, x01, ci11));
    ko[2] = cfms_d(ko[2], wgt, cfma_d(x10 * ci00, x11, ci01));
    ko[3] = cfms_d(ko[3], wgt, cfma_d(x10 * ci01, x11, ci11));
}

// one CTA per (pattern, chunk of its contour points): per point t_l the inverse G (the
// forward's sweep), K block by block, then Re(-1/2 t (s G - G K G)) added to the chunk's own slot
// (packed upper triangle of 2n x 2n; every entry has one owner thread, so the sums over l are in a
// fixed order).
//
// Bound by the FP64 pipe (two lanes a clock and SM, whatever the number of active lanes): what counts
// is the number of FP64 instructions a warp issues.  LOW (orders 1 and 2): a diagonal block's groups
// over 16 lanes and the off-diagonal blocks, a single group each, in warps of their own; with a thread
// a block every warp held a diagonal block and went through its n groups nearly alone.  Products are
// fused, and of the second one, Re(h G T) with h multiplied into T first, only the real part is formed.
// Measured on a GB300, 128 patterns of 8 to 16 clicks at order 2: 37.6 -> 10.4 ms (with 16 instead of two
// CTAs an SM to choose from, so that the largest patterns do not finish alone).
template <bool LOW>
__global__ void __launch_bounds__(kMinorThreads, LOW ? 2 : 1) approx_minors_adjoint_kernel(
    int M, const double *__restrict__ O, const uint64_t *__restrict__ pats, int order, int chunks_per,
    ApproxPlan pl, const double *__restrict__ unit_B, double *__restrict__ slots, size_t sst,
    int *__restrict__ flags) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ int modes[128];
    __shared__ int s_bad;
    __shared__ double s_zs[2];
    const int t = threadIdx.x;
    const int p = blockIdx.x / chunks_per, c = blockIdx.x - p * chunks_per;
    const int n = pl.pat_n[p], L = pl.pat_L[p];
    if (n <= 0 || L <= 0 || *pl.overflow) return;
    const int N = 2 * n;
    cx<double> *const Gs = (cx<double> *)smem_raw;      // swept matrix, then four staged columns
    cx<double> *const Kp = Gs + sym(N) + 4 * N;          // K, packed upper triangle
    cx<double> *const Tp = Kp + sym(N);                  // N x kPanel columns of K G
    double *const slot = slots + (size_t)blockIdx.x * sst;
    for (int f = t; f < sym(N); f += kMinorThreads) slot[f] = 0.0;
    if (t == 0) {
        const uint64_t wlo = pats[2 * p], whi = pats[2 * p + 1];
        int q = 0;
        for (int i = 0; i < M; ++i) {
            const uint64_t w = i < 64 ? wlo : whi;
            if (w >> (i & 63) & 1ull) modes[q++] = i;
        }
        s_bad = 0;
    }
    __syncthreads();
    const int U = L / 2 + 1;
    const int l0 = (int)((long long)c * U / chunks_per), l1 = (int)((long long)(c + 1) * U / chunks_per);
    const double rho = pl.pat_rho[p];
    const int nb = n * (n + 1) / 2;
    bool bad = false;
    for (int l = l0; l < l1; ++l) {
        double sn, cs;
        sincospi(2.0 * (double)l / (double)L, &sn, &cs);
        sn *= rho;
        cs *= rho;
        sweep_inverse<double, true>(M, O, modes, n, cs, sn, Gs, &s_bad, s_zs);
        const size_t uo = ((size_t)pl.unit_off[p] + l) * 2 * (kMaxOrder + 1);
        cx<double> cb[kMaxOrder + 1];
        cx<double> sl = mk<double>(0.0, 0.0);
        for (int w = 0; w <= kMaxOrder; ++w) {
            cb[w] = mk<double>(unit_B[uo + 2 * w], unit_B[uo + 2 * w + 1]);
            sl = sl + cb[w] * mk<double>(pl.unit_D[uo + 2 * w], pl.unit_D[uo + 2 * w + 1]);
        }
        const cx<double> zs = mk<double>(s_zs[0], s_zs[1]);
        if constexpr (LOW) {
            const cx<double> z0 = mk<double>(0.0, 0.0);
            const cx<double> w1 = cb[1] * zs, w2 = cb[2] * zs;
            const int lane = t & 31, nd = (n + 1) >> 1, no = (n * (n - 1) / 2 + 31) >> 5;
            for (int task = t >> 5; task < nd + no; task += kMinorThreads / 32) {
                if (task < nd) {
                    // two diagonal blocks a warp: group q of block a is {a}, then {x, a} for the other modes
                    const int a = 2 * task + (lane >> 4), total = order > 1 ? n : 1;
                    cx<double> k00 = z0, k01 = z0, k11 = z0;
                    if (a < n)
                        for (int q = lane & 15; q < total; q += 16) {
                            if (q == 0) {
                                const int m[1] = {a};
                                diag_leaf<0>(Gs, N, m, w1, k00, k01, k11, bad);
                            } else {
                                const int m[2] = {q - 1 < a ? q - 1 : q, a};
                                diag_leaf<1>(Gs, N, m, w2, k00, k01, k11, bad);
                            }
                        }
#pragma unroll
                    for (int off = 8; off; off >>= 1) {
                        k00.re += __shfl_xor_sync(0xffffffffu, k00.re, off);
                        k00.im += __shfl_xor_sync(0xffffffffu, k00.im, off);
                        k01.re += __shfl_xor_sync(0xffffffffu, k01.re, off);
                        k01.im += __shfl_xor_sync(0xffffffffu, k01.im, off);
                        k11.re += __shfl_xor_sync(0xffffffffu, k11.re, off);
                        k11.im += __shfl_xor_sync(0xffffffffu, k11.im, off);
                    }
                    if (a < n && (lane & 15) == 0) {
                        Kp[pidx(N, 2 * a, 2 * a)] = k00;
                        Kp[pidx(N, 2 * a, 2 * a + 1)] = k01;
                        Kp[pidx(N, 2 * a + 1, 2 * a + 1)] = k11;
                    }
                } else {
                    const int r = (task - nd) * 32 + lane;  // the r-th pair a < b
                    if (r < n * (n - 1) / 2) {
                        int m[2];
                        unrank_pair(r, m[0], m[1]);
                        cx<double> ko[4] = {z0, z0, z0, z0};
                        if (order > 1) off_leaf<0>(Gs, N, m, w2, ko, bad);
                        Kp[pidx(N, 2 * m[0], 2 * m[1])] = ko[0];
                        Kp[pidx(N, 2 * m[0], 2 * m[1] + 1)] = ko[1];
                        Kp[pidx(N, 2 * m[0] + 1, 2 * m[1])] = ko[2];
                        Kp[pidx(N, 2 * m[0] + 1, 2 * m[1] + 1)] = ko[3];
                    }
                }
            }
        } else {
        // one 2 x 2 block (a, b) a warp at a time: its lanes split the block's groups W = V + {a, b}: V over the
        // other modes, sizes ascending and each size in colex order (neighbouring lanes mostly
        // share the size, so the leaf code rarely diverges); partial sums meet in a fixed
        // shuffle tree.  Every thread runs every round (the shuffles take the whole warp).
        constexpr int gw = 32;
        const int seg = t / gw, sg = t - seg * gw, nseg = kMinorThreads / gw;
        const int rounds = (nb + nseg - 1) / nseg;
        for (int rd = 0; rd < rounds; ++rd) {
            const int blk = rd * nseg + seg;
            const bool live = blk < nb;
            int a = 0, rem = live ? blk : 0;
            while (rem >= n - a) { rem -= n - a; ++a; }
            const int b = a + rem;
            const bool dg = a == b;
            const int others = dg ? n - 1 : n - 2, base = dg ? 1 : 2;   // |W| = |V| + base
            const int vmax = order - base < others ? order - base : others;
            int cnt[4], total = 0;
            for (int v = 0; v < 4; ++v) {
                cnt[v] = live && v <= vmax ? binom_small(others, v) : 0;
                total += cnt[v];
            }
            const cx<double> z0 = mk<double>(0.0, 0.0);
            cx<double> acc[4] = {z0, z0, z0, z0};
            for (int q = sg; q < total; q += gw) {
                int v = 0, r = q;
                while (r >= cnt[v]) { r -= cnt[v]; ++v; }
                int x[3] = {r, 0, 0};
                if (v == 2) unrank_pair(r, x[0], x[1]);
                else if (v == 3) unrank_triple(r, x[0], x[1], x[2]);
                // ranks among the other modes -> modes (a, then b, skipped)
                for (int i = 0; i < v; ++i) {
                    int y = x[i];
                    if (y >= a) ++y;
                    if (!dg && y >= b) ++y;
                    x[i] = y;
                }
                const cx<double> wz = cb[v + base] * zs;
                if (dg) {
                    if (v == 0) {
                        const int m[1] = {a};
                        diag_leaf<0>(Gs, N, m, wz, acc[0], acc[1], acc[2], bad);
                    } else if (v == 1) {
                        const int m[2] = {x[0], a};
                        diag_leaf<1>(Gs, N, m, wz, acc[0], acc[1], acc[2], bad);
                    } else if (v == 2) {
                        const int m[3] = {x[0], x[1], a};
                        diag_leaf<2>(Gs, N, m, wz, acc[0], acc[1], acc[2], bad);
                    } else {
                        const int m[4] = {x[0], x[1], x[2], a};
                        diag_leaf<3>(Gs, N, m, wz, acc[0], acc[1], acc[2], bad);
                    }
                } else {
                    if (v == 0) {
                        const int m[2] = {a, b};
                        off_leaf<0>(Gs, N, m, wz, acc, bad);
                    } else if (v == 1) {
                        const int m[3] = {x[0], a, b};
                        off_leaf<1>(Gs, N, m, wz, acc, bad);
                    } else {
                        const int m[4] = {x[0], x[1], a, b};
                        off_leaf<2>(Gs, N, m, wz, acc, bad);
                    }
                }
            }
#pragma unroll
            for (int i = 0; i < 4; ++i)
                for (int off = gw >> 1; off; off >>= 1) {
                    acc[i].re += __shfl_xor_sync(0xffffffffu, acc[i].re, off);
                    acc[i].im += __shfl_xor_sync(0xffffffffu, acc[i].im, off);
                }
            if (live && sg == 0) {
                if (dg) {
                    Kp[pidx(N, 2 * a, 2 * a)] = acc[0];
                    Kp[pidx(N, 2 * a, 2 * a + 1)] = acc[1];
                    Kp[pidx(N, 2 * a + 1, 2 * a + 1)] = acc[2];
                } else {
                    Kp[pidx(N, 2 * a, 2 * b)] = acc[0];
                    Kp[pidx(N, 2 * a, 2 * b + 1)] = acc[1];
                    Kp[pidx(N, 2 * a + 1, 2 * b)] = acc[2];
                    Kp[pidx(N, 2 * a + 1, 2 * b + 1)] = acc[3];
                }
            }
        }
        }
        __syncthreads();
        // Re(-1/2 t (s G - G K G)) on the upper triangle, kPanel columns at a time (Gs = -G)
        const cx<double> ht = mk<double>(-0.5 * cs, -0.5 * sn), hs = ht * sl;
        for (int j0 = 0; j0 < N; j0 += kPanel) {
            for (int f = t; f < N * kPanel; f += kMinorThreads) {
                const int r = f / kPanel, j = j0 + (f - r * kPanel);
                cx<double> acc = mk<double>(0.0, 0.0);
                if (j < N)
                    for (int q = 0; q < N; ++q) acc = cfma_d(acc, Kp[pidx_any(N, r, q)], Gs[pidx_any(N, q, j)]);
                Tp[f] = ht * acc;
            }
            __syncthreads();
            for (int f = t; f < N * kPanel; f += kMinorThreads) {
                const int i = f / kPanel, jj = f - i * kPanel, j = j0 + jj;
                if (j >= N || i > j) continue;
                double y = 0.0;
                for (int q = 0; q < N; ++q) {
                    const cx<double> g = Gs[pidx_any(N, i, q)], x = Tp[q * kPanel + jj];
                    y = fma(g.re, x.re, fma(-g.im, x.im, y));
                }
                const cx<double> g = Gs[pidx(N, i, j)];
                slot[pidx(N, i, j)] -= fma(hs.re, g.re, fma(-hs.im, g.im, y));
            }
            __syncthreads();
        }
    }
    if (bad) s_bad = 1;
    __syncthreads();
    if (t == 0 && s_bad) atomicOr(flags + p, 1);
}

// per pattern: F_p = w_p * (sum of its chunk slots, in chunk order), dense 2n x 2n at stride
// fst; zero for a pattern whose forward failed (status other than ok / fit fallback, or no
// sector) or whose adjoint met a non-positive pivot
__global__ void approx_grad_finalize_kernel(int chunks_per, ApproxPlan pl, const double *__restrict__ slots,
                                            size_t sst, const double *__restrict__ w,
                                            const double *__restrict__ logP, const int32_t *__restrict__ status,
                                            const int *__restrict__ flags, double *__restrict__ F, size_t fst) {
    const int p = blockIdx.x;
    const int n = pl.pat_n[p];
    if (n <= 0) return;
    const int D = 2 * n;
    const int st = status[p];
    const bool ok = (st == GBS_OK || st == GBS_E_FIT) && !flags[p] && isfinite(logP[p]);
    for (int f = threadIdx.x; f < D * D; f += blockDim.x) {
        const int i = f / D, j = f - i * D;
        double v = 0.0;
        if (ok) {
            const int q = pidx_any(D, i, j);
            for (int c = 0; c < chunks_per; ++c) v += slots[((size_t)p * chunks_per + c) * sst + q];
            v *= w[p];
        }
        F[(size_t)p * fst + f] = v;
    }
}

__global__ void approx_grad_status_kernel(int n_pat, const int32_t *__restrict__ st_in,
                                          const int *__restrict__ flags, int32_t *__restrict__ st_out) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < n_pat) st_out[p] = (st_in[p] == GBS_OK || st_in[p] == GBS_E_FIT) && flags[p] ? GBS_E_NOT_SPD : st_in[p];
}

size_t align256(size_t x) { return (x + 255) / 256 * 256; }

struct ApproxOffsets {
    size_t counter, total, overflow, info, counter2, pat_n, pat_L, pat_rho, unit_off, unit_flag, sec_off, pat_max,
        pat_ld, unit_D, sec_D, sec_part, sec_slow, counter3, counter4, end;
};

ApproxOffsets approx_offsets(int n_pat, long long units, long long secs = 0) {
    ApproxOffsets o;
    o.counter = 0;
    o.total = 8;
    o.overflow = 16;
    o.info = 24;       // 6 long long
    o.counter2 = 72;   // the CTA-pair minors kernel's work counter
    o.counter3 = 80;   // the slow fits' list length and its work counter
    o.counter4 = 96;   // the work counter of the patterns with an SM to themselves
    o.pat_n = align256(104);
    o.pat_L = align256(o.pat_n + 4 * (size_t)n_pat);
    o.pat_rho = align256(o.pat_L + 4 * (size_t)n_pat);
    o.unit_off = align256(o.pat_rho + 8 * (size_t)n_pat);
    o.unit_flag = align256(o.unit_off + 8 * ((size_t)n_pat + 1));
    o.sec_off = align256(o.unit_flag + 4 * (size_t)n_pat);
    o.pat_max = align256(o.sec_off + 8 * ((size_t)n_pat + 1));
    o.pat_ld = align256(o.pat_max + 8 * (size_t)n_pat);
    o.unit_D = align256(o.pat_ld + 8 * (size_t)kNumShift * n_pat);
    o.sec_D = align256(o.unit_D + 8 * 2 * (kMaxOrder + 1) * (size_t)units);
    o.sec_part = align256(o.sec_D + 8 * (kMaxOrder + 1) * (size_t)secs);
    o.sec_slow = align256(o.sec_part + 8 * (size_t)secs);
    o.end = o.sec_slow + 4 * (size_t)secs;
    return o;
}

ApproxPlan approx_plan_from(void *ws, int n_pat, long long units = 0, long long secs = 0) {
    ApproxOffsets o = approx_offsets(n_pat, units, secs);
    char *b = (char *)ws;
    ApproxPlan pl;
    pl.total = (long long *)(b + o.total);
    pl.overflow = (int *)(b + o.overflow);
    pl.pat_n = (int *)(b + o.pat_n);
    pl.pat_L = (int *)(b + o.pat_L);
    pl.pat_rho = (double *)(b + o.pat_rho);
    pl.unit_off = (long long *)(b + o.unit_off);
    pl.unit_flag = (int *)(b + o.unit_flag);
    pl.unit_D = (double *)(b + o.unit_D);
    pl.info = (long long *)(b + o.info);
    pl.sec_off = (long long *)(b + o.sec_off);
    pl.pat_max = (double *)(b + o.pat_max);
    pl.sec_D = (double *)(b + o.sec_D);
    pl.sec_part = (double *)(b + o.sec_part);
    pl.sec_slow = (uint32_t *)(b + o.sec_slow);
    pl.slow = (unsigned long long *)(b + o.counter3);
    return pl;
}

// the plan's launches: the factorisations by classes of sizes (CTAs an SM by their shared memory: 16,
// 6, 3, 1; a class beyond M clicks is empty), the plan, the offsets
int launch_plan(gbs_ctx *ctx, int M, const double *O, const uint64_t *pats, int n_pat, int n_limit, long long cap,
                int n_single, const ApproxPlan &pl) {
    double *ld = (double *)((char *)ctx->ws + approx_offsets(n_pat, 0).pat_ld);
    const int to[] = {20, 40, 64, kApproxMaxN};
    int from = 1;
    for (int c = 0; c < 4 && from <= M; ++c) {
        const size_t smem = sizeof(double) * (size_t)sym(2 * (to[c] < M ? to[c] : M));
        GBS_CUDA(ctx, cudaFuncSetAttribute(approx_logdet_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        for (int p0 = 0; p0 < n_pat; p0 += 1 << 20) {
            const int np = n_pat - p0 < 1 << 20 ? n_pat - p0 : 1 << 20;
            approx_logdet_kernel<<<dim3(np, kNumShift), kLogdetThreads, smem, ctx->stream>>>(
                M, O, pats + 2 * (size_t)p0, n_limit, from, to[c], ld + (size_t)kNumShift * p0);
        }
        from = to[c] + 1;
    }
    GBS_CUDA(ctx, cudaGetLastError());
    approx_plan_kernel<<<(n_pat + kPlanThreads / 32 - 1) / (kPlanThreads / 32), kPlanThreads, 0, ctx->stream>>>(
        M, pats, n_pat, n_limit, ld, pl);
    approx_scan_kernel<<<1, kScanThreads, 0, ctx->stream>>>(n_pat, cap, n_single, pl);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}

// one launch of the one-CTA minors kernel, for the patterns of n_from to n_to clicks
template <typename R, int TH>
int launch_minors(gbs_ctx *ctx, int M, const double *O, const uint64_t *pats, int n_pat, int order, int n_from, int n_to,
                  size_t counter, const ApproxPlan &pl) {
    // the packed inverse and four staged pivot columns, or the pair phases' items
    // (15 entries each, at least n - 1 of them, up to 8 n while the CTAs per SM stay)
    // (the largest over the range: the kernel sizes each pattern's items from its own n,
    // and the floor to whole items makes the entries fall by up to 14 between some n)
    int ent = sym(2 * n_to) + 2 * InvOps<R>::rows * n_to;  // FP32: no pair phases
    if constexpr (!std::is_same<R, float>::value)
        for (int m = n_from > 1 ? n_from : 1; m <= n_to; ++m) {
            const int e = minor_smem_entries(m, (int)sizeof(cx<R>), MinorPrec<R>::min_blocks);
            if (e > ent) ent = e;
        }
    const size_t minor_smem = sizeof(cx<R>) * (size_t)ent;
    const auto kernel = approx_minors_kernel<R, TH>;
    GBS_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)minor_smem));
    int nb = 0;
    GBS_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, kernel, TH, minor_smem));
    if (nb < 1) nb = 1;
    kernel<<<ctx->num_sms * nb, TH, minor_smem, ctx->stream>>>(M, O, pats, n_pat, order, n_from, n_to, ent,
                                                               (unsigned long long *)((char *)ctx->ws + counter), pl);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}

template <typename R>
int run_approx(gbs_ctx *ctx, int M, const double *O, const double *logdet, const uint64_t *pats,
               int n_pat, int order, double *logP, double *kappa, double *err_bound, int32_t *status,
               double *curves = nullptr, int curve_K = -1, int curve_n = -1, int n_limit = -1) {
    // patterns up to this size are taken: the packed inverse must fit in one CTA's shared
    // memory, or (FP64 and float-float) in a CTA pair's; a caller may lower it
    const int n_cap = MinorPrec<R>::pair ? kPairMaxN : MinorPrec<R>::nmax;
    const int nmax_smem = n_limit > 0 && n_limit < n_cap ? n_limit : n_cap;
    const int n_single = MinorPrec<R>::pair && ctx->pair_from - 1 < MinorPrec<R>::nmax ? ctx->pair_from - 1
                                                                                       : MinorPrec<R>::nmax;
    static_assert(kMaxK + 1 <= 4096, "sector table");
    if (!ctx->ws || ctx->ws_bytes < approx_offsets(n_pat, 0).end) {
        int st = gbs_ws_ensure(ctx, approx_offsets(n_pat, 0).end);
        if (st) return st;
    }
    ApproxPlan pl = approx_plan_from(ctx->ws, n_pat);
    const long long nocap = 1ll << 62;  // sized on the host below
    int pst = launch_plan(ctx, M, O, pats, n_pat, nmax_smem, nocap, n_single, pl);
    if (pst) return pst;
    // size the workspace and the kernels' shared memory from one readback (units,
    // largest n, largest L, sectors); re-plan if the workspace had to grow
    GBS_CUDA(ctx, cudaMemcpyAsync(ctx->pinned, pl.info, 40, cudaMemcpyDeviceToHost, ctx->stream));
    GBS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    const long long units = ((long long *)ctx->pinned)[0], secs = ((long long *)ctx->pinned)[3];
    const int nmax = (int)((long long *)ctx->pinned)[1], Lmax = (int)((long long *)ctx->pinned)[2];
    const int nsmall = (int)((long long *)ctx->pinned)[4];
    const size_t need = approx_offsets(n_pat, units, secs).end;
    if (need > ctx->ws_bytes) {
        int st = gbs_ws_ensure(ctx, need);
        if (st) return st;
        pl = approx_plan_from(ctx->ws, n_pat);
        pst = launch_plan(ctx, M, O, pats, n_pat, nmax_smem, nocap, n_single, pl);
        if (pst) return pst;
    }
    pl = approx_plan_from(ctx->ws, n_pat, units, secs);
    GBS_CUDA(ctx, cudaMemsetAsync(ctx->ws, 0, 8, ctx->stream));  // work counters
    GBS_CUDA(ctx, cudaMemsetAsync((char *)ctx->ws + approx_offsets(n_pat, 0).counter2, 0, 32, ctx->stream));
    int st = gbs_timing_begin(ctx);
    if (st) return st;
    // one CTA a unit: up to n_two clicks two of them (of 256 threads) share an SM; above, the SM
    // holds one, of 512 threads where the inverse is all that counts
    int n_two = nsmall;
    if (std::is_same<R, ff>::value)
        while (n_two > 0 && !minor_shares_sm(n_two)) --n_two;
    if (nsmall > n_two) {
        const size_t c4 = approx_offsets(n_pat, 0).counter4;
        if constexpr (std::is_same<R, ff>::value) {
            if (order <= 2) st = launch_minors<R, kWideThreads>(ctx, M, O, pats, n_pat, order, n_two + 1, nsmall, c4, pl);
            else st = launch_minors<R, kMinorThreads>(ctx, M, O, pats, n_pat, order, n_two + 1, nsmall, c4, pl);
        }
        if (st) return st;
    }
    if (n_two >= 0) {  // empty patterns too: their sector tables come from here
        st = launch_minors<R, kMinorThreads>(ctx, M, O, pats, n_pat, order, 0, n_two, 0, pl);
        if (st) return st;
    }
    if constexpr (MinorPrec<R>::pair) if (nmax > n_single) {
        // half of the packed inverse, and the staged columns or the pair phases' items
        constexpr int rows2 = 2 * InvOps<R>::rows;
        const int pent = pair_part_entries(2 * nmax) + (rows2 * nmax > 15 * (nmax - 2) ? rows2 * nmax : 15 * (nmax - 2));
        const size_t pair_smem = sizeof(cx<R>) * (size_t)pent;
        const bool wide = std::is_same<R, ff>::value && order <= 2;
        auto kernel = approx_minors_pair_kernel<R, kMinorThreads>;
        if constexpr (std::is_same<R, ff>::value)
            if (wide) kernel = approx_minors_pair_kernel<R, kWideThreads>;
        GBS_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pair_smem));
        kernel<<<(ctx->num_sms / 2) * 2, wide ? kWideThreads : kMinorThreads, pair_smem, ctx->stream>>>(
            M, O, pats, n_pat, order, n_single, pent,
            (unsigned long long *)((char *)ctx->ws + approx_offsets(n_pat, 0).counter2), pl);
        GBS_CUDA(ctx, cudaGetLastError());
    }
    st = gbs_timing_end(ctx);
    if (st) return st;
    const size_t dft_smem = sizeof(double) * 2 * (size_t)Lmax;
    GBS_CUDA(ctx, cudaFuncSetAttribute(approx_dft_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)dft_smem));
    const int dft_most = ((order + 1) * Lmax + kDftThreads - 1) / kDftThreads, dft_want = (8 * ctx->num_sms + n_pat - 1) / n_pat;
    const unsigned dft_y = (unsigned)(dft_want < dft_most ? dft_want : dft_most > 0 ? dft_most : 1);
    approx_dft_kernel<<<dim3((unsigned)n_pat, dft_y), kDftThreads, dft_smem, ctx->stream>>>(order, pl);
    GBS_CUDA(ctx, cudaGetLastError());
    const long long want = (secs + kSecThreads / 32 - 1) / (kSecThreads / 32);
    const int fit_blocks = (int)(want < (long long)ctx->num_sms * 16 ? (want > 0 ? want : 1) : ctx->num_sms * 16);
    if (curves) {
        // one pattern: its clicks (read back above) must be the caller's row width - 1
        if (nmax != curve_n)
            return gbs_fail(ctx, GBS_E_INVALID, "gbs_approx_sector_curves: the pattern has %d clicks, not n = %d",
                            nmax, curve_n);
        GBS_CUDA(ctx, cudaMemsetAsync(curves, 0, sizeof(double) * (size_t)(curve_K + 1) * (curve_n + 1),
                                      ctx->stream));
    }
    const double eps = MinorPrec<R>::sector_eps;
    if (curves) {
        approx_sector_fit_kernel<<<fit_blocks, kSecThreads, 0, ctx->stream>>>(n_pat, order, eps, pl, curves, curve_K);
    } else if (secs > 0) {
        if (order == 1) launch_fit_lanes<1>(ctx, secs, n_pat, eps, pl);
        else if (order == 2) launch_fit_lanes<2>(ctx, secs, n_pat, eps, pl);
        else if (order == 3) launch_fit_lanes<3>(ctx, secs, n_pat, eps, pl);
        else launch_fit_lanes<4>(ctx, secs, n_pat, eps, pl);
        GBS_CUDA(ctx, cudaGetLastError());
        approx_fit_slow_kernel<<<ctx->num_sms * kSlowCtas, kSlowThreads, 0, ctx->stream>>>(n_pat, order, pl);
    }
    GBS_CUDA(ctx, cudaGetLastError());
    if (curves) {
        const long long tot = (long long)(curve_K + 1) * (nmax + 1);
        approx_curve_scale_kernel<<<(unsigned)((tot + 127) / 128), 128, 0, ctx->stream>>>(curve_K, nmax, logdet, pl,
                                                                                          curves);
        GBS_CUDA(ctx, cudaGetLastError());
    }
    approx_sum_kernel<<<(n_pat + kSumThreads / 32 - 1) / (kSumThreads / 32), kSumThreads, 0, ctx->stream>>>(
        n_pat, logdet, MinorPrec<R>::floor_flag ? MinorPrec<R>::sector_eps : 0.0, pl, logP, kappa, err_bound, status);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}

}  // namespace

int approx_prob(gbs_ctx *ctx, int M, const double *O, const double *logdet, const uint64_t *patterns,
                int n_pat, int order, int precision, double *logP, double *kappa, double *err_bound,
                int32_t *status) {
    if (order < 1 || order > kMaxOrder)
        return gbs_fail(ctx, GBS_E_INVALID, "gbs_prob: approximation order %d not in 1..%d", order, kMaxOrder);
    if (precision == GBS_FP64)
        return run_approx<double>(ctx, M, O, logdet, patterns, n_pat, order, logP, kappa, err_bound, status);
    if (precision == GBS_FP32_SPLIT)
        return run_approx<float>(ctx, M, O, logdet, patterns, n_pat, order, logP, kappa, err_bound, status);
    if (precision == GBS_FF)
        return run_approx<ff>(ctx, M, O, logdet, patterns, n_pat, order, logP, kappa, err_bound, status);
    return gbs_fail(ctx, GBS_E_INVALID, "gbs_prob: the approximation runs in FP64, float-float or the FP32 split");
}

int approx_sector_curves(gbs_ctx *ctx, int M, const double *O, const double *logdet, const uint64_t *pattern,
                         int n, int order, int precision, int K, double *curves, double *logP, int32_t *status) {
    if (order < 1 || order > kMaxOrder)
        return gbs_fail(ctx, GBS_E_INVALID, "gbs_approx_sector_curves: order %d not in 1..%d", order, kMaxOrder);
    if (n < 1 || n > M || K < 0)
        return gbs_fail(ctx, GBS_E_INVALID, "gbs_approx_sector_curves: bad sizes (n=%d, M=%d, K=%d)", n, M, K);
    if (precision == GBS_FP64)
        return run_approx<double>(ctx, M, O, logdet, pattern, 1, order, logP, nullptr, nullptr, status, curves, K, n);
    if (precision == GBS_FF)
        return run_approx<ff>(ctx, M, O, logdet, pattern, 1, order, logP, nullptr, nullptr, status, curves, K, n);
    return gbs_fail(ctx, GBS_E_INVALID, "gbs_approx_sector_curves: the curves run in FP64 or float-float");
}

int approx_grad(gbs_ctx *ctx, int M, const double *O, const double *logdet, const uint64_t *pats, int n_pat,
                int order, const double *w, double *dsq, double *logP, int32_t *status) {
    if (order < 1 || order > kMaxOrder)
        return gbs_fail(ctx, GBS_E_INVALID, "gbs_grad_approx: order %d not in 1..%d", order, kMaxOrder);
    // every pattern must be valid with at most kGradApproxMaxN clicks: checked on the host
    // from a copy of the pattern words (one small readback)
    const size_t pb = (size_t)n_pat * 16;
    uint64_t *hp = (uint64_t *)malloc(pb + 16);
    if (!hp) return gbs_fail(ctx, GBS_E_NOMEM, "gbs_grad_approx: host buffer");
    cudaError_t ce = cudaMemcpyAsync(hp, pats, pb, cudaMemcpyDeviceToHost, ctx->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(ctx->stream);
    if (ce != cudaSuccess) {
        free(hp);
        GBS_CUDA(ctx, ce);
    }
    int n_max = 0;
    for (int p = 0; p < n_pat; ++p) {
        const uint64_t lo = hp[2 * p], hi = hp[2 * p + 1];
        const int n = __builtin_popcountll(lo) + __builtin_popcountll(hi);
        const bool out_of_range =
            (M < 64 && (lo >> M)) || (M <= 64 && hi) || (M > 64 && M < 128 && (hi >> (M - 64)));
        if (n > kGradApproxMaxN || out_of_range) {
            free(hp);
            return gbs_fail(ctx, GBS_E_INVALID,
                            "gbs_grad_approx: pattern %d has %d clicks (at most %d) or a detector >= M", p, n,
                            kGradApproxMaxN);
        }
        n_max = n > n_max ? n : n_max;
    }
    free(hp);
    // kept across the forward: its log P and status, the adjoint's flags
    const size_t np_ = (size_t)n_pat;
    const size_t o_lp = 0, o_st = align256(8 * np_), o_fl = o_st + align256(4 * np_), keep = o_fl + align256(4 * np_);
    int st = gbs_aux_ensure(ctx, keep, 0);
    if (st) return st;
    {
        char *b = (char *)ctx->aux;
        st = run_approx<double>(ctx, M, O, logdet, pats, n_pat, order, (double *)(b + o_lp), nullptr, nullptr,
                                (int32_t *)(b + o_st), nullptr, -1, -1, kGradApproxMaxN);
        if (st) return st;
    }
    // the plan's sizes (units, largest n, largest L, sectors)
    ApproxPlan pl = approx_plan_from(ctx->ws, n_pat);
    GBS_CUDA(ctx, cudaMemcpyAsync(ctx->pinned, pl.info, 32, cudaMemcpyDeviceToHost, ctx->stream));
    GBS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    const long long units = ((long long *)ctx->pinned)[0], secs = ((long long *)ctx->pinned)[3];
    const int Lmax = (int)((long long *)ctx->pinned)[2];
    pl = approx_plan_from(ctx->ws, n_pat, units, secs);
    // contour points of a pattern split over chunks_per CTAs: about 16 CTAs per SM in all (a pattern's
    // work goes with the fourth power of its clicks, so a wave or two would wait for the largest)
    const int want = (16 * ctx->num_sms + n_pat - 1) / n_pat;
    const int chunks_per = want < 1 ? 1 : (want > 64 ? 64 : want);
    const int Nm = 2 * (n_max > 0 ? n_max : 1);
    const size_t sst = (size_t)sym(Nm), fst = (size_t)Nm * Nm, N2 = (size_t)(2 * M) * (2 * M);
    const size_t o_sb = keep, o_ub = o_sb + align256(8 * (kMaxOrder + 1) * (size_t)secs),
                 o_sl = o_ub + align256(16 * (kMaxOrder + 1) * (size_t)units),
                 o_F = o_sl + align256(8 * np_ * chunks_per * sst), o_H = o_F + align256(8 * np_ * fst),
                 o_T1 = o_H + align256(8 * N2), o_T2 = o_T1 + align256(8 * N2), o_sw = o_T2 + align256(8 * N2),
                 total = o_sw + 256;
    st = gbs_aux_ensure(ctx, total, keep);
    if (st) return st;
    char *b = (char *)ctx->aux;
    double *lp_i = (double *)(b + o_lp);
    int32_t *st_i = (int32_t *)(b + o_st);
    int *flags = (int *)(b + o_fl);
    double *sec_B = (double *)(b + o_sb), *unit_B = (double *)(b + o_ub), *slots = (double *)(b + o_sl);
    double *F = (double *)(b + o_F), *H = (double *)(b + o_H), *T1 = (double *)(b + o_T1), *T2 = (double *)(b + o_T2),
           *sw = (double *)(b + o_sw);
    GBS_CUDA(ctx, cudaMemsetAsync(flags, 0, 4 * np_, ctx->stream));
    if (secs > 0) {
        const long long wsec = (secs + kSecThreads / 32 - 1) / (kSecThreads / 32);
        const int fit_blocks = (int)(wsec < (long long)ctx->num_sms * 16 ? wsec : ctx->num_sms * 16);
        approx_fit_adjoint_kernel<<<fit_blocks, kSecThreads, 0, ctx->stream>>>(n_pat, order, pl, sec_B);
        GBS_CUDA(ctx, cudaGetLastError());
        const size_t dft_smem = sizeof(double) * 2 * (size_t)(Lmax > 0 ? Lmax : 1);
        GBS_CUDA(ctx, cudaFuncSetAttribute(approx_dft_adjoint_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                           (int)dft_smem));
        approx_dft_adjoint_kernel<<<n_pat, kDftThreads, dft_smem, ctx->stream>>>(order, pl, sec_B, unit_B);
        GBS_CUDA(ctx, cudaGetLastError());
    }
    if (n_max > 0) {
        // swept matrix + four staged columns, K, one panel of K G
        const size_t smem = sizeof(cx<double>) * (2 * sst + 4 * (size_t)Nm + (size_t)Nm * kPanel);
        const auto adjoint = order <= 2 ? approx_minors_adjoint_kernel<true> : approx_minors_adjoint_kernel<false>;
        GBS_CUDA(ctx, cudaFuncSetAttribute(adjoint, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
        adjoint<<<(unsigned)(n_pat * chunks_per), kMinorThreads, smem, ctx->stream>>>(
            M, O, pats, order, chunks_per, pl, unit_B, slots, sst, flags);
        GBS_CUDA(ctx, cudaGetLastError());
        approx_grad_finalize_kernel<<<n_pat, 256, 0, ctx->stream>>>(chunks_per, pl, slots, sst, w, lp_i, st_i, flags,
                                                                   F, fst);
        GBS_CUDA(ctx, cudaGetLastError());
    }
    st = grad_chain_sigma(ctx, M, O, pats, n_pat, F, fst, w, H, T1, T2, sw, dsq);
    if (st) return st;
    if (logP) GBS_CUDA(ctx, cudaMemcpyAsync(logP, lp_i, 8 * np_, cudaMemcpyDeviceToDevice, ctx->stream));
    if (status) {
        // a pattern the adjoint could not differentiate reports GBS_E_NOT_SPD
        approx_grad_status_kernel<<<(n_pat + 255) / 256, 256, 0, ctx->stream>>>(n_pat, st_i, flags, status);
        GBS_CUDA(ctx, cudaGetLastError());
    }
    return GBS_OK;
}
