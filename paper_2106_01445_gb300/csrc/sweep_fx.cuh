// The 128-bit fixed-point sweep (GBS_FX), its own kernel: the unit / sub-unit decomposition of
// sweep.cu with every matrix in 30-bit limbs (fl.cuh) from the gather to the register bottom.
//
// One CTA of 128 threads takes a unit: the included prefix modes are eliminated, the 2^s sub-units
// are the leaves of an include/exclude tree over the unit's trailing block, and each sub-unit is
// expanded L = 7 levels breadth first to one two-mode node a thread.
//
// What bounds it.  The IMAD.WIDE pipe (27 lanes per SM clock) and the latency between the CTA's
// barriers: three CTAs of four warps share an SM (shared memory), and a level is three phases.
//  * A pivot is two lanes' work (p00^{-1/2} and det^{-1/2} side by side), whose second halves run the
//    same two products on different operands (b = det^{-1/2} sqrt(p00) on the even lane, c and the
//    child's prefactor on the odd one) instead of four in a row on one lane.
//  * A prefix or tree pivot is computed by the warps that hold rows only (one warp up to 32 rows),
//    not by all four, and its prefix factor by one thread in integers: the double-double products
//    that every thread repeated kept the FP64 pipe (2 lanes a clock) 12% busy.
//  * A sub-unit ends with a sum inside each warp, aligned to the warp's own exponent, and no
//    barrier; the unit's 8 x 4 warp sums are combined once, side by side, at the unit's end.
// Measured on a GB300, 24-mode batch of 1024 patterns (2.42e8 subsets): 29.7 -> 24.0 ms against the
// general kernel with limb levels only (37.8 ms with packed ones); one 20-click pattern 388 ->
// 336 us; the click-number distribution of 24 modes 6.4 -> 2.5 ms (its bins were double-double sums
// over all threads).
#pragma once

namespace fxk {

constexpr int B = Prec<fx>::B;
constexpr int R = kL + B;     // modes of a sub-unit's level-0 matrix
constexpr int kW = kThreads / 32;
constexpr int kSub = 1 << kS;
constexpr int kLast = kThreads - 32;  // the last warp
static_assert(2 * R <= 32, "a row of a level-0 matrix a lane");

// a node's prefactor m 2^e: m in [1, 2) as limbs at scale 117
struct node {
    fl m;
    int e;
};
__device__ __forceinline__ node node_ld(const uint32_t *b, int i) {
    const uint32_t *q = b + 5 * i;
    return node{{{(int32_t)q[0], (int32_t)q[1], (int32_t)q[2], (int32_t)q[3]}}, (int)q[4]};
}
__device__ __forceinline__ void node_st(uint32_t *b, int i, const node &v) {
    uint32_t *q = b + 5 * i;
#pragma unroll
    for (int k = 0; k < 4; ++k) q[k] = (uint32_t)v.m.w[k];
    q[4] = (uint32_t)v.e;
}
__device__ __forceinline__ node node_unit() { return node{{{0, 0, 0, 1 << 27}}, 0}; }
// p (scale 123, in [1/8, 64)) times 2^e as a node
__device__ __forceinline__ node node_norm(const fl5 &p, int e) {
    const int k = (31 - __clz(p.w[4])) - 3;  // floor(log2 p): w[4] = floor(8 p)
    const int s = 6 + k;                     // 123 -> 117, and 2^-k
    node o;
    if (s < 0 || s > 29) return node_unit();  // outside the range (a flagged pivot)
    o.m.w[0] = (int32_t)((((uint32_t)p.w[0] >> s) | ((uint32_t)p.w[1] << (30 - s))) & (uint32_t)kLimbMask);
    o.m.w[1] = (int32_t)((((uint32_t)p.w[1] >> s) | ((uint32_t)p.w[2] << (30 - s))) & (uint32_t)kLimbMask);
    o.m.w[2] = (int32_t)((((uint32_t)p.w[2] >> s) | ((uint32_t)p.w[3] << (30 - s))) & (uint32_t)kLimbMask);
    o.m.w[3] = (int32_t)(((uint32_t)p.w[3] >> s) | ((uint32_t)p.w[4] << (30 - s)));
    o.e = e + k;
    return o;
}
__device__ __forceinline__ node node_mul(const node &a, const fx &rs) {
    int64_t p[5] = {0, 0, 0, 0, 0};
    fl_mac45(p, a.m, fl5_at126(rs));
    return node_norm(fl5_carry(p), a.e);
}
// the mantissa packed, Q16.112
__device__ __forceinline__ fx node_packed(const node &a) { return fx_shr_small(fl_pack(a.m), 5); }
__device__ __forceinline__ node node_mul(const node &a, const node &b) {
    node r = node_mul(a, node_packed(b));
    r.e += b.e;
    return r;
}
__device__ __forceinline__ dd node_dd(const node &a) {
    const dd v = fx_to_dd(node_packed(a));
    const double s = ldexp(1.0, a.e);
    return dd(v.hi * s, v.lo * s);
}

// ---- shared memory ---------------------------------------------------------------------
// X and Y: source and destination of the levels in turn; the unit's prefix matrix (up to 2 kMaxN
// rows) spans X, Y, Ub and Sl before the levels start.  W: the rows U = B R^{-T} of a pivot.
constexpr int level_size(int l) { return (1 << l) * nstride(2 * (R - l)); }
constexpr int max_of(int from) {
    int m = 0;
    for (int l = from; l <= kL; l += 2) m = level_size(l) > m ? level_size(l) : m;
    return m;
}
constexpr int w_entries() {
    int m = 2 * 2 * kMaxN;
    for (int l = 0; l < kL; ++l) {
        const int v = (1 << l) * 2 * (2 * (R - l - 1));
        m = v > m ? v : m;
    }
    return m;
}
// the sub-unit tree's stored matrices: after an include at depth d - 1, modes d and below
constexpr int slot_off(int d) {
    int o = 0;
    for (int e = 1; e < d; ++e) o += sym(2 * (kS + R - e));
    return o;
}
constexpr int dec_off(int m) {  // packed index tables of dimensions 2m, m < R
    int o = 0;
    for (int k = 1; k < m; ++k) o += sym(2 * k);
    return o;
}
struct Lay {
    static constexpr size_t X = 0;
    static constexpr size_t Y = X + sizeof(fl) * max_of(0);
    static constexpr size_t U = Y + sizeof(fl) * max_of(1);
    static constexpr size_t Sl = U + sizeof(fl) * sym(2 * (kS + R));
    static constexpr size_t W = Sl + sizeof(fl) * slot_off(kS);
    static constexpr size_t Q = W + sizeof(fl) * w_entries();          // a pivot's quantities, per warp
    static constexpr size_t sum = Q + 64 * kW;                          // fx [kSub][kW], binned: x 8
    static constexpr size_t tauX(bool bin) { return sum + sizeof(fx) * kSub * kW * (bin ? 8 : 1); }
    static constexpr size_t tauY(bool bin) { return tauX(bin) + 20 * (kThreads / 2); }
    static constexpr size_t ts(bool bin) { return tauY(bin) + 20 * kThreads; }  // node [kSub + 1]
    static constexpr size_t dec(bool bin) { return ts(bin) + 20 * (kSub + 1); }
    static constexpr size_t pos(bool bin) { return dec(bin) + 2 * dec_off(R); }
    static constexpr size_t modes(bool bin) { return pos(bin) + 2 * kMaxN; }
    static constexpr size_t bytes(bool bin) { return (modes(bin) + 128 + 15) / 16 * 16; }
    static_assert(sizeof(fl) * sym(2 * kMaxN) <= W, "prefix matrix must fit in X, Y, Ub and Sl");
};
// 228 KB an SM, 1 KB of it reserved a CTA
static_assert(3 * (Lay::bytes(true) + 1024 + 2500) <= 228 * 1024 && 3 * (Lay::bytes(false) + 1024 + 1600) <= 228 * 1024,
              "three CTAs must fit on an SM");

// f / w for the folded-triangle indices (f < 2^12, w <= 2 kMaxN + 1), by a reciprocal
__device__ __forceinline__ void fold_fast(int f, int D, uint32_t inv, int &i, int &j) {
    const int w = D + 1, p = (int)(((uint32_t)f * inv) >> 20), k = f - p * w;
    const bool low = k < D - p;
    i = low ? p : D - 1 - p;
    j = low ? p + k : i + (k - (D - p));
}
constexpr int kInv = sym(2 * (R - 1)) + 1;  // reciprocals 2^20 / w + 1 of w < kInv

// One 2x2 block pivot eliminated by the whole CTA: rows c0, c0 + 1 of the packed D x D matrix Mx;
// the trailing Schur complement is written to Dst (packed), or in place (Dst null), and
// det^{-1/2} to *rs.  Two barriers; the caller's data must be visible on entry.
__device__ __forceinline__ void elim(const fl *Mx, fl *inplace, int D, int c0, fl *Dst, fl *U, int4 *Qs, fx *rs,
                                     const uint32_t *inv20, int *flag, uint32_t &out) {
    const int t = threadIdx.x, Dt = D - c0 - 2;
    if (t < ((Dt + 31) & ~31)) {
        const fl p00 = Mx[pidx(D, c0, c0)], p01 = Mx[pidx(D, c0, c0 + 1)], p11 = Mx[pidx(D, c0 + 1, c0 + 1)];
        const fx det = fl_det2(p00, p01, p11), pk = fl_pack(p00);
        const bool odd = t & 1;
        fx in;
#pragma unroll
        for (int k = 0; k < 4; ++k) in.w[k] = odd ? det.w[k] : pk.w[k];
        const fx y = fl_rsqrt(in);
        const fx yo = fx_shfl_xor(y, 1);
        int4 *Q = Qs + 4 * (t >> 5);
        if ((t & 31) == 0) {
            const fl_piv v = fl_pivot_from(p00, p01, y, yo);
            Q[0] = make_int4(v.a.w[0], v.a.w[1], v.a.w[2], v.a.w[3]);
            Q[1] = make_int4(v.b.w[0], v.b.w[1], v.b.w[2], v.b.w[3]);
            Q[2] = make_int4(v.c.w[0], v.c.w[1], v.c.w[2], v.c.w[3]);
            Q[3] = make_int4(v.a.w[4], v.b.w[4], v.c.w[4], 0);
            if (t == 0) {
                *rs = yo;
                // a positive determinant of a negative block is outside this form's range only
                const int bad = fl_pivot_bad(det) | (fl_positive(p00) ? 0 : kFlLost);
                if (bad) atomicOr(flag, bad);
            }
        }
        __syncwarp();
        if (t < Dt) {
            const int4 qa = Q[0], qb = Q[1], qc = Q[2], qt = Q[3];
            const fl5 a{{qa.x, qa.y, qa.z, qa.w, qt.x}}, b{{qb.x, qb.y, qb.z, qb.w, qt.y}},
                c{{qc.x, qc.y, qc.z, qc.w, qt.z}};
            fl_urow(a, b, c, Mx[pidx(D, c0, c0 + 2 + t)], Mx[pidx(D, c0 + 1, c0 + 2 + t)], U[t], U[Dt + t], out);
            out |= fl_negative(Mx[pidx(D, c0 + 2 + t, c0 + 2 + t)]);
        }
    }
    __syncthreads();
    const int E = (Dt >> 1) * (Dt + 1);
    const uint32_t inv = inv20[Dt + 1];
    for (int f = t; f < E; f += kThreads) {
        int i, j;
        fold_fast(f, Dt, inv, i, j);
        const int at = pidx(D, c0 + 2 + i, c0 + 2 + j);
        const fl v = fl_sym_update(Mx[at], U[i], U[Dt + i], U[j], U[Dt + j]);
        if (Dst) Dst[pidx(Dt, i, j)] = v;
        else inplace[at] = v;
    }
    __syncthreads();
}

// The range check of one step of the chain of all includes (fl.cuh), t < d: the matrix's diagonal and, of its
// rows below the first pivot, U.  Out of line: the sweep passes here once a pattern, on the last warp
// beside the others' work.
static __device__ __noinline__ uint32_t chain_rows(const fl *P, int d, const int4 *Q, int t) {
    uint32_t out = fl_negative(P[pidx(d, t, t)]);
    if (t >= 2) {
        const int4 qa = Q[0], qb = Q[1], qc = Q[2], qt = Q[3];
        const fl5 a{{qa.x, qa.y, qa.z, qa.w, qt.x}}, b{{qb.x, qb.y, qb.z, qb.w, qt.y}}, c{{qc.x, qc.y, qc.z, qc.w, qt.z}};
        fl u0, u1;
        fl_urow(a, b, c, P[pidx(d, 0, t)], P[pidx(d, 1, t)], u0, u1, out);
    }
    return out;
}
// ... with the pivot's quantities anew (at the register bottom, which keeps them to itself)
static __device__ __noinline__ uint32_t chain_node(const fl *P, int d, int t) {
    uint32_t out = fl_negative(P[pidx(d, t, t)]);
    if (t >= 2) {
        const fl p00 = P[pidx(d, 0, 0)], p01 = P[pidx(d, 0, 1)], p11 = P[pidx(d, 1, 1)];
        const fl_piv v = fl_pivot_from(p00, p01, fl_rsqrt(fl_pack(p00)), fl_rsqrt(fl_det2(p00, p01, p11)));
        fl u0, u1;
        fl_urow(v.a, v.b, v.c, P[pidx(d, 0, t)], P[pidx(d, 1, t)], u0, u1, out);
    }
    return out;
}

template <bool BIN>
__global__ void __launch_bounds__(kThreads, 3) sweep_fx_kernel(int M, const double *__restrict__ O,
                                                              const uint64_t *__restrict__ pats, int n_pat, Plan pl) {
    extern __shared__ __align__(16) unsigned char smem[];
    fl *X = (fl *)(smem + Lay::X);
    fl *Y = (fl *)(smem + Lay::Y);
    fl *Ub = (fl *)(smem + Lay::U);
    fl *Sl = (fl *)(smem + Lay::Sl);
    fl *Wb = (fl *)(smem + Lay::W);
    int4 *Qs = (int4 *)(smem + Lay::Q);
    fx *s_sum = (fx *)(smem + Lay::sum);
    uint32_t *tauX = (uint32_t *)(smem + Lay::tauX(BIN));
    uint32_t *tauY = (uint32_t *)(smem + Lay::tauY(BIN));
    uint32_t *s_ts = (uint32_t *)(smem + Lay::ts(BIN));
    uint16_t *dec = (uint16_t *)(smem + Lay::dec(BIN));
    uint8_t *pos = smem + Lay::pos(BIN);
    uint8_t *modes = smem + Lay::modes(BIN);
    __shared__ long long s_unit;
    __shared__ int s_flag;
    __shared__ float s_abs[kSub * kW];
    __shared__ int s_exp[kSub * kW * (BIN ? 8 : 1)];
    __shared__ fx s_rs[kSub + kMaxN];  // the tree's and the prefix's det^{-1/2}
    __shared__ uint32_t inv20[kInv];

    const int t = threadIdx.x, lane = t & 31, wp = t >> 5;
    const int N2 = 2 * M;
    for (int m = 1; m < R; ++m) {
        const int d = 2 * m;
        for (int i = t; i < d; i += kThreads)
            for (int j = i; j < d; ++j) dec[dec_off(m) + pidx(d, i, j)] = (uint16_t)(i | (j << 8));
    }
    for (int w = t + 1; w < kInv; w += kThreads) inv20[w] = (1u << 20) / (uint32_t)w + 1u;
    const long long total = *pl.total_units;

    for (;;) {
        if (t == 0) {
            s_unit = (long long)atomicAdd(pl.counter, 1ull);
            s_flag = 0;
        }
        __syncthreads();
        const long long u = s_unit;
        if (u >= total) break;
        // sorted pattern position: unit_off[sp] <= u < unit_off[sp + 1]
        int lo = 0, hi = n_pat;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (pl.unit_off[mid] <= u) lo = mid; else hi = mid;
        }
        const int sp = lo;
        const int p = pl.perm[sp];
        const long long prefix = u - pl.unit_off[sp];
        const uint64_t wlo = pats[2 * p], whi = pats[2 * p + 1];
        const int nlo = __popcll(wlo), n = nlo + __popcll(whi);
        int n_eff, L_eff, q, ss;
        unit_shape<fx>(n, n_eff, L_eff, q, ss, pl.split);
        const int r = L_eff + B;           // modes of a sub-unit's level-0 matrix
        const int qs = q - ss;             // prefix levels fixed by the unit index
        const int rp = ss + r;             // modes after the unit's prefix elimination
        const int k = __popcll((unsigned long long)prefix);
        // the clicked modes, and the rows of the unit matrix: included prefix modes, then modes
        // qs .. n_eff - 1
        if (t < M) {
            const uint64_t w = t < 64 ? wlo : whi, bit = 1ull << (t & 63);
            if (w & bit) modes[(t < 64 ? 0 : nlo) + __popcll(w & (bit - 1))] = (uint8_t)t;
        }
        if (t < qs) {
            if (prefix >> t & 1) pos[__popcll((unsigned long long)prefix & ((1ull << t) - 1))] = (uint8_t)t;
        } else if (t < n_eff) {
            pos[k + t - qs] = (uint8_t)t;
        }
        __syncthreads();
        const int D0 = 2 * (k + rp);
        uint32_t out = 0;  // bits of rows and diagonal entries beyond the limb form's range (fl.cuh)
        // gather I - O on those rows into X, padding modes as identity
        {
            const uint32_t inv = inv20[D0 + 1];
            for (int f = t; f < (D0 >> 1) * (D0 + 1); f += kThreads) {
                int i, j;
                fold_fast(f, D0, inv, i, j);
                const int a = pos[i >> 1], b = pos[j >> 1];
                fl v{{0, 0, 0, i == j ? 1 << 24 : 0}};
                if (a < n && b < n) {
                    const int si = modes[a] + (i & 1) * M, sj = modes[b] + (j & 1) * M;
                    const double o = O[(size_t)si * N2 + sj];
                    if (!(fabs(o) <= 4.0)) atomicOr(&s_flag, kFlLost);
                    v = fl_from_fx(fx_from_double(i == j ? 1.0 : 0.0) - fx_from_double(o));
                }
                X[pidx(D0, i, j)] = v;
            }
        }
        __syncthreads();
        // eliminate the included prefix modes (2x2 block pivots)
        for (int e = 0; e < k; ++e)
            elim(X, X, D0, 2 * e, nullptr, Wb, Qs, s_rs + kSub + e, inv20, &s_flag, out);
        // the unit's trailing block -> Ub, through registers: the prefix matrix may extend over Ub
        {
            const int d = 2 * rp, o = 2 * k, E = (d >> 1) * (d + 1);
            constexpr int kPer = (sym(2 * (kS + R)) + kThreads - 1) / kThreads;
            const uint32_t inv = inv20[d + 1];
            fl tmp[kPer];
#pragma unroll
            for (int c = 0; c < kPer; ++c) {
                const int f = t + c * kThreads;
                int i, j;
                fold_fast(f < E ? f : 0, d, inv, i, j);
                tmp[c] = X[pidx(D0, o + i, o + j)];
            }
            __syncthreads();
#pragma unroll
            for (int c = 0; c < kPer; ++c) {
                const int f = t + c * kThreads;
                int i, j;
                fold_fast(f < E ? f : 0, d, inv, i, j);
                if (f < E) Ub[pidx(d, i, j)] = tmp[c];
            }
        }
        __syncthreads();
        const int nsub = 1 << ss;
        // The sub-units: the include (1) / exclude (0) choices of the next ss modes of Ub,
        // walked as a tree, depth e choosing mode e: the matrix after an include at depth e is
        // stored (in slot e + 1, or in X at the last depth), an exclude is a view of the same
        // matrix one mode further on; leaf `leaf` takes the choices of its bits from the top, so
        // consecutive leaves share every choice above the one that turns include.  jv[e]: the
        // slot of the matrix the node at depth e views (0: Ub).  The include that leaf `leaf`
        // starts with leaves its det^{-1/2} in s_rs[leaf].
        int jv[kS + 1];
#pragma unroll
        for (int e = 0; e <= kS; ++e) jv[e] = 0;
        for (int leaf = 0; leaf < nsub; ++leaf) {
            const int kk = __popc(leaf);
            const bool all = k == qs && kk == ss;  // its last node at every level has all modes included
            // the depth whose choice turns include (none at the first leaf); deeper choices
            // are excludes
            const int ds = leaf ? ss - 1 - (31 - __clz(leaf ^ (leaf - 1))) : ss;
            int j0 = 0;
#pragma unroll
            for (int e = 0; e <= kS; ++e)
                if (e == (leaf ? ds : ss)) j0 = jv[e];
            const fl *src = j0 ? Sl + slot_off(1) + (j0 == 2 ? slot_off(2) : 0) : Ub;
            const int D = 2 * (rp - j0);
            bool in_x = false;
            if (leaf) {
                in_x = ds + 1 == ss;
                fl *dst = in_x ? X : Sl + (ds == 1 ? slot_off(2) : 0);
                elim(src, nullptr, D, 2 * (ds - j0), dst, Wb, Qs, s_rs + leaf, inv20, &s_flag, out);
#pragma unroll
                for (int e = 0; e <= kS; ++e)
                    if (e > ds) jv[e] = ds + 1;
            }
            // level 0 of the expansion: the leaf's matrix, packed into X (already there after an
            // include at the last depth)
            if (!in_x) {
                const int j1 = leaf ? ds + 1 : 0;
                const fl *s1 = j1 ? Sl + (j1 == 2 ? slot_off(2) : 0) : Ub;
                const int D1 = 2 * (rp - j1), o = 2 * (ss - j1), d = 2 * r;
                const uint32_t inv = inv20[d + 1];
                for (int f = t; f < (d >> 1) * (d + 1); f += kThreads) {
                    int i, j;
                    fold_fast(f, d, inv, i, j);
                    X[pidx(d, i, j)] = s1[pidx(D1, o + i, o + j)];
                }
            }
            if (t == 0) node_st(tauX, 0, node_unit());
            __syncthreads();
            // breadth-first expansion of L_eff levels: node c at level l + 1 is child
            // c & 1 (0 exclude, 1 include) of parent c >> 1
            for (int l = 0; l < L_eff; ++l) {
                const fl *src = (l & 1) ? Y : X;
                fl *dst = (l & 1) ? X : Y;
                const uint32_t *tsrc = (l & 1) ? tauY : tauX;
                uint32_t *tdst = (l & 1) ? tauX : tauY;
                int4 *Qb = (int4 *)dst;  // the parents' pivot quantities, read before the children are written
                const int d = 2 * (r - l), dc = d - 2;
                const int sstr = nstride(d), dstr = nstride(dc), Ec = sym(dc);
                const int np = 1 << l;
                // (a) the parents' pivot quantities and the children's prefactors: two lanes a
                // parent, whole warps (for the shuffle)
                if (t < ((2 * np + 31) & ~31)) {
                    const int cp = min(t >> 1, np - 1);
                    const bool odd = t & 1;
                    const fl *P = src + cp * sstr;
                    const fl p00 = P[pidx(d, 0, 0)], p01 = P[pidx(d, 0, 1)], p11 = P[pidx(d, 1, 1)];
                    const fx det = fl_det2(p00, p01, p11), pk = fl_pack(p00);
                    fx in;
#pragma unroll
                    for (int c = 0; c < 4; ++c) in.w[c] = odd ? det.w[c] : pk.w[c];
                    const fx y = fl_rsqrt(in);   // even: p00^{-1/2}, odd: det^{-1/2}
                    const fx yo = fx_shfl_xor(y, 1);
                    fx rsv;
#pragma unroll
                    for (int c = 0; c < 4; ++c) rsv.w[c] = odd ? y.w[c] : yo.w[c];
                    const fl5 rr = fl5_at126(rsv), aa = fl5_at123(y);
                    // even: sqrt(p00) = p00 a, then b = sqrt(p00) rs; odd: c = p01 rs, then the
                    // include child's prefactor m rs
                    const node tp = node_ld(tsrc, cp);
                    fl f1;
                    fl5 g1;
#pragma unroll
                    for (int c = 0; c < 4; ++c) f1.w[c] = odd ? p01.w[c] : p00.w[c];
#pragma unroll
                    for (int c = 0; c < 5; ++c) g1.w[c] = odd ? rr.w[c] : aa.w[c];
                    int64_t pp[5] = {0, 0, 0, 0, 0}, qq[5] = {0, 0, 0, 0, 0};
                    fl_mac45(pp, f1, g1);
                    const fl5 h1 = fl5_carry(pp);
                    fl f2;
                    f2.w[0] = odd ? tp.m.w[0] : h1.w[0];
                    f2.w[1] = odd ? tp.m.w[1] : h1.w[1];
                    f2.w[2] = odd ? tp.m.w[2] : h1.w[2];
                    f2.w[3] = odd ? tp.m.w[3] : h1.w[3] + (h1.w[4] << 30);
                    fl_mac45(qq, f2, rr);
                    const fl5 h2 = fl5_carry(qq);
                    if (t < 2 * np) {
                        int4 *Q = Qb + 4 * cp;
                        int *Qt = (int *)(Q + 3);
                        if (odd) {
                            Q[2] = make_int4(h1.w[0], h1.w[1], h1.w[2], h1.w[3]);
                            Qt[2] = h1.w[4];
                            node_st(tdst, 2 * cp, tp);
                            node_st(tdst, 2 * cp + 1, node_norm(h2, tp.e));
                            const int bad = fl_chol_bad(p00, det);
                            if (bad) atomicOr(&s_flag, bad);
                        } else {
                            Q[0] = make_int4(aa.w[0], aa.w[1], aa.w[2], aa.w[3]);
                            Q[1] = make_int4(h2.w[0], h2.w[1], h2.w[2], h2.w[3]);
                            Qt[0] = aa.w[4];
                            Qt[1] = h2.w[4];
                        }
                    }
                }
                __syncthreads();
                // (b) the rows of U = B R^{-T}, dc per parent: u0 rows, then u1 rows
                const int nr = np * dc;
                {
                    const uint32_t inv = inv20[dc];
                    for (int f = t; f < nr; f += kThreads) {
                        const int cp = (int)(((uint32_t)f * inv) >> 20), i = f - cp * dc;
                        const fl *P = src + cp * sstr;
                        const int4 *Q = Qb + 4 * cp;
                        const int4 qa = Q[0], qb = Q[1], qc = Q[2], qt = Q[3];
                        const fl5 a{{qa.x, qa.y, qa.z, qa.w, qt.x}}, b{{qb.x, qb.y, qb.z, qb.w, qt.y}},
                            c{{qc.x, qc.y, qc.z, qc.w, qt.z}};
                        fl_urow(a, b, c, P[pidx(d, 0, i + 2)], P[pidx(d, 1, i + 2)], Wb[f], Wb[nr + f]);
                    }
                    if (all && t >= kLast && t < kLast + d)
                        out |= chain_rows(src + (np - 1) * sstr, d, Qb + 4 * (np - 1), t - kLast);
                }
                __syncthreads();
                // (c) both children of every parent: the exclude child is the parent's
                // trailing block, the include child its Schur complement
                const uint16_t *dtab = dec + dec_off(dc >> 1);
                const uint32_t einv = inv20[Ec];
                const int qstep = (int)((kThreads * einv) >> 20), rstep = kThreads - qstep * Ec;
                int cp = (int)(((uint32_t)t * einv) >> 20), e = t - cp * Ec;
                auto step = [&]() {
                    e += rstep;
                    cp += qstep;
                    if (e >= Ec) {
                        e -= Ec;
                        ++cp;
                    }
                };
                int f = t;
                for (; f + kThreads < np * Ec; f += 2 * kThreads) {
                    const int ij = dtab[e], i = ij & 0xff, j = ij >> 8, at = 2 * cp * dstr + e;
                    const fl v = src[cp * sstr + pidx(d, i + 2, j + 2)];
                    const fl *U0 = Wb + cp * dc, *U1 = U0 + nr;
                    const fl a0 = U0[i], a1 = U1[i], b0 = U0[j], b1 = U1[j];
                    step();
                    const int ij2 = dtab[e], i2 = ij2 & 0xff, j2 = ij2 >> 8, at2 = 2 * cp * dstr + e;
                    const fl v2 = src[cp * sstr + pidx(d, i2 + 2, j2 + 2)];
                    const fl *V0 = Wb + cp * dc, *V1 = V0 + nr;
                    const fl c0 = V0[i2], c1 = V1[i2], d0 = V0[j2], d1 = V1[j2];
                    step();
                    const fl r1 = fl_sym_update(v, a0, a1, b0, b1);
                    const fl r2 = fl_sym_update(v2, c0, c1, d0, d1);
                    dst[at] = v;
                    dst[at2] = v2;
                    dst[at + dstr] = r1;
                    dst[at2 + dstr] = r2;
                }
                if (f < np * Ec) {
                    const int ij = dtab[e], i = ij & 0xff, j = ij >> 8, at = 2 * cp * dstr + e;
                    const fl v = src[cp * sstr + pidx(d, i + 2, j + 2)];
                    const fl *U0 = Wb + cp * dc, *U1 = U0 + nr;
                    dst[at] = v;
                    dst[at + dstr] = fl_sym_update(v, U0[i], U1[i], U0[j], U1[j]);
                }
                __syncthreads();
            }
            // the register bottom: each thread's two-mode node, relative to its prefactor m 2^e
            const fl *nodes = (L_eff & 1) ? Y : X;
            const bool has = t < (1 << L_eff);
            if (all && t >= kLast && t < kLast + 2 * B)
                out |= chain_node(nodes + ((1 << L_eff) - 1) * nstride(2 * B), 2 * B, t - kLast);
            int e = -(1 << 20);
            node tn = node_unit();
            const int nreal = n - (n_eff - B);
            if (has) {
                tn = node_ld((L_eff & 1) ? tauY : tauX, t);
                e = tn.e;
            }
            const int at = leaf * kW + wp;
            if constexpr (BIN) {
                // unsigned, by subset size (a lane's bin b, 0..B, belongs to the warp's size
                // popc(lane) + b): every size aligned to the largest exponent among the lanes that
                // hold it, so that a size keeps its last bits beside one of larger terms (a
                // mode included may scale them by 16); then lane (z, part) sums every fourth
                // lane's share of the warp's size z = 0..7
                const int pc = __popc(lane);
                int by = -(1 << 20);  // lane c: the largest exponent of the lanes with c includes
#pragma unroll
                for (int c = 0; c <= 5; ++c) {
                    const int v = __reduce_max_sync(0xffffffffu, pc == c ? e : -(1 << 20));
                    if (lane == c) by = v;
                }
                int ez = by;          // lane z: of the lanes that hold size z
#pragma unroll
                for (int b = 1; b <= B; ++b) ez = max(ez, __shfl_sync(0xffffffffu, by, (lane - b) & 31));
                fx *scratch = (fx *)((L_eff & 1) ? X : Y) + wp * 32 * (B + 1);
                BinAcc<fx, B + 1> acc;
#pragma unroll
                for (int b = 0; b <= B; ++b) acc.v[b] = fx_zero();
                acc.bad = 0;
                if (has) {
                    SmemMat<fl, B> A{nodes + t * nstride(2 * B)};
                    dfs<fx, B, 0, false>(A, fx_one(), 0, nreal, acc, 0);
                    if (acc.bad) atomicOr(&s_flag, acc.bad);
                    const fx mp = node_packed(tn);
#pragma unroll
                    for (int b = 0; b <= B; ++b) acc.v[b] = fx_mul_uu(acc.v[b], mp);
                }
#pragma unroll
                for (int b = 0; b <= B; ++b)
                    scratch[lane * (B + 1) + b] = fx_shr(acc.v[b], __shfl_sync(0xffffffffu, ez, pc + b) - e + 4);
                __syncwarp();
                const int z = lane & 7, part = lane >> 3;
                fx s = fx_zero();
#pragma unroll
                for (int c = 0; c < 8; ++c) {
                    const int t2 = part * 8 + c, b = z - __popc(t2);
                    if (b >= 0 && b <= B) s = s + scratch[t2 * (B + 1) + b];
                }
                s = s + fx_shfl_xor(s, 8);
                s = s + fx_shfl_xor(s, 16);
                if (lane < 8) {
                    s_sum[at * 8 + lane] = s;
                    s_exp[at * 8 + lane] = ez;
                }
                __syncthreads();  // the scratch lies in the next sub-unit's matrices
            } else {
                const int em = __reduce_max_sync(0xffffffffu, e);
                fx v = fx_zero();
                float ab = 0.0f;
                if (has) {
                    Acc<fx> acc{fx_zero(), fx_zero(), 0, 0};
                    SmemMat<fl, B> A{nodes + t * nstride(2 * B)};
                    dfs<fx, B, 0, false>(A, fx_one(), 0, nreal, acc, 0);
                    const int excl = (qs - k) + (ss - kk) + (L_eff - __popc(t));
                    v = fx_neg_if(fx_mul_su(acc.hi, node_packed(tn)), excl & 1);  // |v| < 2^11
                    ab = acc.abs * ((float)(tn.m.w[3] >> 11) * (1.0f / 65536.0f));
                    if (acc.bad) atomicOr(&s_flag, acc.bad);
                }
                // align to 2^(em + 4): the unit's sums of 128 such terms stay below 2^14
                v = fx_shr(v, em - e + 4);
                ab = ldexpf(ab, max(e - em, -126));
#pragma unroll
                for (int off = 16; off; off >>= 1) {
                    v = v + fx_shfl_xor(v, off);
                    ab += __shfl_xor_sync(0xffffffffu, ab, off);
                }
                if (lane == 0) {
                    s_sum[at] = v;
                    s_abs[at] = ab;
                    s_exp[at] = em;
                }
                // X and Y: the nodes were read from Y (or this was the only sub-unit), and the
                // next sub-unit writes Y after a barrier only
            }
        }
        if (out) atomicOr(&s_flag, 2);  // not positive definite: beside a pivot that says so, or alone
        __syncthreads();
        if (t < 32) {
            // the prefix factor (a tree of products over the lanes) and each sub-unit's (the
            // includes on its path, from the top)
            node tp = node_unit();
            for (int e = t; e < k; e += 32) tp = node_mul(tp, s_rs[kSub + e]);
            const int top = k < 32 ? k : 32;
            for (int off = 1; off < top; off <<= 1) {
                node o;
#pragma unroll
                for (int c = 0; c < 4; ++c) o.m.w[c] = __shfl_down_sync(0xffffffffu, tp.m.w[c], off);
                o.e = __shfl_down_sync(0xffffffffu, tp.e, off);
                if ((t & (2 * off - 1)) == 0 && t + off < top) tp = node_mul(tp, o);
            }
            if (t == 0) node_st(s_ts, kSub, tp);
            if (t < nsub) {
                node ts = node_unit();
                for (int b = ss - 1; b >= 0; --b)
                    if (t >> b & 1) ts = node_mul(ts, s_rs[t & ~((1 << b) - 1)]);
                node_st(s_ts, t, ts);
            }
        }
        if constexpr (BIN) __syncthreads();
        else __syncwarp();
        if constexpr (BIN) {
            // sub-unit `leaf`, size z (0..9 within it): the four warps' sums (warp w holds the
            // sizes popc(w) + 0..7), aligned to the size's largest exponent, times the sub-unit's
            // factor, then per size of the unit
            dd *part = (dd *)X;
            if (t < 10 * nsub) {
                const int leaf = t / 10, z = t - 10 * leaf;
                int em = -(1 << 20);
#pragma unroll
                for (int w = 0; w < kW; ++w) {
                    const int b = z - __popc(w);
                    if (b >= 0 && b < 8) em = max(em, s_exp[(leaf * kW + w) * 8 + b]);
                }
                fx S = fx_zero();
#pragma unroll
                for (int w = 0; w < kW; ++w) {
                    const int b = z - __popc(w), at = (leaf * kW + w) * 8 + b;
                    if (b >= 0 && b < 8) S = S + fx_shr(s_sum[at], em - s_exp[at]);
                }
                const dd sv = fx_to_dd(S);
                const double sc = ldexp(1.0, em + 4);  // (a size without terms: 0)
                part[t] = node_dd(node_ld(s_ts, leaf)) * dd(sv.hi * sc, sv.lo * sc);
            }
            __syncthreads();
            double *out = pl.partials + (size_t)2 * (n + 1) * u;
            const dd tp = node_dd(node_ld(s_ts, kSub));
            for (int z = t; z <= n; z += kThreads) {
                dd s = dd(0.0);
                for (int leaf = 0; leaf < nsub; ++leaf) {
                    const int b = z - k - __popc(leaf);
                    if (b >= 0 && b < 10) s += part[10 * leaf + b];
                }
                store2(out + 2 * z, tp * s);
            }
            if (t == 0 && s_flag) atomicOr(pl.pflags + sp, 1);
            __syncthreads();
        } else if (t < 32) {
            // the sub-units' sums, one lane each: the four warps aligned to the largest exponent
            // and added, times the sub-unit's prefix factor; added over the lanes in a fixed
            // pairing, times the unit's prefix factor
            dd s = dd(0.0);
            double a = 0.0;
            if (t < nsub) {
                const int *ex = s_exp + t * kW;
                int em = ex[0];
#pragma unroll
                for (int w = 1; w < kW; ++w) em = max(em, ex[w]);
                fx S = fx_shr(s_sum[t * kW], em - ex[0]);
                float AB = ldexpf(s_abs[t * kW], max(ex[0] - em, -126));
#pragma unroll
                for (int w = 1; w < kW; ++w) {
                    S = S + fx_shr(s_sum[t * kW + w], em - ex[w]);
                    AB += ldexpf(s_abs[t * kW + w], max(ex[w] - em, -126));
                }
                const dd ts = node_dd(node_ld(s_ts, t)), sv = fx_to_dd(S);
                const double sc = ldexp(1.0, em + 4);
                s = ts * dd(sv.hi * sc, sv.lo * sc);
                a = ts.hi * ldexp((double)AB, em);
            }
#pragma unroll
            for (int off = 1; off < kSub; off <<= 1) {
                const double oh = __shfl_xor_sync(0xffffffffu, s.hi, off), ol = __shfl_xor_sync(0xffffffffu, s.lo, off);
                const double oa = __shfl_xor_sync(0xffffffffu, a, off);
                s = s + dd(oh, ol);
                a += oa;
            }
            if (t == 0) {
                const dd tp = node_dd(node_ld(s_ts, kSub));
                s = s * tp;
                double *out = pl.partials + 3 * u;
                out[0] = s.hi;
                out[1] = s.lo;
                out[2] = a * tp.hi;
                if (s_flag) atomicOr(pl.pflags + sp, fl_unit_flags(s_flag));
            }
        }
    }
}

}  // namespace fxk
