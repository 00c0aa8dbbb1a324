// Gradients of L = sum_p w_p log P_p (not in the paper; the state-build adjoint
// lets squeezing, loss and the interferometer be fitted to click data).
//
// From log P = -1/2 log det sigma_Q + log T(A_S), A = sigma_Q^{-1} and
// d det(A_Z)^{-1/2} = -1/2 det(A_Z)^{-1/2} tr(A_Z^{-1} dA_Z):
//     dT = tr(Gbar dA_S),  Gbar = sum_Z (-1)^{n-|Z|} (-1/2) tau_Z A_Z^{-1},
//     dL/dsigma_Q = -1/2 (sum_p w_p) A - A H A,   H = sum_p (w_p / T_p) embed(Gbar_p).
// Gbar and T cancel together by the condition number kappa of the signed sum
// (1e14..1e19 on improbable patterns), so the whole computation is in 110-bit software floating
// point (double-double for the patterns that cancel by more than 1e24);
// after the division by T the result is an ordinary FP64 number.  Gbar = dT/dA_S is
// computed in reverse mode through the same include/exclude Schur recursion that
// evaluates T (O(2^n) work instead of a factorisation and inverse per subset); one
// CTA per pattern, its units in order (deterministic).
//
// Then the chain through sigma_Q = eta R diag(d) R^T + (1 - eta/2) I (R the xp
// form of U, d = e^{-2r}/2 on x, e^{2r}/2 on p) and through the rectangular
// mesh U = T_last ... T_1, T(theta, phi) = [[e^{i phi} cos, -sin], [e^{i phi} sin, cos]].
#include <cooperative_groups.h>

#include "dd.cuh"
#include "gbs_internal.cuh"
#include "kappa.cuh"
#include "qf.cuh"

namespace {

constexpr int kGradMaxN = 24;            // clicks per pattern on the gradient path
constexpr int kGD = 2 * kGradMaxN;       // largest pattern matrix (48 x 48)
constexpr int kTM = 7;                   // modes of a unit's subtree (2^7 leaves)
constexpr int kTreeThreads = 256;
constexpr int kChunkBits = 8;            // a chunk: at most 2^8 units sharing their high prefix modes
constexpr int kGroupBits = 4;            // a group: at most 2^4 units walked as a tree

__host__ __device__ constexpr int gsym(int d) { return d * (d + 1) / 2; }
// packed upper-triangle index of (i, j), i <= j.  The rows of the trailing block of modes below
// are the suffix of the array: the block left when the first mode is excluded starts 2 d - 1
// entries further on and is packed itself.
__host__ __device__ constexpr int gpidx(int d, int i, int j) { return i * d - (i * (i - 1)) / 2 + (j - i); }
__device__ __forceinline__ int gpany(int d, int i, int j) { return i <= j ? gpidx(d, i, j) : gpidx(d, j, i); }
// the include children of a unit's subtree, level after level, after its root
__host__ __device__ constexpr int lvl_off(int l) {
    int s = gsym(2 * kTM);
    for (int q = 1; q < l; ++q) s += (1 << (q - 1)) * gsym(2 * (kTM - q));
    return s;
}
__host__ __device__ constexpr int adj_cap() {
    int m = gsym(2 * (kTM + kGroupBits));
    for (int l = 0; l < kTM; ++l) m = (1 << l) * gsym(2 * (kTM - l)) > m ? (1 << l) * gsym(2 * (kTM - l)) : m;
    return m;
}
__host__ __device__ constexpr int row_cap() {  // 2 x dc entries of every parent of a level
    int m = 2 * (kGD - 2);
    for (int l = 0; l < kTM; ++l) m = (1 << l) * 4 * (kTM - l - 1) > m ? (1 << l) * 4 * (kTM - l - 1) : m;
    return m;
}
__host__ __device__ constexpr int tri_sum(int from, int to) {  // packed matrices of from .. to modes
    int s = 0;
    for (int m = from; m <= to; ++m) s += gsym(2 * m);
    return s;
}
constexpr int kNodes = (1 << kTM) - 1;   // nodes of levels 0..kTM-1
constexpr int kUD = 2 * (kChunkBits + kTM);  // largest group matrix (middle prefix modes, group, subtree)
// shared memory (qf elements), SM at the end (its size is the batch's).
// UM: the group's matrix; Gam: the adjoint of SM's trailing block summed over the groups; Sl, Gx,
// dS: the group tree's include matrices, exclude adjoints and sums; Lv: the subtree's include
// matrices, and between subtrees the group's (Gf) or the chunk's (Gs) adjoint; SM: the chunk's matrix
constexpr int kOffUM = 0, kOffGam = kOffUM + gsym(kUD), kOffSl = kOffGam + gsym(kUD);
constexpr int kOffGx = kOffSl + tri_sum(kTM + 1, kTM + kGroupBits - 1);
constexpr int kOffLv = kOffGx + tri_sum(kTM, kTM + kGroupBits - 1);
constexpr int kLvCap = lvl_off(kTM) > gsym(kGD) ? lvl_off(kTM) : gsym(kGD);
constexpr int kOffAdjA = kOffLv + kLvCap, kOffAdjB = kOffAdjA + adj_cap();
constexpr int kOffQ = kOffAdjB + adj_cap(), kOffRs = kOffQ + 3 * kNodes, kOffS = kOffRs + kNodes;
constexpr int kOffZ = kOffS + kNodes, kOffY = kOffZ + row_cap(), kOffM2 = kOffY + row_cap();
constexpr int kOffDQ = kOffM2 + 3 * (1 << (kTM - 1)), kOffDRs = kOffDQ + 3 * kGroupBits, kOffDS = kOffDRs + kGroupBits;
constexpr int kOffPreQ = kOffDS + kGroupBits + 2, kOffPreRs = kOffPreQ + 3 * kChunkBits;
constexpr int kOffHiQ = kOffPreRs + kChunkBits, kOffHiRs = kOffHiQ + 3 * kGradMaxN;
constexpr int kOffSM = kOffHiRs + kGradMaxN;
__host__ __device__ constexpr int tree_smem(int n_max) { return kOffSM + gsym(2 * n_max); }

// (i, j), i <= j, of packed entry f of an even dimension d: rows p and d - 1 - p folded
__device__ __forceinline__ void fold_ij(int f, int d, int &i, int &j) {
    const int w = d + 1, p = f / w, k = f - p * w;
    if (k < d - p) {
        i = p;
        j = p + k;
    } else {
        i = d - 1 - p;
        j = i + (k - (d - p));
    }
}

// One level of include steps, forward.  Parent cp (of np) is the packed d x d matrix at base +
// noff[cp]; its pivot block is the first mode.  Stores P^{-1} (the off-diagonal entry negated, here
// and wherever P^{-1} is kept) in Q + 3 cp and det^{-1/2} in rs[cp], and writes the include child
// C - W B^T (W = P^{-1} B) to dst + cp * gsym(d - 2) (which may be the parent's own trailing block),
// with the children's places in nchild (exclude, include) where it is given.  d = 2: pivots only.
__device__ __noinline__ void tree_forward(qf *base, int np, int d, const uint16_t *noff, qf *dst, uint16_t *nchild,
                                          qf *Q, qf *rs, qf *W, int *bad) {
    const int t = threadIdx.x, dc = d - 2, stc = gsym(dc);
    // four lanes a parent: the determinant and its root on each, then one product each
    if (t < 4 * np) {
        const int cp = t >> 2, k = t & 3;
        const qf *P = base + noff[cp];
        const qf p00 = P[0], p01 = P[1], p11 = P[d];
        const qf det = qf_dot2s(false, p00, p11, true, p01, p01);
        const qf r = qf_rsqrt(det), inv = r * r;
        qf f;
#pragma unroll
        for (int c = 0; c < 4; ++c) f.w[c] = k == 0 ? p11.w[c] : k == 1 ? p01.w[c] : p00.w[c];
        f = f * inv;
        if (k < 3) {
            Q[3 * cp + k] = f;
        } else {
            rs[cp] = r;
            if (!qf_positive(det) || qf_saturated(det)) atomicOr(bad, 1);
            if (nchild) {
                nchild[2 * cp] = (uint16_t)(noff[cp] + 2 * d - 1);
                nchild[2 * cp + 1] = (uint16_t)(dst - base + cp * stc);
            }
        }
    }
    __syncthreads();
    if (dc == 0) return;
    for (int f = t; f < np * dc * 2; f += kTreeThreads) {
        const int cp = f / (2 * dc), x = f - cp * 2 * dc, i = x >> 1, a = x & 1;
        const qf *P = base + noff[cp], *q = Q + 3 * cp;
        W[f] = qf_dot2s(a, q[a], P[2 + i], !a, q[1 + a], P[d + 1 + i]);
    }
    __syncthreads();
    for (int f = t; f < np * stc; f += kTreeThreads) {
        const int cp = f / stc, e = f - cp * stc;
        int i, j;
        fold_ij(e, dc, i, j);
        const qf *P = base + noff[cp], *w = W + 2 * (cp * dc + i);
        const int at = gpidx(dc, i, j);
        dst[cp * stc + at] = qf_fms2(P[2 * d - 1 + at], w[0], P[2 + j], w[1], P[d + 1 + j]);
    }
    __syncthreads();
}

// One level of include steps, backward: from the children's adjoints to the parents'.  Parent cp's
// include child has the adjoint Gi + cp * gs (packed, d - 2 rows) and the sum Si[cp * ss]; its
// exclude child, unless Ge is null, Ge + cp * gs and Se[cp * ss].  With Y = P^{-1} B Gi the parent's
// adjoint is, times rs,
//   rest: Gi - Ge / rs,   pivot rows: -Y,   pivot block: P^{-1} (B Gi B^T) P^{-1} - Si P^{-1} / 2
// (Ge null: the pivot of a shared prefix, whose factor is in Si already: no rs, and the rest stays
// where it is, out's own trailing block).  So, Ao: the parents' sums and, to 20 bits, the sums of their
// terms' sizes.  K: slices of a row sum, for levels with few parents.
__device__ __noinline__ void tree_backward(const qf *base, int np, int d, const uint16_t *noff, const qf *Gi,
                                           const qf *Ge, int gs, qf *out, const qf *Q, const qf *rs, const qf *Si,
                                           const qf *Se, int ss, qf *So, const double *Ai, const double *Ae, double *Ao, qf *Z,
                                           qf *Y, qf *M2, int K) {
    const int t = threadIdx.x, t2 = kTreeThreads - 1 - t, dc = d - 2, st = gsym(d), stc = gsym(dc);
    // Z = B Gi, slice k of K of entry (a, j): whole warps, for the sums over the slices
    const int nz = np * dc * 2 * K;
    for (int f = t; f < ((nz + 31) & ~31); f += kTreeThreads) {
        const int g = min(f, nz - 1) / K, k = f & (K - 1), cp = g / (2 * dc), x = g - cp * 2 * dc, j = x >> 1, a = x & 1;
        const qf *b = base + noff[cp] + (a ? d + 1 : 2), *G = Gi + cp * gs;
        qf z = qf_dot(k, K, dc, [&](int i) { return G + gpany(dc, i, j); }, [&](int i) { return b + i; });
        for (int off = 1; off < K; off <<= 1) {
            qf o;
#pragma unroll
            for (int c = 0; c < 4; ++c) o.w[c] = __shfl_xor_sync(0xffffffffu, z.w[c], off);
            z = z + o;
        }
        if (f < nz && k == 0) Z[g] = z;
    }
    if (So && t2 < np) {
        So[t2] = qf_fma<false, true>(Se[t2 * ss], rs[t2], Si[t2 * ss]);
        Ao[t2] = fma(qf_approx(rs[t2]), Ai[t2 * ss], Ae[t2 * ss]);
    }
    __syncthreads();
    for (int f = t; f < np * dc * 2; f += kTreeThreads) {
        const int cp = f / (2 * dc), x = f - cp * 2 * dc, j = x >> 1, a = x & 1;
        const qf *q = Q + 3 * cp, *z = Z + 2 * (cp * dc + j);
        Y[f] = qf_dot2s(a, q[a], z[0], !a, q[1 + a], z[1]);
    }
    for (int f = t2; f < np * 3; f += kTreeThreads) {
        const int cp = f / 3, ij = f - 3 * cp;  // (0, 0), (0, 1), (1, 1)
        const qf *z = Z + 2 * cp * dc + (ij == 2), *b = base + noff[cp] + (ij ? d + 1 : 2);
        M2[f] = qf_dot(0, 1, dc, [&](int c) { return z + 2 * c; }, [&](int c) { return b + c; });
    }
    __syncthreads();
    const int nrest = Ge ? np * stc : 0;
    for (int f = t; f < nrest; f += kTreeThreads) {
        const int cp = f / stc, e = f - cp * stc;
        out[cp * st + 2 * d - 1 + e] = qf_fma<false, true>(Ge[cp * gs + e], rs[cp], Gi[cp * gs + e]);
    }
    for (int f = t; f < np * dc * 2; f += kTreeThreads) {
        const int cp = f / (2 * dc), x = f - cp * 2 * dc, j = x >> 1, a = x & 1;
        out[cp * st + (a ? d + 1 : 2) + j] = qf_mul<true>(Ge ? rs[cp] : qf_one(), Y[f]);
    }
    for (int f = t2; f < np * 3; f += kTreeThreads) {
        const int cp = f / 3, ij = f - 3 * cp, i = ij == 2, j = ij != 0;
        const qf *q = Q + 3 * cp, *m = M2 + 3 * cp;
        // column j of M2 P^{-1}, then row i of P^{-1} times it
        const qf u0 = qf_dot2s(j, m[0], q[j], !j, m[1], q[1 + j]), u1 = qf_dot2s(j, m[1], q[j], !j, m[2], q[1 + j]);
        const qf v = qf_dot2s(i, q[i], u0, !i, q[1 + i], u1), h = qf_half(Si[cp * ss]);
        const qf r = ij == 1 ? qf_fma<false>(v, h, q[1]) : qf_fma<true>(v, h, q[ij]);
        out[cp * st + (ij == 2 ? d : ij)] = Ge ? rs[cp] * r : r;
    }
    __syncthreads();
}

// Gbar_p = dT/dA_S by reverse mode through the include/exclude Schur recursion.
// Units = (pattern, include/exclude choice of the first q = n - m modes), m = min(n, 7), the
// subtree over the last m modes.  S(node) = rs S(include child) - S(exclude child), 1 at a leaf;
// Gamma(node) = dS(node)/dC_node from the children's (tree_backward); a node's exclude child is the
// suffix of its packed matrix, so only include children are stored.
// One CTA per chunk: an aligned run of 2^b units of one pattern.  Of the prefix modes the high
// ones (b and up) are fixed by the chunk and eliminated once; the others are the bits of the unit,
// the last kGroupBits of them (the group's) walked depth first as a tree over the units' subtrees,
// each include's matrix and each exclude's adjoint kept per depth, so that a unit costs one tree
// pivot and one step back on average; the ones between (middle) are eliminated once per group.
// The group's adjoint goes back through its middle pivots into Gam, and Gam at the end
// through the chunk's high pivots with V = the chunk's sum (the adjoint of a shared step is linear in
// what flows into it).
//
// What bounds it: integer instructions and, with two CTAs an SM, the latency of about 40 phases a
// unit; the work of a phase is cut fine for that (a row sum in up to four slices, a pivot over
// four lanes, long jobs on the last warps beside the short ones on the first).  Measured on the
// 32-mode Clements workload (512 patterns, n = 8..16): 69.5 ms in double-double (FP64 pipe 70% busy),
// 49.9 with the same kernel in qf (barriers, divergence), 18.0 as it is here.
__global__ void __launch_bounds__(kTreeThreads, 2) grad_tree_kernel(int M, const double *__restrict__ O,
                                                               const uint64_t *__restrict__ pats,
                                                               const int *__restrict__ chunk_p,
                                                               const long long *__restrict__ chunk_u, size_t pst,
                                                               qf *__restrict__ part, qf *__restrict__ part_T,
                                                               double *__restrict__ part_A,
                                                               int *__restrict__ flags) {
    extern __shared__ __align__(16) unsigned char gsm[];
    qf *const base = (qf *)gsm;
    qf *const SM = base + kOffSM, *const Gs = base + kOffLv, *const UM = base + kOffUM, *const Gf = base + kOffLv;
    qf *const Gam = base + kOffGam, *const Lv = base + kOffLv;
    qf *const nQ = base + kOffQ, *const nrs = base + kOffRs, *const nS = base + kOffS;
    qf *const Zb = base + kOffZ, *const Yb = base + kOffY, *const M2 = base + kOffM2;
    qf *const dQ = base + kOffDQ, *const dRs = base + kOffDRs, *const dS = base + kOffDS;
    qf *const preQ = base + kOffPreQ, *const prers = base + kOffPreRs;
    qf *const hiQ = base + kOffHiQ, *const hiRs = base + kOffHiRs;
    __shared__ uint8_t modes[128], smrow[kGD], umrow[kUD];  // rows of SM and UM: see below
    __shared__ uint16_t nptr[kNodes + 1], s_off[1], dptr[kGroupBits + 1];
    __shared__ int s_bad;
    __shared__ qf s_T, s_V, s_S[2];
    __shared__ double nA[kNodes], dA[kGroupBits], s_A[2], s_Asum;
    __shared__ float s_guess;
    const int t = threadIdx.x, ch = blockIdx.x, p = chunk_p[ch], N2 = 2 * M;
    const long long u_begin = chunk_u[2 * ch], u_end = chunk_u[2 * ch + 1];
    const uint64_t wlo = pats[2 * p], whi = pats[2 * p + 1];
    const int nlo = __popcll(wlo), n = nlo + __popcll(whi), m = n < kTM ? n : kTM, q = n - m, Dn = 2 * n;
    if (t < M) {
        const uint64_t w = t < 64 ? wlo : whi, bit = 1ull << (t & 63);
        if (w & bit) modes[(t < 64 ? 0 : nlo) + __popcll(w & (bit - 1))] = (uint8_t)t;
    }
    if (t == 0) {
        s_bad = 0;
        s_Asum = 0.0;
        s_T = n == 0 && u_begin == 0 ? qf_one() : qf_zero();
    }
    // the chunk's 2^bl units vary the prefix modes 0..bl-1: the middle ones 0..bm-1 and the group's
    // g modes bm..bl-1; modes bl..q-1 are fixed by u_begin
    const int bl = u_end > u_begin ? 63 - __clzll(u_end - u_begin) : 0;
    const int g = bl < kGroupBits ? bl : kGroupBits, bm = bl - g;
    const unsigned long long hi = (unsigned long long)u_begin >> bl;
    const int kh = __popcll(hi), Ds = 2 * (kh + bl + m), Dr = 2 * (bl + m);
    // SM: the included high modes, then modes 0..bl-1, then the subtree's; smrow: row -> pattern row
    if (t < q) {
        const int a = t;
        int r = -1;
        if (a < bl) r = kh + a;
        else if (hi >> (a - bl) & 1) r = __popcll(hi & ((1ull << (a - bl)) - 1));
        if (r >= 0) {
            smrow[2 * r] = (uint8_t)(2 * a);
            smrow[2 * r + 1] = (uint8_t)(2 * a + 1);
        }
    } else if (t < n) {
        const int r = kh + bl + t - q;
        smrow[2 * r] = (uint8_t)(2 * t);
        smrow[2 * r + 1] = (uint8_t)(2 * t + 1);
    }
    __syncthreads();
    if (n >= kGuessFrom) {  // alike in all chunks of the pattern
        if (t < 32) {
            const float k = kappa_guess(O, M, modes, n);
            if (t == 0) s_guess = k;
        }
        __syncthreads();
        if (s_guess > kGuessRedo) {
            if (t == 0) atomicOr(flags + p, 1);
            return;
        }
    }
    // the chunk's rows of A = I - O, its high pivots, and a zero Gam
    for (int f = t; f < gsym(Ds); f += kTreeThreads) {
        int i, j;
        fold_ij(f, Ds, i, j);
        const int ri = smrow[i], rj = smrow[j];
        const int gi = modes[ri >> 1] + (ri & 1) * M, gj = modes[rj >> 1] + (rj & 1) * M;
        const double o = O[(size_t)gi * N2 + gj];
        if (!(fabs(o) <= 0x1p100)) atomicOr(&s_bad, 1);  // not finite, or far beyond any state: left to double-double
        SM[gpidx(Ds, i, j)] = (i == j ? qf_one() : qf_zero()) - qf_from_double(o);
    }
    for (int f = t; f < gsym(Dr); f += kTreeThreads) Gam[f] = qf_zero();
    // where the packed trailing block of the last d rows of a D-row matrix starts
    auto tail = [](int D, int d) { return gsym(D) - gsym(d); };
    for (int e = 0; e < kh; ++e) {
        const int d = Ds - 2 * e;
        if (t == 0) s_off[0] = (uint16_t)(SM - base + tail(Ds, d));
        __syncthreads();
        tree_forward(base, 1, d, s_off, SM + tail(Ds, d - 2), nullptr, hiQ + 3 * e, hiRs + e, Zb, &s_bad);
    }
    const int groups = n > 0 ? 1 << bm : 0;
    for (int gr = 0; gr < groups; ++gr) {
        const int kl = __popc(gr), D0 = 2 * (kl + g + m), k0 = kh + kl;
        // UM: SM's trailing block on the group's included middle modes, its own modes and the
        // subtree; umrow: row -> row of SM's trailing block
        if (t < bm) {
            if (gr >> t & 1) {
                const int r = __popc(gr & ((1 << t) - 1));
                umrow[2 * r] = (uint8_t)(2 * t);
                umrow[2 * r + 1] = (uint8_t)(2 * t + 1);
            }
        } else if (t < bl + m) {
            const int r = kl + t - bm;
            umrow[2 * r] = (uint8_t)(2 * t);
            umrow[2 * r + 1] = (uint8_t)(2 * t + 1);
        }
        __syncthreads();
        for (int f = t; f < gsym(D0); f += kTreeThreads) {
            int i, j;
            fold_ij(f, D0, i, j);
            UM[gpidx(D0, i, j)] = SM[gpidx(Ds, 2 * kh + umrow[i], 2 * kh + umrow[j])];
        }
        for (int e = 0; e < kl; ++e) {
            const int d = D0 - 2 * e;
            if (t == 0) s_off[0] = (uint16_t)(UM - base + tail(D0, d));
            __syncthreads();
            tree_forward(base, 1, d, s_off, UM + tail(D0, d - 2), nullptr, preQ + 3 * e, prers + e, Zb, &s_bad);
        }
        // the group's tree: depth e chooses mode e; dptr[e]: the matrix of the path's node there
        const int dg = 2 * (g + m);
        if (t == 0) {
            dptr[0] = (uint16_t)(UM - base + tail(D0, dg));
            for (int e = 0; e < g; ++e) dptr[e + 1] = (uint16_t)(dptr[e] + 2 * (dg - 2 * e) - 1);
        }
        __syncthreads();
        qf *cur = nullptr;
        int cs = 0;  // s_S[cs]: the sum that belongs to cur
        for (int leaf = 0; leaf < 1 << g; ++leaf) {
            if (leaf) {
                // the depth whose choice turns include; deeper choices are excludes
                const int e = g - __ffs(leaf), d = dg - 2 * e;
                qf *dst = e + 1 == g ? Lv : base + kOffSl;
                if (e + 1 < g)
                    for (int x = 1; x <= e; ++x) dst += gsym(dg - 2 * x);
                tree_forward(base, 1, d, dptr + e, dst, nullptr, dQ + 3 * e, dRs + e, Zb, &s_bad);
                if (t == 0) {
                    dptr[e + 1] = (uint16_t)(dst - base);
                    for (int x = e + 1; x < g; ++x) dptr[x + 1] = (uint16_t)(dptr[x] + 2 * (dg - 2 * x) - 1);
                }
                __syncthreads();
            }
            if (t == 0) nptr[0] = dptr[g];
            __syncthreads();
            // the subtree, forward
            for (int l = 0; l < m; ++l) {
                const int np = 1 << l;
                tree_forward(base, np, 2 * (m - l), nptr + np - 1, Lv + lvl_off(l + 1), l < m - 1 ? nptr + 2 * np - 1 : nullptr,
                             nQ + 3 * (np - 1), nrs + np - 1, Zb, &s_bad);
            }
            // its last level: S = rs - 1, Gamma = -rs P^{-1} / 2
            qf *Ach = base + ((m - 1) & 1 ? kOffAdjB : kOffAdjA);
            for (int f = t; f < 4 << (m - 1); f += kTreeThreads) {
                const int c = f >> 2, x = f & 3, node = (1 << (m - 1)) - 1 + c;
                if (x == 3) {
                    nS[node] = nrs[node] - qf_one();
                    nA[node] = qf_approx(nrs[node]) + 1.0;
                } else {
                    const qf h = qf_half(nrs[node]), v = nQ[3 * node + x];
                    Ach[3 * c + x] = x == 1 ? h * v : qf_mul<true>(h, v);
                }
            }
            __syncthreads();
            for (int l = m - 2; l >= 0; --l) {
                const int np = 1 << l, d = 2 * (m - l);
                const qf *Ac = base + ((l + 1) & 1 ? kOffAdjB : kOffAdjA);
                qf *Ap = base + (l & 1 ? kOffAdjB : kOffAdjA);
                const int stc = gsym(d - 2);
                tree_backward(base, np, d, nptr + np - 1, Ac + stc, Ac, 2 * stc, Ap, nQ + 3 * (np - 1), nrs + np - 1,
                              nS + 2 * np, nS + 2 * np - 1, 2, nS + np - 1, nA + 2 * np, nA + 2 * np - 1,
                              nA + np - 1, Zb, Yb, M2, l < 2 ? 4 : l < 4 ? 2 : 1);
            }
            // up the group's tree: an include's adjoint joins the kept exclude's, an exclude's is kept
            cur = base + kOffAdjA;
            if (t == 0) {
                s_S[0] = nS[0];
                s_A[0] = nA[0];
            }
            cs = 0;
            __syncthreads();
            for (int e = g - 1; e >= 0; --e) {
                const int d = dg - 2 * e, stc = gsym(d - 2);
                qf *Gx = base + kOffGx;
                for (int x = 0; x < e; ++x) Gx += gsym(dg - 2 * (x + 1));
                if (leaf >> (g - 1 - e) & 1) {
                    qf *out = base + (cur == base + kOffAdjA ? kOffAdjB : kOffAdjA);
                    tree_backward(base, 1, d, dptr + e, cur, Gx, stc, out, dQ + 3 * e, dRs + e, s_S + cs, dS + e, 0,
                                  s_S + (cs ^ 1), s_A + cs, dA + e, s_A + (cs ^ 1), Zb, Yb, M2, 4);
                    cur = out;
                    cs ^= 1;
                } else {
                    for (int f = t; f < stc; f += kTreeThreads) Gx[f] = cur[f];
                    if (t == 0) {
                        dS[e] = s_S[cs];
                        dA[e] = s_A[cs];
                    }
                    __syncthreads();
                    break;
                }
            }
        }
        // the group's value and adjoint, back through its middle pivots and into Gam
        if (t == 0) {
            qf tau = qf_one();
            for (int e = 0; e < kh; ++e) tau = tau * hiRs[e];
            for (int e = 0; e < kl; ++e) tau = tau * prers[e];
            if ((q - g - k0) & 1) tau = -tau;
            s_S[cs ^ 1] = tau;
            s_V = tau * s_S[cs];
            s_T = s_T + s_V;
            s_Asum += fabs(qf_approx(tau)) * s_A[cs];
        }
        __syncthreads();
        for (int f = t; f < gsym(dg); f += kTreeThreads) Gf[tail(D0, dg) + f] = s_S[cs ^ 1] * cur[f];
        __syncthreads();
        for (int e = kl - 1; e >= 0; --e) {
            const int d = D0 - 2 * e;
            if (t == 0) s_off[0] = (uint16_t)(UM - base + tail(D0, d));
            __syncthreads();
            tree_backward(base, 1, d, s_off, Gf + tail(D0, d - 2), nullptr, 0, Gf + tail(D0, d), preQ + 3 * e, nullptr,
                          &s_V, nullptr, 0, nullptr, nullptr, nullptr, nullptr, Zb, Yb, M2, 4);
        }
        for (int f = t; f < gsym(D0); f += kTreeThreads) {
            int i, j;
            fold_ij(f, D0, i, j);
            qf &x = Gam[gpidx(Dr, umrow[i], umrow[j])];
            x = x + Gf[gpidx(D0, i, j)];
        }
        __syncthreads();
    }
    // the chunk: Gam as the adjoint of SM's trailing block, back through the high pivots
    // with the chunk's sum as their V
    for (int f = t; f < gsym(Dr); f += kTreeThreads) Gs[tail(Ds, Dr) + f] = Gam[f];
    __syncthreads();
    for (int e = kh - 1; e >= 0; --e) {
        const int d = Ds - 2 * e;
        if (t == 0) s_off[0] = (uint16_t)(SM - base + tail(Ds, d));
        __syncthreads();
        tree_backward(base, 1, d, s_off, Gs + tail(Ds, d - 2), nullptr, 0, Gs + tail(Ds, d), hiQ + 3 * e, nullptr, &s_T,
                      nullptr, 0, nullptr, nullptr, nullptr, nullptr, Zb, Yb, M2, 4);
    }
    // dense partial (row stride 2n): zero, then the chunk's rows
    for (int f = t; f < Dn * Dn; f += kTreeThreads) part[ch * pst + f] = qf_zero();
    __syncthreads();
    for (int f = t; f < gsym(Ds); f += kTreeThreads) {
        int i, j;
        fold_ij(f, Ds, i, j);
        const qf x = Gs[gpidx(Ds, i, j)];
        const int ri = smrow[i], rj = smrow[j];
        part[ch * pst + (size_t)ri * Dn + rj] = x;
        part[ch * pst + (size_t)rj * Dn + ri] = x;
    }
    if (t == 0) {
        part_T[ch] = s_T;
        part_A[ch] = n == 0 ? 1.0 : s_Asum;
        if (s_bad) atomicOr(flags + p, 1);
    }
}

// ---- the same adjoint in double-double --------------------------------------------------------
// For patterns whose sum cancels by more than kRedo: there the result is limited by the arithmetic
// (a relative error of about 3e-34 kappa in double-double, a tenth of that in qf, against a quadruple
// precision sum over the subsets), the two come to differ by 1e-9, and callers keep the values
// they had.  What the guess names beforehand (kappa.cuh) comes here alone.  CTAs of other patterns leave at
// once.  A batch with a few such patterns pays for one chunk's time here (about 5 ms on the 32-mode workload).
namespace ddk {
constexpr int kTM = 7;                   // modes of a unit's subtree (2^7 leaves)
constexpr int kTreeThreads = 128;

// level l of a unit's subtree: 2^l nodes of dimension 2 (kTM - l), packed, back to back
__host__ __device__ constexpr int lvl_off(int l) {
    int s = 0;
    for (int q = 0; q < l; ++q) s += (1 << q) * gsym(2 * (kTM - q));
    return s;
}
constexpr int lvl_cap() {
    int m = 0;
    for (int l = 0; l < kTM; ++l) m = (1 << l) * gsym(2 * (kTM - l)) > m ? (1 << l) * gsym(2 * (kTM - l)) : m;
    return m;
}
constexpr int y_cap() {
    int m = 2 * (kGD - 2);
    for (int l = 0; l < kTM; ++l) m = (1 << l) * 4 * (kTM - l - 1) > m ? (1 << l) * 4 * (kTM - l - 1) : m;
    return m;
}
constexpr int kNodes = (1 << kTM) - 1;   // nodes of levels 0..kTM-1
// shared memory (double-double elements)
constexpr int kChunkBits = 8;           // a chunk: at most 2^8 units sharing their high prefix modes
constexpr int kUD = 2 * (kChunkBits + kTM);  // largest unit matrix (low prefix modes + subtree)
// SM: the chunk's matrix (included high prefix modes, every low prefix mode, the subtree
// modes), then its adjoint Gs; UM, Gf: one unit's matrix and adjoint; Gam: the adjoint of
// SM's trailing block after the high pivots, summed over the chunk's units
constexpr int kOffSM = 0, kOffGs = gsym(kGD), kOffUM = 2 * gsym(kGD), kOffGf = kOffUM + gsym(kUD),
              kOffGam = kOffGf + gsym(kUD), kOffLv = kOffGam + gsym(kUD);
constexpr int kOffAdjA = kOffLv + lvl_off(kTM), kOffAdjB = kOffAdjA + lvl_cap();
constexpr int kOffQ = kOffAdjB + lvl_cap(), kOffRs = kOffQ + 3 * kNodes, kOffS = kOffRs + kNodes;
constexpr int kOffY = kOffS + kNodes, kOffPreQ = kOffY + y_cap(), kOffPreRs = kOffPreQ + 3 * kGradMaxN;
constexpr int kOffHiQ = kOffPreRs + kGradMaxN, kOffHiRs = kOffHiQ + 3 * kGradMaxN;
constexpr int kTreeSmem = kOffHiRs + kGradMaxN;

// One 2x2 pivot of the packed D x D unit matrix, eliminated by the CTA: rows and
// columns >= c0 + 2 receive C - W B^T (W = B P^{-1}); the pivot rows stay as they were
// (the reverse pass reads them).  Returns det^{-1/2}; stores P^{-1} and det^{-1/2}.
__device__ dd tree_pivot(dd *UM, int D, int c0, dd *Wb, dd *Qout, dd *rsout, int *bad) {
    const int t = threadIdx.x;
    const dd p00 = UM[gpidx(D, c0, c0)], p01 = UM[gpidx(D, c0, c0 + 1)], p11 = UM[gpidx(D, c0 + 1, c0 + 1)];
    const dd det = dd_dot2(p00, p11, -p01, p01);
    const dd rs = dd_rsqrt(det), inv = rs * rs;
    const dd q00 = p11 * inv, q01 = -p01 * inv, q11 = p00 * inv;
    if (t == 0) {
        Qout[0] = q00;
        Qout[1] = q01;
        Qout[2] = q11;
        *rsout = rs;
        if (!(det.hi > 0.0)) atomicOr(bad, 1);
    }
    const int Dt = D - c0 - 2;
    for (int i = t; i < Dt; i += kTreeThreads) {
        const dd b0 = UM[gpidx(D, c0, c0 + 2 + i)], b1 = UM[gpidx(D, c0 + 1, c0 + 2 + i)];
        Wb[2 * i] = dd_dot2(q00, b0, q01, b1);
        Wb[2 * i + 1] = dd_dot2(q01, b0, q11, b1);
    }
    __syncthreads();
    for (int f = t; f < gsym(Dt); f += kTreeThreads) {
        int i, j;
        fold_ij(f, Dt, i, j);
        dd &c = UM[gpidx(D, c0 + 2 + i, c0 + 2 + j)];
        c = dd_fms2(c, Wb[2 * i], UM[gpidx(D, c0, c0 + 2 + j)], Wb[2 * i + 1], UM[gpidx(D, c0 + 1, c0 + 2 + j)]);
    }
    __syncthreads();
    return rs;
}

// Back through the pivots e = np - 1 .. 0 of the packed D x D matrix Mx (pivot rows kept):
// G holds the adjoint of the trailing block below the last pivot; each pivot adds its rows,
// -rs Y with Y = P^{-1} B G, and its block, (Y B^T P^{-1})(i, j) - V P^{-1} / 2 (the
// prefactor's det^{-1/2}, V the value it multiplies).  Q: 3 entries of P^{-1} per pivot.
__device__ void reverse_pivots(const dd *Mx, dd *G, int D, int np, const dd *Qs, dd V, dd *Yb) {
    const int t = threadIdx.x;
    for (int e = np - 1; e >= 0; --e) {
        const int c0 = 2 * e, R = D - c0 - 2;
        const dd *Q = Qs + 3 * e;
        for (int j = t; j < R; j += kTreeThreads) {
            dd z0 = dd(0.0), z1 = dd(0.0);
            for (int i = 0; i < R; ++i) {
                const dd g = G[gpany(D, c0 + 2 + i, c0 + 2 + j)];
                z0 = z0 + Mx[gpidx(D, c0, c0 + 2 + i)] * g;
                z1 = z1 + Mx[gpidx(D, c0 + 1, c0 + 2 + i)] * g;
            }
            Yb[2 * j] = dd_dot2(Q[0], z0, Q[1], z1);
            Yb[2 * j + 1] = dd_dot2(Q[1], z0, Q[2], z1);
        }
        __syncthreads();
        for (int f = t; f < 2 * R + 3; f += kTreeThreads) {
            if (f < 2 * R) {
                const int a = f / R, j = f - a * R;
                G[gpidx(D, c0 + a, c0 + 2 + j)] = -Yb[2 * j + a];
            } else {
                const int i = (f - 2 * R) == 2 ? 1 : 0, j = (f - 2 * R) == 0 ? 0 : 1;
                dd yb0 = dd(0.0), yb1 = dd(0.0);
                for (int c = 0; c < R; ++c) {
                    const dd y = Yb[2 * c + i];
                    yb0 = yb0 + y * Mx[gpidx(D, c0, c0 + 2 + c)];
                    yb1 = yb1 + y * Mx[gpidx(D, c0 + 1, c0 + 2 + c)];
                }
                const dd qj0 = Q[j == 0 ? 0 : 1], qj1 = Q[j == 0 ? 1 : 2];
                G[gpidx(D, c0 + i, c0 + j)] = dd_dot2(yb0, qj0, yb1, qj1) - V * Q[i + j] * dd(0.5);
            }
        }
        __syncthreads();
    }
}

// Gbar_p = dT/dA_S by reverse mode through the include/exclude Schur recursion.
// Units = (pattern, include/exclude choice of the first q = n - m modes), m = min(n, 7).
// A unit's value V = (-1)^{q-k} tau_prefix S(root): its k included prefix modes are
// eliminated (pivot rows kept), then the subtree over the last m modes is expanded
// breadth first with every level kept, S(node) = rs S(include child) - S(exclude child)
// (S = 1 at a leaf).  Reverse, with Gamma(node) = dS(node)/dC_node:
//   rest block:  rs Gamma(inc) - Gamma(exc)
//   pivot rows:  -rs Y,  Y = P^{-1} B Gamma(inc)
//   pivot block: rs (Y B^T P^{-1} - S(inc) P^{-1} / 2)
// then back through the prefix pivots the same way (with -V P^{-1} / 2 from tau_prefix).
// One CTA per chunk: an aligned run of 2^b units of one pattern, whose first b prefix modes
// (the low ones) vary and the rest (the high ones) are fixed.  The chunk eliminates its
// included high modes once, from the matrix on its high, low and subtree rows (SM); each
// unit then takes SM's trailing block on its included low modes and the subtree, eliminates
// those, runs the subtree and its reverse, and adds its adjoint into the trailing block's
// (Gam); at the end Gam goes back through the high pivots once, with V = the chunk's sum
// (the adjoint of a shared step is linear in what flows into it), and the chunk's partial
// Gbar and T are written; the chunks of a pattern are summed in order afterwards.
__global__ void __launch_bounds__(kTreeThreads) grad_tree_dd_kernel(int M, const double *__restrict__ O,
                                                               const uint64_t *__restrict__ pats,
                                                               const int *__restrict__ chunk_p,
                                                               const long long *__restrict__ chunk_u, size_t pst,
                                                               const int *__restrict__ redo, dd *__restrict__ part,
                                                               dd *__restrict__ part_T, int *__restrict__ flags) {
    extern __shared__ __align__(16) unsigned char gsm[];
    dd *const base = (dd *)gsm;
    dd *const SM = base + kOffSM, *const Gs = base + kOffGs, *const UM = base + kOffUM, *const Gf = base + kOffGf;
    dd *const Gam = base + kOffGam, *const Lv = base + kOffLv;
    dd *const nQ = base + kOffQ, *const nrs = base + kOffRs, *const nS = base + kOffS, *const Yb = base + kOffY;
    dd *const preQ = base + kOffPreQ, *const prers = base + kOffPreRs;
    dd *const hiQ = base + kOffHiQ, *const hiRs = base + kOffHiRs;
    __shared__ int modes[128];
    __shared__ int smrow[kGD];   // row of SM -> pattern row (2 x detector index + x/p)
    __shared__ int umrow[kUD];   // row of a unit's matrix -> row of SM's trailing block
    __shared__ int s_n, s_kh, s_kl, s_bad;
    __shared__ dd s_T, s_V;
    const int t = threadIdx.x, ch = blockIdx.x, p = chunk_p[ch], N2 = 2 * M;
    if (!redo[p]) return;
    const long long u_begin = chunk_u[2 * ch], u_end = chunk_u[2 * ch + 1];
    if (t == 0) {
        int n = 0;
        for (int i = 0; i < M; ++i) {
            const uint64_t w = i < 64 ? pats[2 * p] : pats[2 * p + 1];
            if (w >> (i & 63) & 1ull) modes[n++] = i;
        }
        s_n = n;
        s_bad = 0;
        s_T = dd(n == 0 && u_begin == 0 ? 1.0 : 0.0);
    }
    __syncthreads();
    const int n = s_n, m = n < kTM ? n : kTM, q = n - m, Dn = 2 * n;
    // the chunk's 2^bl units vary the prefix modes 0..bl-1; modes bl..q-1 are fixed by u_begin
    const int bl = u_end > u_begin ? 63 - __clzll(u_end - u_begin) : 0;
    const long long hi = u_begin >> bl;
    if (t == 0) {
        int r = 0;
        for (int a = bl; a < q; ++a)
            if (hi >> (a - bl) & 1) {
                smrow[r++] = 2 * a;
                smrow[r++] = 2 * a + 1;
            }
        s_kh = r / 2;
        for (int a = 0; a < bl; ++a) {
            smrow[r++] = 2 * a;
            smrow[r++] = 2 * a + 1;
        }
        for (int a = q; a < n; ++a) {
            smrow[r++] = 2 * a;
            smrow[r++] = 2 * a + 1;
        }
    }
    __syncthreads();
    const int kh = s_kh, Ds = 2 * (kh + bl + m), Dr = 2 * (bl + m);
    // the chunk's rows of A = I - O (exact in double-double), its high pivots, and a zero Gam
    for (int f = t; f < gsym(Ds); f += kTreeThreads) {
        int i, j;
        fold_ij(f, Ds, i, j);
        const int ri = smrow[i], rj = smrow[j];
        const int gi = modes[ri >> 1] + (ri & 1) * M, gj = modes[rj >> 1] + (rj & 1) * M;
        SM[gpidx(Ds, i, j)] = dd_two_sum(i == j ? 1.0 : 0.0, -O[(size_t)gi * N2 + gj]);
    }
    for (int f = t; f < gsym(Dr); f += kTreeThreads) Gam[f] = dd(0.0);
    __syncthreads();
    dd tau_h = dd(1.0);
    for (int e = 0; e < kh; ++e) tau_h = tau_h * tree_pivot(SM, Ds, 2 * e, Yb, hiQ + 3 * e, hiRs + e, &s_bad);
    for (long long u = u_begin; n > 0 && u < u_end; ++u) {
        const long long lb = u - u_begin;
        if (t == 0) {
            int r = 0;
            for (int a = 0; a < bl; ++a)
                if (lb >> a & 1) {
                    umrow[r++] = 2 * a;
                    umrow[r++] = 2 * a + 1;
                }
            s_kl = r / 2;
            for (int a = 0; a < m; ++a) {
                umrow[r++] = 2 * (bl + a);
                umrow[r++] = 2 * (bl + a) + 1;
            }
        }
        __syncthreads();
        const int kl = s_kl, k = kh + kl, D0 = 2 * (kl + m), o = 2 * kh;
        // the unit's matrix: SM's trailing block on its included low modes and the subtree
        for (int f = t; f < gsym(D0); f += kTreeThreads) {
            int i, j;
            fold_ij(f, D0, i, j);
            UM[gpidx(D0, i, j)] = SM[gpidx(Ds, o + umrow[i], o + umrow[j])];
        }
        __syncthreads();
        dd tau = tau_h;
        for (int e = 0; e < kl; ++e) tau = tau * tree_pivot(UM, D0, 2 * e, Yb, preQ + 3 * e, prers + e, &s_bad);
        // level 0 of the subtree: the trailing 2m x 2m block
        for (int f = t; f < gsym(2 * m); f += kTreeThreads) {
            int i, j;
            fold_ij(f, 2 * m, i, j);
            Lv[gpidx(2 * m, i, j)] = UM[gpidx(D0, 2 * kl + i, 2 * kl + j)];
        }
        __syncthreads();
        // forward: pivots of every level, children of every level but the last
        for (int l = 0; l < m; ++l) {
            const int d = 2 * (m - l), dc = d - 2, np = 1 << l, st = gsym(d), stc = gsym(dc);
            const dd *Lp = Lv + lvl_off(l);
            for (int c = t; c < np; c += kTreeThreads) {
                const dd *P = Lp + c * st;
                const dd p00 = P[gpidx(d, 0, 0)], p01 = P[gpidx(d, 0, 1)], p11 = P[gpidx(d, 1, 1)];
                const dd det = dd_dot2(p00, p11, -p01, p01);
                const dd rs = dd_rsqrt(det), inv = rs * rs;
                const int node = np - 1 + c;
                nQ[3 * node] = p11 * inv;
                nQ[3 * node + 1] = -p01 * inv;
                nQ[3 * node + 2] = p00 * inv;
                nrs[node] = rs;
                if (!(det.hi > 0.0)) atomicOr(&s_bad, 1);
            }
            __syncthreads();
            if (l == m - 1) break;
            for (int f = t; f < np * dc; f += kTreeThreads) {
                const int cp = f / dc, i = f - cp * dc, node = np - 1 + cp;
                const dd *P = Lp + cp * st;
                const dd b0 = P[gpidx(d, 0, i + 2)], b1 = P[gpidx(d, 1, i + 2)];
                const dd q00 = nQ[3 * node], q01 = nQ[3 * node + 1], q11 = nQ[3 * node + 2];
                Yb[2 * f] = dd_dot2(q00, b0, q01, b1);
                Yb[2 * f + 1] = dd_dot2(q01, b0, q11, b1);
            }
            __syncthreads();
            dd *Lc = Lv + lvl_off(l + 1);
            for (int f = t; f < np * stc; f += kTreeThreads) {
                const int cp = f / stc, e = f - cp * stc;
                int i, j;
                fold_ij(e, dc, i, j);
                const dd *P = Lp + cp * st;
                const dd *W = Yb + 2 * (cp * dc + i);
                const dd v = P[gpidx(d, i + 2, j + 2)];
                Lc[(2 * cp) * stc + gpidx(dc, i, j)] = v;
                Lc[(2 * cp + 1) * stc + gpidx(dc, i, j)] =
                    dd_fms2(v, W[0], P[gpidx(d, 0, j + 2)], W[1], P[gpidx(d, 1, j + 2)]);
            }
            __syncthreads();
        }
        // subtree sums, leaves up
        for (int l = m - 1; l >= 0; --l) {
            const int np = 1 << l;
            for (int c = t; c < np; c += kTreeThreads) {
                const int node = np - 1 + c;
                if (l == m - 1) {
                    nS[node] = nrs[node] - dd(1.0);
                } else {
                    const int ch = 2 * np - 1 + 2 * c;  // exclude child; ch + 1 includes
                    nS[node] = nrs[node] * nS[ch + 1] - nS[ch];
                }
            }
            __syncthreads();
        }
        if (t == 0) {
            dd V = tau * nS[0];
            if ((q - k) & 1) V = -V;
            s_V = V;
            s_T += V;
        }
        __syncthreads();
        const dd V = s_V;
        // reverse through the subtree: the last level's pivot blocks, then upwards
        dd *Ach = base + ((m - 1) & 1 ? kOffAdjB : kOffAdjA);
        for (int c = t; c < (1 << (m - 1)); c += kTreeThreads) {
            const int node = (1 << (m - 1)) - 1 + c;
            const dd h = nrs[node] * dd(-0.5);
            Ach[3 * c] = h * nQ[3 * node];
            Ach[3 * c + 1] = h * nQ[3 * node + 1];
            Ach[3 * c + 2] = h * nQ[3 * node + 2];
        }
        __syncthreads();
        for (int l = m - 2; l >= 0; --l) {
            const int d = 2 * (m - l), dc = d - 2, np = 1 << l, st = gsym(d), stc = gsym(dc);
            const dd *Lp = Lv + lvl_off(l);
            const dd *Ac = base + ((l + 1) & 1 ? kOffAdjB : kOffAdjA);
            dd *Ap = base + (l & 1 ? kOffAdjB : kOffAdjA);
            // Y = P^{-1} B Gamma(inc), one column j per job
            for (int f = t; f < np * dc; f += kTreeThreads) {
                const int cp = f / dc, j = f - cp * dc, node = np - 1 + cp;
                const dd *P = Lp + cp * st;
                const dd *Gi = Ac + (2 * cp + 1) * stc;
                dd z0 = dd(0.0), z1 = dd(0.0);
                for (int i = 0; i < dc; ++i) {
                    const dd g = Gi[gpany(dc, i, j)];
                    z0 = z0 + P[gpidx(d, 0, i + 2)] * g;
                    z1 = z1 + P[gpidx(d, 1, i + 2)] * g;
                }
                const dd q00 = nQ[3 * node], q01 = nQ[3 * node + 1], q11 = nQ[3 * node + 2];
                Yb[2 * f] = dd_dot2(q00, z0, q01, z1);
                Yb[2 * f + 1] = dd_dot2(q01, z0, q11, z1);
            }
            __syncthreads();
            for (int f = t; f < np * st; f += kTreeThreads) {
                const int cp = f / st, e = f - cp * st, node = np - 1 + cp;
                int i, j;
                fold_ij(e, d, i, j);
                const dd rs = nrs[node];
                dd g;
                if (i >= 2) {
                    g = rs * Ac[(2 * cp + 1) * stc + gpidx(dc, i - 2, j - 2)] - Ac[(2 * cp) * stc + gpidx(dc, i - 2, j - 2)];
                } else if (j >= 2) {
                    g = -(rs * Yb[2 * (cp * dc + j - 2) + i]);
                } else {
                    // (Y B^T P^{-1})(i, j) - S(inc) P^{-1}(i, j) / 2, times rs
                    const dd *P = Lp + cp * st;
                    dd yb0 = dd(0.0), yb1 = dd(0.0);
                    for (int c = 0; c < dc; ++c) {
                        const dd y = Yb[2 * (cp * dc + c) + i];
                        yb0 = yb0 + y * P[gpidx(d, 0, c + 2)];
                        yb1 = yb1 + y * P[gpidx(d, 1, c + 2)];
                    }
                    const dd qj0 = nQ[3 * node + (j == 0 ? 0 : 1)], qj1 = nQ[3 * node + (j == 0 ? 1 : 2)];
                    const dd qij = nQ[3 * node + i + j];
                    g = rs * (dd_dot2(yb0, qj0, yb1, qj1) - nS[2 * np - 1 + 2 * cp + 1] * qij * dd(0.5));
                }
                Ap[cp * st + gpidx(d, i, j)] = g;
            }
            __syncthreads();
        }
        // the unit's adjoint: the root's, scaled, then back through its low pivots, then
        // into Gam at the unit's rows
        {
            const dd fac = (((q - k) & 1) ? -tau : tau);
            const dd *Ar = base + kOffAdjA;  // level 0
            for (int f = t; f < gsym(2 * m); f += kTreeThreads) {
                int i, j;
                fold_ij(f, 2 * m, i, j);
                Gf[gpidx(D0, 2 * kl + i, 2 * kl + j)] = fac * Ar[gpidx(2 * m, i, j)];
            }
        }
        __syncthreads();
        reverse_pivots(UM, Gf, D0, kl, preQ, V, Yb);
        for (int f = t; f < gsym(D0); f += kTreeThreads) {
            int i, j;
            fold_ij(f, D0, i, j);
            dd &g = Gam[gpidx(Dr, umrow[i], umrow[j])];
            g = g + Gf[gpidx(D0, i, j)];
        }
        __syncthreads();
    }
    // the chunk: Gam as the adjoint of SM's trailing block, back through the high pivots
    // with the chunk's sum as their V
    for (int f = t; f < gsym(Dr); f += kTreeThreads) {
        int i, j;
        fold_ij(f, Dr, i, j);
        Gs[gpidx(Ds, 2 * kh + i, 2 * kh + j)] = Gam[gpidx(Dr, i, j)];
    }
    __syncthreads();
    reverse_pivots(SM, Gs, Ds, kh, hiQ, s_T, Yb);
    // dense partial (row stride 2n): zero, then the chunk's rows
    for (int f = t; f < Dn * Dn; f += kTreeThreads) part[ch * pst + f] = dd(0.0);
    __syncthreads();
    for (int f = t; f < gsym(Ds); f += kTreeThreads) {
        int i, j;
        fold_ij(f, Ds, i, j);
        const dd g = Gs[gpidx(Ds, i, j)];
        const int ri = smrow[i], rj = smrow[j];
        part[ch * pst + (size_t)ri * Dn + rj] = g;
        part[ch * pst + (size_t)rj * Dn + ri] = g;
    }
    if (t == 0) {
        part_T[ch] = s_T;
        if (s_bad) atomicOr(flags + p, 1);
    }
}

}  // namespace ddk

// the patterns that the double-double kernel takes: kappa = sum |terms| / |T| above kRedo (or no number), a
// pivot that is not positive, or left out by the first kernel (kappa.cuh); their flags start afresh
constexpr double kRedo = 1e24;
__global__ void grad_redo_kernel(int n_pat, const long long *__restrict__ chunk_off, const qf *__restrict__ part_T,
                                 const double *__restrict__ part_A, int *__restrict__ redo, int *__restrict__ flags) {
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pat) return;
    qf T = qf_zero();
    double A = 0.0;
    for (long long c = chunk_off[p]; c < chunk_off[p + 1]; ++c) {
        T = T + part_T[c];
        A += part_A[c];
    }
    redo[p] = flags[p] == 0 && A < kRedo * fabs(qf_approx(T)) ? 0 : 1;
    if (redo[p]) flags[p] = 0;
}

// per pattern: sum the chunk partials in order, F_p = (w_p / T_p) Gbar_p, log P_p
__global__ void grad_finalize_kernel(int M, const uint64_t *__restrict__ pats, int n_pat,
                                     const long long *__restrict__ chunk_off, size_t pst,
                                     const int *__restrict__ redo, const qf *__restrict__ part,
                                     const qf *__restrict__ part_T, const double *__restrict__ w,
                                     const double *__restrict__ logdet, double *__restrict__ F,
                                     double *__restrict__ logP, int32_t *__restrict__ status,
                                     const int *__restrict__ flags) {
    const int p = blockIdx.x;
    __shared__ double s_scale;
    __shared__ int s_n;
    if (threadIdx.x == 0) {
        int n = __popcll(pats[2 * p]) + __popcll(pats[2 * p + 1]);
        s_n = n;
        dd T = dd(0.0);
        if (redo[p]) {
            for (long long c = chunk_off[p]; c < chunk_off[p + 1]; ++c) T += ((const dd *)part_T)[c];
        } else {
            qf Tq = qf_zero();
            for (long long c = chunk_off[p]; c < chunk_off[p + 1]; ++c) Tq = Tq + part_T[c];
            T = qf_to_dd(Tq);
        }
        int st = flags[p] ? GBS_E_NOT_SPD : (T.hi > 0.0 ? GBS_OK : GBS_E_NONPOSITIVE);
        if (status) status[p] = st;
        if (logP) logP[p] = st ? nan("") : -0.5 * (*logdet) + log(T.hi) + log1p(T.lo / T.hi);
        s_scale = st ? 0.0 : w[p] / (T.hi + T.lo);
    }
    __syncthreads();
    const int D = 2 * s_n;
    for (int f = threadIdx.x; f < D * D; f += blockDim.x) {
        dd s = dd(0.0);
        if (redo[p]) {
            for (long long c = chunk_off[p]; c < chunk_off[p + 1]; ++c) s += ((const dd *)part)[(size_t)c * pst + f];
        } else {
            qf sq = qf_zero();
            for (long long c = chunk_off[p]; c < chunk_off[p + 1]; ++c) sq = sq + part[(size_t)c * pst + f];
            s = qf_to_dd(sq);
        }
        F[(size_t)p * kGD * kGD + f] = (s.hi + s.lo) * s_scale;
    }
}

// H[i][j] = sum_p F_p at the rows of S_p (patterns in order: deterministic); sumw
__global__ void grad_scatter_kernel(int M, const uint64_t *__restrict__ pats, int n_pat,
                                    const double *__restrict__ F, size_t fst, const double *__restrict__ w,
                                    double *__restrict__ H, double *__restrict__ sumw) {
    const int N = 2 * M;
    const int i = blockIdx.y * blockDim.y + threadIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
    if (i == 0 && j == 0) {
        double s = 0.0;
        for (int p = 0; p < n_pat; ++p) s += w[p];
        *sumw = s;
    }
    if (i >= N || j >= N) return;
    const int mi = i < M ? i : i - M, ai = i < M ? 0 : 1;
    const int mj = j < M ? j : j - M, aj = j < M ? 0 : 1;
    double h = 0.0;
    for (int p = 0; p < n_pat; ++p) {
        const uint64_t lo = pats[2 * p], hi = pats[2 * p + 1];
        auto has = [&](int m) { return ((m < 64 ? lo >> m : hi >> (m - 64)) & 1ull) != 0; };
        if (!has(mi) || !has(mj)) continue;
        // S-local index = rank of the mode among the clicked ones
        auto rank = [&](int m) {
            int r = __popcll(lo & (m >= 64 ? ~0ull : ((1ull << m) - 1)));
            if (m >= 64) r += __popcll(hi & ((1ull << (m - 64)) - 1));
            return r;
        };
        const int n = __popcll(lo) + __popcll(hi);
        const int D = 2 * n;
        h += F[(size_t)p * fst + (2 * rank(mi) + ai) * D + (2 * rank(mj) + aj)];
    }
    H[(size_t)i * N + j] = h;
}

// C = X Y for N x N row-major matrices, with X, Y = I - O when the flag says so
__global__ void grad_matmul_kernel(int N, const double *__restrict__ X, int x_is_A,
                                   const double *__restrict__ Y, int y_is_A, double *__restrict__ C) {
    const int i = blockIdx.y * blockDim.y + threadIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N || j >= N) return;
    double s = 0.0;
    for (int k = 0; k < N; ++k) {
        double x = X[(size_t)i * N + k], y = Y[(size_t)k * N + j];
        if (x_is_A) x = (i == k ? 1.0 : 0.0) - x;
        if (y_is_A) y = (k == j ? 1.0 : 0.0) - y;
        s = fma(x, y, s);
    }
    C[(size_t)i * N + j] = s;
}

// dsigma_Q = -1/2 sumw A - AHA   (AHA precomputed)
__global__ void grad_sigma_kernel(int N, const double *__restrict__ O, const double *__restrict__ AHA,
                                  const double *__restrict__ sumw, double *__restrict__ dsq) {
    const int i = blockIdx.y * blockDim.y + threadIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N || j >= N) return;
    const double a = (i == j ? 1.0 : 0.0) - O[(size_t)i * N + j];
    dsq[(size_t)i * N + j] = -0.5 * (*sumw) * a - AHA[(size_t)i * N + j];
}

// chain: dR = 2 eta W R diag(d), dr_j, deta (W the symmetrised dsigma_Q)
__device__ __forceinline__ double R_of(const double *U, int M, int i, int j) {
    int ui = i < M ? i : i - M, uj = j < M ? j : j - M;
    double re = U[2 * (ui * M + uj)], im = U[2 * (ui * M + uj) + 1];
    if (i < M) return j < M ? re : -im;
    return j < M ? im : re;
}

// WR = W R with W = (dsq + dsq^T)/2
__global__ void grad_wr_kernel(int M, const double *__restrict__ U, const double *__restrict__ dsq,
                               double *__restrict__ WR) {
    const int N = 2 * M;
    const int i = blockIdx.y * blockDim.y + threadIdx.y, j = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= N || j >= N) return;
    double s = 0.0;
    for (int k = 0; k < N; ++k) s += 0.5 * (dsq[(size_t)i * N + k] + dsq[(size_t)k * N + i]) * R_of(U, M, k, j);
    WR[(size_t)i * N + j] = s;
}

// one CTA: the 2M weights (an exp each) once, and the columns' sums q_j = (R^T W R)_jj side by side.
// (One thread's chains over 4 M^2 terms and four exps an entry of dU took 390 us at 32 modes.)
constexpr int kParamThreads = 1024;
__global__ void __launch_bounds__(kParamThreads)
    grad_params_kernel(int M, const double *__restrict__ U, const double *__restrict__ r, double eta,
                       const double *__restrict__ dsq, const double *__restrict__ pw, double *__restrict__ dU,
                       double *__restrict__ dr, double *__restrict__ deta) {
    __shared__ double dv[256], q[256];
    const int N = 2 * M, t = threadIdx.x;
    for (int j = t; j < N; j += kParamThreads) dv[j] = 0.5 * exp(j < M ? -2.0 * r[j] : 2.0 * r[j - M]);
    // q_j = sum_k R_kj (W R)_kj: warp w sums rows w, w + 32, ... of 32 columns
    __shared__ double sums[32][33];
    const int lane = t & 31, wp = t >> 5;
    for (int j0 = 0; j0 < N; j0 += 32) {
        const int j = j0 + lane;
        double s = 0.0;
        if (j < N)
            for (int k = wp; k < N; k += 32) s += R_of(U, M, k, j) * pw[(size_t)k * N + j];
        sums[wp][lane] = s;
        __syncthreads();
        double v = sums[lane][wp];  // column j0 + wp
        for (int off = 16; off; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
        if (lane == 0 && j0 + wp < N) q[j0 + wp] = v;
        __syncthreads();
    }
    // dU from dR = 2 eta (W R) diag(d)
    for (int f = t; f < M * M; f += kParamThreads) {
        const int i = f / M, j = f - i * M;
        const double dr_ij = 2 * eta * pw[i * N + j] * dv[j], dr_iMjM = 2 * eta * pw[(i + M) * N + j + M] * dv[j + M];
        const double dr_ijM = 2 * eta * pw[i * N + j + M] * dv[j + M], dr_iMj = 2 * eta * pw[(i + M) * N + j] * dv[j];
        dU[2 * f] = dr_ij + dr_iMjM;
        dU[2 * f + 1] = -dr_ijM + dr_iMj;
    }
    for (int j = t; j < M; j += kParamThreads) dr[j] = eta * (-2.0 * dv[j] * q[j] + 2.0 * dv[j + M] * q[j + M]);
    if (wp == 0) {
        double s = 0.0;
        for (int j = lane; j < N; j += 32) s += dv[j] * q[j] - 0.5 * dsq[(size_t)j * N + j];
        for (int off = 16; off; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
        if (lane == 0) *deta = s;
    }
}

// ---- the rectangular mesh ----------------------------------------------------------------------
// Layer l holds the cells on modes (m, m + 1) with m of the parity of l; its cells act on disjoint
// rows and every column of U evolves by itself.  One cluster of eight CTAs, each with an eighth of
// the columns (C lanes a cell, C a power of two); the sines and cosines of a chunk of layers are
// computed once per cluster and copied through distributed shared memory.  Cell after cell in one
// CTA, with the sines on every thread, the chain of 496 cells at 32 modes took 1.37 ms forward
// and 2.97 ms backward on a GB300; layer by layer it is 27 and 70 us.
namespace cg = cooperative_groups;
constexpr int kMeshCtas = 8, kMeshThreads = 256, kMeshCells = 512;  // cells of a chunk: whole layers

__host__ __device__ constexpr int mesh_cells(int M, int l) { return (M - (l & 1)) / 2; }
// cells before layer l
__host__ __device__ constexpr int mesh_base(int M, int l) { return ((l + 1) / 2) * (M / 2) + (l / 2) * ((M - 1) / 2); }
__host__ __device__ inline int mesh_lanes(int M) {
    int C = 1;
    while (C * kMeshCtas < M) C *= 2;
    return C;
}
struct sc4 {
    double st, ct, sp, cp;
};
// the sines and cosines of cells c0 .. c1-1 into cells[0 ..], every CTA of the cluster a share
__device__ void mesh_angles(const cg::cluster_group &cl, int c0, int c1, const double *theta, const double *phi,
                            sc4 *cells) {
    const int rank = (int)cl.block_rank();
    for (int f = rank + kMeshCtas * threadIdx.x; f < 2 * (c1 - c0); f += kMeshCtas * kMeshThreads) {
        const int c = f >> 1;
        double s, co;
        sincos(f & 1 ? phi[c0 + c] : theta[c0 + c], &s, &co);
        double *o = &cells[c].st + 2 * (f & 1);
        o[0] = s;
        o[1] = co;
    }
    cl.sync();
    for (int f = threadIdx.x; f < 2 * (c1 - c0); f += kMeshThreads) {
        const int own = f & (kMeshCtas - 1);
        if (own == rank) continue;
        const double *src = cl.map_shared_rank(&cells[f >> 1].st + 2 * (f & 1), own);
        double *o = &cells[f >> 1].st + 2 * (f & 1);
        o[0] = src[0];
        o[1] = src[1];
    }
    cl.sync();
}

__global__ void __cluster_dims__(kMeshCtas, 1, 1) __launch_bounds__(kMeshThreads)
    clements_unitary_kernel(int M, int C, const double *__restrict__ theta, const double *__restrict__ phi,
                            double *__restrict__ U) {
    extern __shared__ __align__(16) double cs[];
    sc4 *cells = (sc4 *)cs;                  // kMeshCells
    double2 *Uc = (double2 *)(cells + kMeshCells);  // M x C: this CTA's columns
    const cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x, col0 = (int)cl.block_rank() * C;
    for (int f = t; f < M * C; f += kMeshThreads) Uc[f] = make_double2(f / C == col0 + f % C ? 1.0 : 0.0, 0.0);
    __syncthreads();
    for (int l0 = 0; l0 < M;) {
        int l1 = l0 + 1;
        while (l1 < M && mesh_base(M, l1 + 1) - mesh_base(M, l0) <= kMeshCells) ++l1;
        const int c0 = mesh_base(M, l0);
        mesh_angles(cl, c0, mesh_base(M, l1), theta, phi, cells);
        for (int l = l0; l < l1; ++l) {
            for (int f = t; f < mesh_cells(M, l) * C; f += kMeshThreads) {
                const int x = f / C, col = f - x * C, m = (l & 1) + 2 * x;
                const sc4 k = cells[mesh_base(M, l) - c0 + x];
                const double2 a = Uc[m * C + col], b = Uc[(m + 1) * C + col];
                const double ear = k.cp * a.x - k.sp * a.y, eai = k.cp * a.y + k.sp * a.x;  // e^{i phi} a
                Uc[m * C + col] = make_double2(k.ct * ear - k.st * b.x, k.ct * eai - k.st * b.y);
                Uc[(m + 1) * C + col] = make_double2(k.st * ear + k.ct * b.x, k.st * eai + k.ct * b.y);
            }
            __syncthreads();
        }
        l0 = l1;
    }
    for (int f = t; f < M * C; f += kMeshThreads) {
        const int row = f / C, col = col0 + f % C;
        if (col < M) {
            U[2 * (row * M + col)] = Uc[f].x;
            U[2 * (row * M + col) + 1] = Uc[f].y;
        }
    }
}

// reverse pass through the mesh: the cell inputs are recovered from its outputs
// (T is unitary), so no forward storage is needed
__global__ void __cluster_dims__(kMeshCtas, 1, 1) __launch_bounds__(kMeshThreads)
    clements_grad_kernel(int M, int C, const double *__restrict__ theta, const double *__restrict__ phi,
                         const double *__restrict__ Ufinal, const double *__restrict__ dU,
                         double *__restrict__ dtheta, double *__restrict__ dphi) {
    extern __shared__ __align__(16) double cs[];
    sc4 *cells = (sc4 *)cs;                          // kMeshCells
    double2 *sums = (double2 *)(cells + kMeshCells);  // kMeshCells: this CTA's share of (dtheta, dphi)
    double2 *Uc = sums + kMeshCells, *G = Uc + M * C;
    const cg::cluster_group cl = cg::this_cluster();
    const int t = threadIdx.x, rank = (int)cl.block_rank(), col0 = rank * C;
    for (int f = t; f < M * C; f += kMeshThreads) {
        const int row = f / C, col = col0 + f % C;
        const bool in = col < M;  // columns beyond the last: zero, and they stay zero
        const size_t at = 2 * ((size_t)row * M + (in ? col : 0));
        Uc[f] = in ? make_double2(Ufinal[at], Ufinal[at + 1]) : make_double2(0.0, 0.0);
        G[f] = in ? make_double2(dU[at], dU[at + 1]) : make_double2(0.0, 0.0);
    }
    __syncthreads();
    for (int l1 = M; l1 > 0;) {
        int l0 = l1 - 1;
        while (l0 > 0 && mesh_base(M, l1) - mesh_base(M, l0 - 1) <= kMeshCells) --l0;
        const int c0 = mesh_base(M, l0), c1 = mesh_base(M, l1);
        mesh_angles(cl, c0, c1, theta, phi, cells);
        for (int l = l1 - 1; l >= l0; --l) {
            const int jobs = mesh_cells(M, l) * C;
            for (int f0 = 0; f0 < jobs; f0 += kMeshThreads) {  // whole warps: the sums over C lanes
                const int f = f0 + t, x = min(f, jobs - 1) / C, col = f & (C - 1), m = (l & 1) + 2 * x;
                const sc4 k = cells[mesh_base(M, l) - c0 + x];
                double gth = 0.0, gph = 0.0;
                if (f < jobs) {
                    const double2 o0 = Uc[m * C + col], o1 = Uc[(m + 1) * C + col];
                    // inputs: e a = ct o0 + st o1, b = -st o0 + ct o1
                    const double ear = k.ct * o0.x + k.st * o1.x, eai = k.ct * o0.y + k.st * o1.y;
                    const double br = -k.st * o0.x + k.ct * o1.x, bi = -k.st * o0.y + k.ct * o1.y;
                    const double2 g0 = G[m * C + col], g1 = G[(m + 1) * C + col];
                    // do0/dtheta = -st (e a) - ct b, do1/dtheta = ct (e a) - st b
                    const double d0r = -k.st * ear - k.ct * br, d0i = -k.st * eai - k.ct * bi;
                    const double d1r = k.ct * ear - k.st * br, d1i = k.ct * eai - k.st * bi;
                    gth = g0.x * d0r + g0.y * d0i + g1.x * d1r + g1.y * d1i;
                    // do0/dphi = i ct (e a), do1/dphi = i st (e a)
                    gph = g0.x * (-k.ct * eai) + g0.y * (k.ct * ear) + g1.x * (-k.st * eai) + g1.y * (k.st * ear);
                    // a = e^{-i phi} (e a); adjoint inputs G_a = e^{-i phi} (ct g0 + st g1), G_b = -st g0 + ct g1
                    const double hr = k.ct * g0.x + k.st * g1.x, hi = k.ct * g0.y + k.st * g1.y;
                    G[m * C + col] = make_double2(k.cp * hr + k.sp * hi, k.cp * hi - k.sp * hr);
                    G[(m + 1) * C + col] = make_double2(-k.st * g0.x + k.ct * g1.x, -k.st * g0.y + k.ct * g1.y);
                    Uc[m * C + col] = make_double2(k.cp * ear + k.sp * eai, k.cp * eai - k.sp * ear);
                    Uc[(m + 1) * C + col] = make_double2(br, bi);
                }
                for (int off = 1; off < C; off <<= 1) {
                    gth += __shfl_xor_sync(0xffffffffu, gth, off);
                    gph += __shfl_xor_sync(0xffffffffu, gph, off);
                }
                if (f < jobs && col == 0) sums[mesh_base(M, l) - c0 + x] = make_double2(gth, gph);
            }
            __syncthreads();
        }
        cl.sync();
        // the CTAs' shares, in rank order
        for (int c = rank + kMeshCtas * t; c < c1 - c0; c += kMeshCtas * kMeshThreads) {
            double2 s = make_double2(0.0, 0.0);
            for (int r = 0; r < kMeshCtas; ++r) {
                const double2 v = cl.map_shared_rank(sums, r)[c];
                s.x += v.x;
                s.y += v.y;
            }
            dtheta[c0 + c] = s.x;
            dphi[c0 + c] = s.y;
        }
        cl.sync();  // before the sums are written again, or a CTA exits
        l1 = l0;
    }
}

// one partial per pattern
size_t al(size_t x) { return (x + 255) / 256 * 256; }

}  // namespace

int grad_sigmaQ(gbs_ctx *ctx, int M, const double *O, const double *logdet, const uint64_t *pats,
                int n_pat, const double *w, double *dsq, double *logP, int32_t *status) {
    // every pattern must be valid and have at most kGradMaxN clicks: checked on the host
    // from a copy of the pattern words (one small readback), which also sizes the chunks
    size_t pb = (size_t)n_pat * 16;
    uint64_t *hp = (uint64_t *)malloc(pb + 16);
    if (!hp) return gbs_fail(ctx, GBS_E_NOMEM, "gbs_grad: host buffer");
    GBS_CUDA(ctx, cudaMemcpyAsync(hp, pats, pb, cudaMemcpyDeviceToHost, ctx->stream));
    GBS_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
    long long total_units = 0;
    int n_max = 0;
    for (int p = 0; p < n_pat; ++p) {
        uint64_t lo = hp[2 * p], hi = hp[2 * p + 1];
        int n = __builtin_popcountll(lo) + __builtin_popcountll(hi);
        bool out_of_range = (M < 64 && (lo >> M)) || (M <= 64 && hi) || (M > 64 && M < 128 && (hi >> (M - 64)));
        if (n > kGradMaxN || out_of_range) {
            free(hp);
            return gbs_fail(ctx, GBS_E_INVALID, "gbs_grad: pattern %d has %d clicks (at most %d) or a detector >= M",
                            p, n, kGradMaxN);
        }
        total_units += 1ll << (n > kTM ? n - kTM : 0);
        n_max = n > n_max ? n : n_max;
    }
    // chunks: aligned runs of `per` = 2^b consecutive units of one pattern (all of them if it
    // has fewer), b sized for about 32 chunks per SM over the whole batch and at most
    // kChunkBits: the largest patterns no longer set the time of the launch alone, and the
    // more of the prefix modes are fixed within a chunk, the more pivots its units share
    // (82 ms against 109 ms with 8 chunks per SM on the 32-mode workload)
    const long long target = 32ll * ctx->num_sms;
    long long per = 1;
    while (per < (1ll << kChunkBits) && per * target < total_units) per *= 2;
    long long chunks = 0;
    for (int p = 0; p < n_pat; ++p) {
        const int n = __builtin_popcountll(hp[2 * p]) + __builtin_popcountll(hp[2 * p + 1]);
        const long long units = 1ll << (n > kTM ? n - kTM : 0);
        chunks += (units + per - 1) / per;
    }
    const size_t tb = sizeof(long long) * ((size_t)n_pat + 1) + sizeof(long long) * 2 * (size_t)chunks +
                      sizeof(int) * (size_t)chunks;
    char *ht = (char *)malloc(tb);
    if (!ht) {
        free(hp);
        return gbs_fail(ctx, GBS_E_NOMEM, "gbs_grad: host buffer");
    }
    long long *h_off = (long long *)ht, *h_u = h_off + (n_pat + 1);
    int *h_p = (int *)(h_u + 2 * chunks);
    long long c = 0;
    for (int p = 0; p < n_pat; ++p) {
        const int n = __builtin_popcountll(hp[2 * p]) + __builtin_popcountll(hp[2 * p + 1]);
        const long long units = 1ll << (n > kTM ? n - kTM : 0);
        h_off[p] = c;
        for (long long u0 = 0; u0 < units; u0 += per, ++c) {
            h_p[c] = p;
            h_u[2 * c] = u0;
            h_u[2 * c + 1] = u0 + per < units ? u0 + per : units;
        }
    }
    h_off[n_pat] = c;
    free(hp);
    const int N = 2 * M;
    const size_t pst = (size_t)(2 * n_max) * (2 * n_max);  // one chunk's dense partial (row stride 2n)
    size_t o_off = 0, o_cu = al(o_off + 8 * ((size_t)n_pat + 1)), o_cp = al(o_cu + 16 * (size_t)chunks),
           o_flags = al(o_cp + 4 * (size_t)chunks), o_part = al(o_flags + 4 * (size_t)n_pat),
           o_pT = al(o_part + sizeof(qf) * (size_t)chunks * pst), o_pA = al(o_pT + sizeof(qf) * (size_t)chunks),
           o_redo = al(o_pA + 8 * (size_t)chunks),
           o_F = al(o_redo + 4 * (size_t)n_pat), o_H = al(o_F + 8 * (size_t)n_pat * kGD * kGD),
           o_T1 = al(o_H + 8 * (size_t)N * N), o_T2 = al(o_T1 + 8 * (size_t)N * N), o_sw = al(o_T2 + 8 * (size_t)N * N),
           total = o_sw + 64;
    int st = gbs_ws_ensure(ctx, total);
    if (st) {
        free(ht);
        return st;
    }
    char *b = (char *)ctx->ws;
    long long *chunk_off = (long long *)(b + o_off), *chunk_u = (long long *)(b + o_cu);
    int *chunk_p = (int *)(b + o_cp);
    int *flags = (int *)(b + o_flags);
    qf *part = (qf *)(b + o_part), *pT = (qf *)(b + o_pT);
    double *pA = (double *)(b + o_pA);
    int *redo = (int *)(b + o_redo);
    double *F = (double *)(b + o_F), *H = (double *)(b + o_H), *T1 = (double *)(b + o_T1),
           *T2 = (double *)(b + o_T2), *sw = (double *)(b + o_sw);
    // the chunk table (copied before the host buffer is released)
    cudaError_t ce = cudaMemcpyAsync(chunk_off, h_off, sizeof(long long) * ((size_t)n_pat + 1),
                                     cudaMemcpyHostToDevice, ctx->stream);
    if (ce == cudaSuccess)
        ce = cudaMemcpyAsync(chunk_u, h_u, sizeof(long long) * 2 * (size_t)chunks, cudaMemcpyHostToDevice, ctx->stream);
    if (ce == cudaSuccess)
        ce = cudaMemcpyAsync(chunk_p, h_p, sizeof(int) * (size_t)chunks, cudaMemcpyHostToDevice, ctx->stream);
    if (ce == cudaSuccess) ce = cudaStreamSynchronize(ctx->stream);
    free(ht);
    GBS_CUDA(ctx, ce);
    GBS_CUDA(ctx, cudaMemsetAsync(flags, 0, sizeof(int) * (size_t)n_pat, ctx->stream));
    const size_t smem = sizeof(qf) * (size_t)tree_smem(n_max);
    GBS_CUDA(ctx, cudaFuncSetAttribute(grad_tree_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    st = gbs_timing_begin(ctx);
    if (st) return st;
    grad_tree_kernel<<<(unsigned)chunks, kTreeThreads, smem, ctx->stream>>>(M, O, pats, chunk_p, chunk_u, pst, part, pT,
                                                                           pA, flags);
    GBS_CUDA(ctx, cudaGetLastError());
    grad_redo_kernel<<<(n_pat + 127) / 128, 128, 0, ctx->stream>>>(n_pat, chunk_off, pT, pA, redo, flags);
    const size_t dsmem = sizeof(dd) * (size_t)ddk::kTreeSmem;
    GBS_CUDA(ctx, cudaFuncSetAttribute(ddk::grad_tree_dd_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)dsmem));
    ddk::grad_tree_dd_kernel<<<(unsigned)chunks, ddk::kTreeThreads, dsmem, ctx->stream>>>(
        M, O, pats, chunk_p, chunk_u, pst, redo, (dd *)part, (dd *)pT, flags);
    GBS_CUDA(ctx, cudaGetLastError());
    st = gbs_timing_end(ctx);
    if (st) return st;
    grad_finalize_kernel<<<n_pat, 256, 0, ctx->stream>>>(M, pats, n_pat, chunk_off, pst, redo, part, pT, w, logdet, F,
                                                         logP, status, flags);
    GBS_CUDA(ctx, cudaGetLastError());
    return grad_chain_sigma(ctx, M, O, pats, n_pat, F, (size_t)kGD * kGD, w, H, T1, T2, sw, dsq);
}

int grad_chain_sigma(gbs_ctx *ctx, int M, const double *O, const uint64_t *pats, int n_pat, const double *F,
                     size_t fst, const double *w, double *H, double *T1, double *T2, double *sw, double *dsq) {
    const int N = 2 * M;
    dim3 blk(16, 16), grd((N + 15) / 16, (N + 15) / 16);
    grad_scatter_kernel<<<grd, blk, 0, ctx->stream>>>(M, pats, n_pat, F, fst, w, H, sw);
    grad_matmul_kernel<<<grd, blk, 0, ctx->stream>>>(N, H, 0, O, 1, T1);    // H A
    grad_matmul_kernel<<<grd, blk, 0, ctx->stream>>>(N, O, 1, T1, 0, T2);   // A (H A)
    grad_sigma_kernel<<<grd, blk, 0, ctx->stream>>>(N, O, T2, sw, dsq);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}

int grad_params(gbs_ctx *ctx, int M, const double *U, const double *r, double eta, const double *dsq,
                double *dU, double *dr, double *deta) {
    const int N = 2 * M;
    int st = gbs_ws_ensure(ctx, sizeof(double) * (size_t)N * N);
    if (st) return st;
    double *WR = (double *)ctx->ws;
    dim3 blk(16, 16), grd((N + 15) / 16, (N + 15) / 16);
    grad_wr_kernel<<<grd, blk, 0, ctx->stream>>>(M, U, dsq, WR);
    grad_params_kernel<<<1, kParamThreads, 0, ctx->stream>>>(M, U, r, eta, dsq, WR, dU, dr, deta);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}

int clements_unitary(gbs_ctx *ctx, int M, const double *theta, const double *phi, double *U) {
    const int C = mesh_lanes(M);
    const size_t smem = sizeof(sc4) * kMeshCells + sizeof(double2) * (size_t)M * C;
    GBS_CUDA(ctx, cudaFuncSetAttribute(clements_unitary_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    clements_unitary_kernel<<<kMeshCtas, kMeshThreads, smem, ctx->stream>>>(M, C, theta, phi, U);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}

int clements_grad(gbs_ctx *ctx, int M, const double *theta, const double *phi, const double *U,
                  const double *dU, double *dtheta, double *dphi) {
    const int C = mesh_lanes(M);
    const size_t smem = (sizeof(sc4) + sizeof(double2)) * kMeshCells + 2 * sizeof(double2) * (size_t)M * C;
    GBS_CUDA(ctx, cudaFuncSetAttribute(clements_grad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    clements_grad_kernel<<<kMeshCtas, kMeshThreads, smem, ctx->stream>>>(M, C, theta, phi, U, dU, dtheta, dphi);
    GBS_CUDA(ctx, cudaGetLastError());
    return GBS_OK;
}
