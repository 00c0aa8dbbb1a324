"""Performance cases: what a user of this library has it compute, through its Python binding.

The sizes are those of the repository's own workloads (`gbs_inputs.CONFIGS`: devices of 8, 24, 32,
50 and 100 modes and their click ranges) and of its tests; `draw` spreads them over the ranges
between.  A case is one device (mode count, squeezed inputs, squeezing range, transmission), a batch
of uniformly drawn click patterns, and one call on them:

* ``state``    the state build alone (a sweep over squeezing or loss settings);
* ``exact``    log P of every pattern by the signed subset sum;
* ``approx``   log P by the order-1..4 moment approximation;
* ``grad``     exact log P of a batch and its gradient with respect to squeezing, transmission and
               the mesh phases (a step of a likelihood fit), through autograd;
* ``agrad``    the same with the approximation;
* ``clicks``   the whole device's click-number distribution.
"""
import functools
import math

import numpy as np
import torch

import gbs_inputs as g
from paper_2106_01445_gb300.api import Context, LogProbClements, LogProbClementsApprox, patterns_tensor


def _case(name, kind, M, K, r_lo, r_hi, eta, n_lo=0, n_hi=0, n_pat=0, order=0, precision="auto"):
    c = dict(kind=kind, M=M, K=K, r_lo=r_lo, r_hi=r_hi, eta=eta, n_lo=n_lo, n_hi=n_hi, n_pat=n_pat, order=order,
             precision=precision)
    return dict(name=name, **c) if name else c


M24 = (24, 12, 0.6, 1.2, 0.5)
M32 = (32, 16, 0.6, 1.2, 0.6)
M50 = (50, 25, 0.8, 1.4, 0.4)
M100 = (100, 50, 1.1, 1.6, 0.3)


def listed():
    return [
        # the smallest call: one device's covariance and O, where launch and host time count
        _case("state_m50", "state", *M50),
        # every outcome of a small device (all 256 patterns of 8 modes): small sums, many patterns
        _case("exact_m8_all", "exact", 8, 8, 0.8, 0.8, 1.0, 0, 8, 256),
        # one large outcome by itself: how well a single pattern fills the GPU
        _case("exact_m24_one", "exact", *M24, 20, 20, 1),
        # the benchmark batch: 1024 outcomes of uneven size
        _case("exact_m24_batch", "exact", *M24, 12, 20, 1024),
        # large outcomes of a large device: sums that cancel beyond 128 bits, which the automatic
        # precision sweeps again in 192 bits
        _case("exact_m100_deep", "exact", *M100, 22, 24, 6),
        # double-double arithmetic, which states outside the fixed-point range fall back to
        _case("exact_m24_dd", "exact", *M24, 10, 18, 181, 0, "dd"),
        # the approximation at its cheapest useful order, where plan, transform and fit count
        _case("approx_m50_o2", "approx", *M50, 10, 40, 256, 2),
        # the approximation at its highest order: the group minors
        _case("approx_m50_o4", "approx", *M50, 10, 40, 96, 4),
        # large outcomes, some of them beyond what one block's shared memory holds
        _case("approx_m100_o2", "approx", *M100, 40, 90, 64, 2),
        # one step of a likelihood fit: forward and backward through the mesh
        _case("grad_m32", "grad", *M32, 8, 16, 512),
        # the same with the approximation
        _case("agrad_m32_o2", "agrad", *M32, 8, 16, 128, 2),
        # the click-number distribution of a whole device (all 2^M subsets)
        _case("clicks_m24", "clicks", *M24),
    ]


# ---- drawn cases -------------------------------------------------------------------------------

def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# the most subsets (exact sums), tree nodes (gradients) or weighted minors (approximations) that a
# drawn case may ask for: below the largest listed cases of the kind
_MOST = {"exact": 2.0e8, "dd": 2.0e7, "fx192": 4.0e7, "grad": 1.0e7, "clicks": 1.6e7}


def draw(rng):
    kind = rng.choice(("state", "exact", "exact", "exact", "approx", "approx", "grad", "agrad", "clicks"))
    eta = round(rng.uniform(0.3, 1.0), 3)
    r_lo = round(rng.uniform(0.4, 1.0), 3)
    r_hi = round(r_lo + rng.uniform(0.0, 0.4), 3)
    if kind == "state":
        M = _log_int(rng, 4, 100)
        return _case(None, kind, M, max(1, M // 2), r_lo, r_hi, eta)
    if kind == "clicks":
        M = rng.randint(8, 23)
        return _case(None, kind, M, max(1, M // 2), r_lo, r_hi, eta)
    if kind == "exact":
        M = _log_int(rng, 8, 100)
        precision = rng.choice(("auto", "auto", "auto", "fx", "dd", "fx192"))
        n_hi = rng.randint(4, min(M, 21))
        n_lo = rng.randint(max(0, n_hi - 8), n_hi)
        n_pat = _log_int(rng, 1, 2048)
        most = _MOST.get(precision, _MOST["exact"])
        while n_hi > 4 and 2.0 ** n_hi > most:
            n_hi -= 1
        n_lo = min(n_lo, n_hi)
        n_pat = max(1, min(n_pat, int(most / _mean(n_lo, n_hi, lambda n: 2.0 ** n))))
        return _case(None, kind, M, max(1, M // 2), r_lo, r_hi, eta, n_lo, n_hi, n_pat, 0, precision)
    if kind == "grad":
        M = rng.randint(8, 40)
        n_hi = rng.randint(5, min(M, 17))
        n_lo = rng.randint(max(1, n_hi - 8), n_hi)
        n_pat = max(1, min(_log_int(rng, 1, 512), int(_MOST["grad"] / _mean(n_lo, n_hi, lambda n: 2.0 ** n))))
        return _case(None, kind, M, max(1, M // 2), r_lo, r_hi, eta, n_lo, n_hi, n_pat)
    if kind == "agrad":
        M = rng.randint(12, 40)
        n_hi = rng.randint(6, min(M, 18))
        n_lo = rng.randint(max(4, n_hi - 8), n_hi)
        return _case(None, kind, M, max(1, M // 2), r_lo, r_hi, eta, n_lo, n_hi, _log_int(rng, 1, 96), 2)
    order = rng.choice((2, 2, 3, 4))
    M = _log_int(rng, 20, 100)
    n_hi = rng.randint(8, min(M, {2: 90, 3: 48, 4: 40}[order]))
    n_lo = max(6, n_hi - rng.randint(0, 30))
    n_pat = max(1, min(_log_int(rng, 1, 256), int(2.5e5 / n_hi ** 2) if order == 2 else int(4e3 / n_hi)))
    # squeezing of the repository's own devices: the photon-number sectors of an almost vacuum state
    # underflow before they reach 90 clicks
    return _case(None, kind, M, max(1, M // 2), max(r_lo, 0.8), max(r_hi, 1.2), min(eta, 0.5), n_lo, n_hi, n_pat, order)


# ---- inputs ------------------------------------------------------------------------------------

@functools.lru_cache(maxsize=None)
def _context():
    """The one context that a program keeps for all its calls."""
    return Context(0)


def _inputs(case, seed):
    """Host inputs from the seed: mesh phases or interferometer, squeezing, patterns, weights."""
    s = 1000003 * int(seed) + 17
    M = case["M"]
    x = dict(r=g.squeezing(M, case["K"], case["r_lo"], case["r_hi"], s), eta=case["eta"])
    if case["kind"] in ("grad", "agrad"):
        x["theta"], x["phi"] = g.clements_phases(M, s)
        x["w"] = 0.5 + g.uniform01(g.philox_words(s, 7, np.arange(case["n_pat"]), 1)[:, 0])
    else:
        x["U"] = g.haar_unitary(M, s)
    if case["n_pat"]:
        if case["kind"] == "exact" and case["n_pat"] == 1 << M:
            x["pats"] = g.all_patterns(M)
        else:
            x["pats"] = g.gen_patterns(s, M, case["n_lo"], case["n_hi"], case["n_pat"])
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    ctx = _context()
    dev = ctx.device
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device=dev)  # noqa: E731
    s = dict(case=case, ctx=ctx, eta=x["eta"])
    if "pats" in x:
        s["pats"] = patterns_tensor(x["pats"], dev)
    if case["kind"] in ("grad", "agrad"):
        s["par"] = [d(x["r"]).requires_grad_(True), torch.tensor(x["eta"], dtype=torch.float64, requires_grad=True),
                    d(x["theta"]).requires_grad_(True), d(x["phi"]).requires_grad_(True)]
        s["w"] = d(x["w"])
    elif case["kind"] == "state":
        s["U"], s["r"] = d(x["U"]), d(x["r"])
    else:
        st = ctx.build_state(d(x["U"]), d(x["r"]), x["eta"])
        s["O"], s["logdet"] = st["O"], st["logdet"]
    return s


def run(s):
    c, ctx = s["case"], s["ctx"]
    kind = c["kind"]
    if kind == "state":
        st = ctx.build_state(s["U"], s["r"], s["eta"], want_sigma=True, check=False)
        return {k: st[k] for k in ("sigma", "O", "logdet", "status")}
    if kind in ("exact", "approx"):
        return ctx.prob(s["O"], s["logdet"], s["pats"], order=c["order"], precision=c["precision"])
    if kind == "clicks":
        logp, kappa = ctx.click_distribution(s["O"], s["logdet"])
        return dict(logp=logp, kappa=kappa)
    if kind == "grad":
        logp = LogProbClements.apply(*s["par"], s["pats"], ctx)
    else:
        logp = LogProbClementsApprox.apply(*s["par"], s["pats"], ctx, c["order"])
    dr, deta, dth, dph = torch.autograd.grad((s["w"] * logp).sum(), s["par"])
    return dict(logP=logp.detach(), dr=dr, deta=deta, dtheta=dth, dphi=dph)


# ---- the work that a call cannot do without ------------------------------------------------------

def _mean(lo, hi, f):
    return sum(f(n) for n in range(lo, hi + 1)) / (hi - lo + 1)


def _subset_flops(n):
    """2 x 2 pivots and rank-2 updates of the include/exclude recursion, in operations of the sum's
    own precision: 44 a subset (see bench.py)."""
    return 44.0 * 2.0 ** n


def work(case):
    M, P = case["M"], case["n_pat"]
    state = 8.0 * (2 * M) ** 2
    lo, hi = case["n_lo"], case["n_hi"]
    kind = case["kind"]
    if kind == "state":
        return dict(bytes=16.0 * M * M + 8 * M + 2 * state + 12, flops=2.0 * 4 * (2 * M) ** 2 * M)
    if kind == "clicks":
        return dict(bytes=state + 16 * (M + 1) + 8, flops=_subset_flops(M))
    if kind == "exact":
        return dict(bytes=state + P * (16 + 28) + 8, flops=P * _mean(lo, hi, _subset_flops))
    if kind == "grad":
        # the recursion forward for log P, and forward and back for the gradient
        return dict(bytes=P * 32 + 8 * (2 * M * M) * 2, flops=P * _mean(lo, hi, lambda n: 4 * _subset_flops(n)))
    j = case["order"]

    def minors(n):
        # n contour points (half of the sectors around 2 n photons), at each the inverse of a complex
        # symmetric 2n x 2n matrix and about 34 complex products a group of up to j detectors
        return n * 8.0 * ((2 * n) ** 3 / 2 + sum(34.0 * math.comb(n, w) for w in range(1, j + 1)))

    back = 3.0 if kind == "agrad" else 1.0
    return dict(bytes=state + P * (16 + 28) + 8, flops=back * P * _mean(lo, hi, minors))


# ---- what the results are, in 64 bits ----------------------------------------------------------
# The signed sums cancel by ten to twenty orders of magnitude, so the reference carries every
# number as an unevaluated sum of two 64-bit ones (Dekker's products, Knuth's sums).

class _Two:
    """Pairs (h, l) of FP64 tensors, value h + l."""

    def __init__(self, h, l=None):
        self.h, self.l = h, torch.zeros_like(h) if l is None else l

    def __getitem__(self, k):
        return _Two(self.h[k], self.l[k])

    def __neg__(self):
        return _Two(-self.h, -self.l)

    @staticmethod
    def _sum(a, b):
        s = a + b
        t = s - a
        return s, (a - (s - t)) + (b - t)

    @staticmethod
    def _quick(a, b):
        s = a + b
        return _Two(s, b - (s - a))

    def __add__(self, o):
        s, e = _Two._sum(self.h, o.h)
        t, f = _Two._sum(self.l, o.l)
        v = _Two._quick(s, e + t)
        return _Two._quick(v.h, v.l + f)

    def __sub__(self, o):
        return self + (-o)

    def __mul__(self, o):
        split = lambda a: (lambda c: (c - (c - a), a - (c - (c - a))))(134217729.0 * a)  # noqa: E731
        p = self.h * o.h
        ah, al = split(self.h)
        bh, bl = split(o.h)
        e = ((ah * bh - p) + ah * bl + al * bh) + al * bl
        return _Two._quick(p, e + (self.h * o.l + self.l * o.h))

    def rsqrt(self):
        y = _Two(torch.rsqrt(self.h))
        one, half = _Two(torch.ones_like(self.h)), _Two(torch.full_like(self.h, 0.5))
        for _ in range(2):
            y = y + y * (one - self * y * y) * half
        return y

    @staticmethod
    def cat(a, b, dim):
        return _Two(torch.cat((a.h, b.h), dim), torch.cat((a.l, b.l), dim))

    def total(self, dim):
        """The sum over a dimension, halving it."""
        v = self
        while v.h.shape[dim] > 1:
            n = v.h.shape[dim]
            a, b = _Two(v.h.narrow(dim, 0, n // 2), v.l.narrow(dim, 0, n // 2)), \
                _Two(v.h.narrow(dim, n - n // 2, n // 2), v.l.narrow(dim, n - n // 2, n // 2))
            w = a + b
            if n & 1:
                w = _Two.cat(w, _Two(v.h.narrow(dim, n // 2, 1), v.l.narrow(dim, n // 2, 1)), dim)
            v = w
        return _Two(v.h.squeeze(dim), v.l.squeeze(dim))


def _state64(x):
    """sigma, A = sigma_Q^-1, O and log det sigma_Q, in numpy."""
    U, r, eta = x["U"], x["r"], x["eta"]
    M = len(r)
    R = np.block([[U.real, -U.imag], [U.imag, U.real]])
    sq = np.concatenate((np.exp(-2 * r), np.exp(2 * r))) / 2
    sigma = eta * (R * sq) @ R.T + (1 - eta) * np.eye(2 * M) / 2
    Q = sigma + np.eye(2 * M) / 2
    return sigma, np.eye(2 * M) - np.linalg.inv(Q), np.linalg.slogdet(Q)[1]


def _start64(O, modes):
    """A = I - O on the modes of each pattern (B, n), as B x 2n x 2n pairs, rows (x, p) by mode."""
    M, n = O.shape[0] // 2, modes.shape[1]
    at = torch.stack((modes, modes + M), 2).reshape(len(modes), 2 * n)
    h = O[at[:, :, None], at[:, None, :]]
    s, e = _Two._sum(torch.eye(2 * n, dtype=h.dtype, device=h.device).expand_as(h), -h)
    return _Two(s, e)


def _terms64(A, n, binned):
    """All subset terms det(A_Z)^(-1/2) of B patterns of n modes: the include/exclude tree, one
    mode a step.  Returns their signed sum and the sum of their sizes (B), or, binned, their sums by
    subset size (n + 1, B)."""
    B = A.h.shape[0]
    A = A[:, None]
    tau = _Two(torch.ones(B, 1, dtype=torch.float64, device=A.h.device))
    size = torch.zeros(1, dtype=torch.int64, device=A.h.device)
    for k in range(n):
        p = [A[:, :, i, j] for i, j in ((0, 0), (0, 1), (1, 1))]
        det = p[0] * p[2] - p[1] * p[1]
        rs = det.rsqrt()
        inc = tau * rs
        rest = A[:, :, 2:, 2:]
        if k < n - 1:
            inv = rs * rs
            q = [(inv * v)[:, :, None] for v in (p[2], -p[1], p[0])]
            b0, b1 = A[:, :, 0, 2:], A[:, :, 1, 2:]
            w0, w1 = q[0] * b0 + q[1] * b1, q[1] * b0 + q[2] * b1
            upd = rest - w0[:, :, :, None] * b0[:, :, None, :] - w1[:, :, :, None] * b1[:, :, None, :]
            A = _Two.cat(rest, upd, 1)
        tau = _Two.cat(tau, inc, 1)
        size = torch.cat((size, size + 1))
    if binned:
        out = []
        for z in range(n + 1):
            k = torch.nonzero(size == z)[:, 0]
            out.append(tau[:, k].total(1))
        return out
    sign = (1 - 2 * ((n - size) & 1)).to(torch.float64)[None]
    return _Two(tau.h * sign, tau.l * sign).total(1), tau.h.sum(1)


def exact(case, seed):
    kind = case["kind"]
    # the approximation's fit in 64 bits over every group minor, and gradients of sums that cancel
    # beyond 64 bits (a matrix inverse a subset, in pairs), take minutes in plain torch
    if kind in ("approx", "grad", "agrad"):
        return None
    x = _inputs(case, seed)
    sigma, O, logdet = _state64(x)
    if kind == "state":
        return dict(sigma=sigma, O=O, logdet=np.array([logdet]), status=None)
    # the sums from the same 64-bit O that the call is given
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    Od = torch.as_tensor(O, device=dev)
    M = case["M"]
    if kind == "clicks":
        E = _terms64(_start64(Od, torch.arange(M, device=dev)[None]), M, True)
        logp, kap = [], []
        for n in range(M + 1):
            c = [(-1.0) ** (n - z) * math.comb(M - z, n - z) for z in range(n + 1)]
            t = _Two(torch.stack([E[z].h for z in range(n + 1)]), torch.stack([E[z].l for z in range(n + 1)])) * \
                _Two(torch.tensor(c, dtype=torch.float64, device=dev)[:, None])
            s = t.total(0)
            logp.append(math.log(float(s.h)) - 0.5 * logdet)
            kap.append(float(t.h.abs().sum()) / float(s.h))
        return dict(logp=np.array(logp), kappa=np.array(kap))
    modes = [g.pattern_modes(p) for p in x["pats"]]
    logP, kappa = np.zeros(len(modes)), np.ones(len(modes))
    for n in sorted({len(m) for m in modes}):
        at = [i for i, m in enumerate(modes) if len(m) == n]
        if n == 0:
            logP[at] = -0.5 * logdet
            continue
        step = max(1, (1 << 21) >> n)
        for k in range(0, len(at), step):
            sel = at[k:k + step]
            T, a = _terms64(_start64(Od, torch.tensor([modes[i] for i in sel], device=dev)), n, False)
            logP[sel] = (torch.log(T.h) - 0.5 * logdet).cpu().numpy()
            kappa[sel] = (a / T.h.abs()).cpu().numpy()
    return dict(logP=logP, kappa=kappa, err_bound=None, status=None)

