"""Patterns whose sum cancels beyond what the 110-bit arithmetic is used for: the double-double pass of GBS_DD and of
the gradient, tried after the 110-bit one or, where a guess of kappa suffices, instead of it."""
import numpy as np
import pytest
import torch

import gbs_inputs as g

pytestmark = pytest.mark.gpu
REDO = 1e24


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def np_of(out):
    return {k: v.cpu().numpy() for k, v in out.items()}


def in_dd(ctx, st, pats):
    """All units of the batch in double-double (the slices' arithmetic)."""
    part, flag = ctx.prob_partial(st["O"], pats, 0, 1, "dd")
    return np_of(ctx.prob_combine(st["logdet"], pats, part[None], flag[None], "dd"))


def weak(ctx, M, lo, hi, eta, seed):
    return ctx.build_state(g.haar_unitary(M, seed), g.squeezing(M, M // 2, lo, hi, seed), eta)


@pytest.mark.parametrize("M,lo,hi,eta,n1,n2", [(100, 0.4, 0.6, 0.3, 12, 18), (40, 0.3, 0.5, 0.4, 13, 16), (50, 0.5, 0.8, 0.5, 13, 19),
                                               (24, 0.6, 1.2, 0.5, 13, 18)])
def test_double_double_where_it_cancels(ctx, M, lo, hi, eta, n1, n2):
    st = weak(ctx, M, lo, hi, eta, 5)
    pats = g.gen_patterns(9, M, n1, n2, 40)
    pats[7] = 0
    got, dd, wide = np_of(ctx.prob(st["O"], st["logdet"], pats, precision="dd")), in_dd(ctx, st, pats), \
        np_of(ctx.prob(st["O"], st["logdet"], pats, precision="fx192"))
    assert np.array_equal(got["status"], dd["status"]) and np.array_equal(got["status"], wide["status"])
    ok = got["status"] == 0
    assert ok.all()
    over = wide["kappa"] > 1.01 * REDO
    # the same units, sums and digits
    assert np.array_equal(got["logP"][over], dd["logP"][over]) and np.array_equal(got["kappa"][over], dd["kappa"][over])
    # below, either arithmetic: 2^-111 kappa covers double-double
    tol = 2.0 ** -111 * wide["kappa"] + 2e-14 * (1 + np.abs(wide["logP"]))
    assert (np.abs(got["logP"] - wide["logP"]) <= tol).all()
    assert over.any() == (M in (100, 40))


def test_no_second_price(ctx):
    """A batch of cancelling patterns takes about double-double's time, not both passes' (1.47 of it)."""
    st = weak(ctx, 100, 0.4, 0.6, 0.3, 5)
    pats = torch.as_tensor(g.gen_patterns(9, 100, 18, 18, 40).view(np.int64), device="cuda")
    assert (ctx.prob(st["O"], st["logdet"], pats, precision="fx192")["kappa"] > 1e24).all()

    def ms(f):
        best = []
        for _ in range(8):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            f()
            b.record()
            torch.cuda.synchronize()
            best.append(a.elapsed_time(b))
        return sorted(best)[2]
    assert ms(lambda: ctx.prob(st["O"], st["logdet"], pats, precision="dd")) <= 1.25 * ms(lambda: ctx.prob_partial(st["O"], pats, 0, 1, "dd"))


def single(ctx, st, pat):
    d, lp, status = ctx.grad(st["O"], st["logdet"], pat[None], torch.ones(1, dtype=torch.float64, device="cuda"))
    return d.cpu().numpy(), float(lp[0]), int(status[0])


@pytest.mark.parametrize("M,K,n1,n2,seed", [(32, 8, 8, 13, 23), (40, 20, 13, 15, 3)])
def test_gradient_against_differences(ctx, M, K, n1, n2, seed):
    """dL/dsigma_Q of single patterns, kappa 1e21 to 1e27, against central differences of the 192-bit log P along
    random directions of A on the pattern's modes."""
    local = seed != 3
    U = g.clements_unitary(M, *g.clements_phases(M, seed)) if local else g.haar_unitary(M, seed)
    st = ctx.build_state(U, g.squeezing(M, K, *((0.6, 1.2) if local else (0.3, 0.4)), seed), 0.6 if local else 0.4)
    pats = g.gen_patterns(7, M, n1, n2, 64)
    kap = np_of(ctx.prob(st["O"], st["logdet"], pats, precision="fx192"))["kappa"]
    below, above = np.nonzero((kap > 1e21) & (kap < REDO))[0][:3], np.nonzero((kap > REDO) & (kap < 1e27))[0][:5]
    assert len(above) > 0
    O = st["O"].cpu().numpy()
    A, S = np.eye(2 * M) - O, np.linalg.inv(np.eye(2 * M) - O)
    rng = np.random.default_rng(1)
    for p in list(below) + list(above):
        d, lp, status = single(ctx, st, pats[p])
        assert status == 0
        H = -S @ (d + 0.5 * A) @ S  # (1 / T) dT/dA, on the pattern's rows
        rows = np.array([m + x for m in g.pattern_modes(pats[p]) for x in (0, M)])
        off = np.ones((2 * M, 2 * M), bool)
        off[np.ix_(rows, rows)] = False
        assert np.abs(H[off]).max() <= 1e-7 * np.abs(H).max()
        for _ in range(2):
            D = rng.standard_normal((len(rows), len(rows)))
            D = (D + D.T) / 2
            size = np.linalg.norm(H) * np.linalg.norm(D)
            h = 1e-4 / size
            lps, Os = [], []
            for s in (h, -h):
                X = O.copy()
                X[np.ix_(rows, rows)] -= s * D
                Os.append(X)
                out = ctx.prob(torch.as_tensor(X, device="cuda"), st["logdet"], pats[p:p + 1], precision="fx192")
                assert int(out["status"][0]) == 0
                lps.append(float(out["logP"][0]))
            want = ((Os[1] - Os[0]) * H).sum()  # the step as rounded
            # of the step 1e-4 times the gradient's size: differences 1e-8 (third order) and 1e-10 (rounding of log P),
            # double-double 3e-34 kappa, below 3e-7
            assert abs((lps[0] - lps[1]) - want) <= 2e-6 * 2e-4, (kap[p], lps[0] - lps[1], want)


def test_largest_chunks(ctx):
    """256 units a chunk, four middle modes (a batch of 6.5e5 units), against two units a chunk."""
    M, n, k = 24, 20, 80
    st = ctx.build_state(g.haar_unitary(M, 22), g.squeezing(M, M // 2, 0.6, 1.2, 22), 0.6)
    base = g.gen_patterns(6, M, n, n, 2)
    w = torch.as_tensor(0.25 + np.arange(k) % 7, device="cuda")
    d, lp, status = ctx.grad(st["O"], st["logdet"], base[np.arange(k) % 2], w)
    assert (status == 0).all()
    ref = 0
    for i in range(2):
        di, li, si = ctx.grad(st["O"], st["logdet"], base[i:i + 1], torch.ones(1, dtype=torch.float64, device="cuda"))
        assert int(si[0]) == 0 and float((lp[i::2] - li[0]).abs().max()) <= 1e-12
        ref = ref + w[i::2].sum() * di
    assert float((d - ref).abs().max()) <= 1e-11 * float(ref.abs().max())
