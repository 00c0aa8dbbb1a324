"""The tree adjoint's decomposition: patterns around the subtree's seven modes, chunks whose units are
one, a group, and several groups with middle modes between, against the oracle (small patterns) and
against single-pattern calls (one unit a chunk: every prefix mode fixed); and patterns whose sums
cancel beyond what the 110-bit path takes."""
import numpy as np
import pytest

import gbs_inputs as g

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def device(M, seed, eta=0.6):
    return g.haar_unitary(M, seed), g.squeezing(M, M // 2, 0.6, 1.2, seed), eta


def grad(ctx, st, pats, w):
    import torch
    d, lp, status = ctx.grad(st["O"], st["logdet"], pats, torch.as_tensor(w, device="cuda"))
    return d.cpu().numpy(), lp.cpu().numpy(), status.cpu().numpy()


@pytest.mark.parametrize("n", [0, 1, 2, 3, 6, 7, 8, 9])
def test_sizes_against_oracle(ctx, n):
    import oracle
    from oracle import grad as og
    U, r, eta = device(12, 21)
    pats = g.gen_patterns(5, 12, n, n, 3)
    w = np.array([1.0, -0.5, 0.75])
    st = ctx.build_state(U, r, eta)
    d, lp, status = grad(ctx, st, pats, w)
    so = oracle.build_state(U, r, eta)
    ref = og.grad_sigmaQ(so, pats, w)
    assert (status == 0).all()
    # kappa < 1e12 on these: FP64 state and matrix products of the chain
    assert np.abs(d - ref).max() <= 1e-10 * np.abs(ref).max()
    assert np.abs(lp - oracle.prob_exact(so, pats)["logP"]).max() <= 1e-10 * np.abs(lp).max()


# patterns x 2^(n - 7) units against 32 chunks an SM (4864): 1, 2, 16, 64 units a chunk
@pytest.mark.parametrize("n,n_pat", [(9, 8), (13, 101), (14, 500), (14, 1300)])
def test_chunks_against_single_patterns(ctx, n, n_pat):
    U, r, eta = device(20, 22)
    st = ctx.build_state(U, r, eta)
    base = g.gen_patterns(6, 20, n, n, 4)
    idx = np.arange(n_pat) % 4
    w = 0.25 + np.arange(n_pat) % 7
    d, lp, status = grad(ctx, st, base[idx], w)
    ref = 0.0
    for k in range(4):
        dk, lk, sk = grad(ctx, st, base[k:k + 1], np.array([1.0]))
        assert sk[0] == 0
        # 110-bit sums of kappa < 1e17 terms
        assert np.abs(lp[idx == k] - lk[0]).max() <= 1e-12
        ref = ref + w[idx == k].sum() * dk
    assert (status == 0).all()
    assert np.abs(d - ref).max() <= 1e-11 * np.abs(ref).max()


def test_cancelling_sums_take_the_double_double_kernel(ctx):
    # a few squeezed inputs of a local interferometer: kappa of the sum passes 1e24 on some patterns
    M = 32
    st = ctx.build_state(g.clements_unitary(M, *g.clements_phases(M, 23)), g.squeezing(M, 8, 0.6, 1.2, 23), 0.6)
    pats = g.gen_patterns(7, M, 8, 13, 48)
    kap = ctx.prob(st["O"], st["logdet"], pats, precision="fx192")["kappa"].cpu().numpy()
    assert (kap > 1e24).any() and (kap < 1e24).any()
    d, lp, status = grad(ctx, st, pats, np.ones(len(pats)))
    ex = ctx.prob(st["O"], st["logdet"], pats, precision="fx192")
    lx = ex["logP"].cpu().numpy()
    ok = (status == 0) & (kap < 1e27)
    # error of log P in double-double: a few 2^-104 a term
    assert (np.abs(lp - lx)[ok] <= 1e-11 + 1e-30 * kap[ok]).all()
    assert np.isfinite(d).all()
