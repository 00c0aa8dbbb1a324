"""The exact sweep at the edges of its units: click counts around the register bottom, the breadth-first
levels and the prefix levels of a CTA's loop; and the patterns the double-double mode takes in two passes."""
import numpy as np
import pytest
import torch

import gbs_inputs as g
import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def run(ctx, st, pats, precision):
    out = ctx.prob(st["O"], st["logdet"], pats, precision=precision)
    return {k: v.cpu().numpy() for k, v in out.items()}


def state(ctx, M, lo=0.6, hi=1.2, eta=0.5, seed=5):
    U, r = g.haar_unitary(M, seed), g.squeezing(M, M // 2, lo, hi, seed)
    return ctx.build_state(U, r, eta), oracle.build_state(U, r, eta)


@pytest.mark.parametrize("precision", ["fx", "dd"])
@pytest.mark.parametrize("n", [0, 1, 2, 3, 4, 8, 9, 10, 11, 12, 13, 14, 15, 17])
def test_click_counts(ctx, precision, n):
    st, ref = state(ctx, 24)
    pats = g.gen_patterns(n + 1, 24, n, n, 3)
    want = oracle.prob_exact(ref, pats, dd=True)
    got = run(ctx, st, pats, precision)
    assert (got["status"] == 0).all() and (want["status"] == 0).all()
    # each side within its bound (the double-double one), and the last digits of log P itself
    tol = 2 * (4 * got["kappa"] * (2 * n + 8) * 2.0 ** -106) + 1e-14 * (abs(got["logP"]) + 50)
    same = np.abs(got["logP"] - run(ctx, st, pats, "fx192")["logP"])
    assert (same <= tol).all()
    assert (np.abs(got["logP"] - want["logP"]) <= 1e-10).all()
    # fx sums |terms| in FP32
    assert np.allclose(got["kappa"], want["kappa"], rtol=1e-4 if precision == "fx" else 1e-9)


def test_two_passes(ctx):
    """Patterns on both sides of the kappa that the second pass takes, with empty and invalid ones between."""
    U, r = g.haar_unitary(100, 1), g.squeezing(100, 50, 0.8, 1.4, 1)
    st = ctx.build_state(U, r, 0.3)
    pats = np.concatenate([g.gen_patterns(s, 100, n, n, k) for s, n, k in ((1, 27, 3), (2, 5, 20), (3, 0, 1), (4, 18, 4))])
    pats[10] = ~np.uint64(0)
    got, wide = run(ctx, st, pats, "dd"), run(ctx, st, pats, "fx192")
    assert got["status"][10] == wide["status"][10] == 1
    ok = np.arange(len(pats)) != 10
    assert (got["status"][ok] == 0).all() and (wide["status"][ok] == 0).all()
    assert (got["kappa"][:3] > 1e22).all() and (got["kappa"][ok][3:] < 1e22).all()
    assert (np.abs(got["logP"] - wide["logP"])[ok] <= got["err_bound"][ok] + 1e-14 * (abs(got["logP"][ok]) + 50)).all()
    alone = run(ctx, st, pats[:3], "dd")
    assert np.array_equal(alone["logP"], got["logP"][:3])


def test_not_positive(ctx):
    """A = I - O with an indefinite 2 x 2 block on one mode: refused with it, not without."""
    M = 12
    O = torch.zeros(2 * M, 2 * M, dtype=torch.float64, device="cuda")
    O[7, 7] = 3.0  # mode 7's block is diag(1 - 3, 1) over rows 7 and M + 7
    ld = torch.zeros(1, dtype=torch.float64, device="cuda")
    pats = np.zeros((3, 2), dtype=np.uint64)
    pats[:, 0] = [0b1111, 0b11111111, 0b111111111111 ^ (1 << 7)]
    got = ctx.prob(O, ld, pats, precision="dd")
    st = got["status"].cpu().numpy()
    assert st.tolist() == [4, 5, 4]  # the other sums are zero: vacuum does not click
