"""Entries of O that are not finite: the patterns that touch them are refused, the others keep their values."""
import numpy as np
import pytest
import torch

import gbs_inputs as g

pytestmark = pytest.mark.gpu
M = 14


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf, -1e300])
@pytest.mark.parametrize("rows", ["x", "p", "xp", "cross"])
@pytest.mark.parametrize("mode", [0, 5, 13])
def test_gradient_refuses(ctx, bad, rows, mode):
    U, r = g.haar_unitary(M, 3), g.squeezing(M, M // 2, 0.6, 1.2, 3)
    st = ctx.build_state(U, r, 0.6)
    O = st["O"].clone()
    for i in {"x": [mode], "p": [mode + M], "xp": [mode, mode + M], "cross": []}[rows]:
        O[i, i] = bad
    if rows == "cross":
        O[mode, mode + M] = O[mode + M, mode] = bad
    every = (1 << M) - 1
    pats = np.zeros((4, 2), dtype=np.uint64)
    pats[:, 0] = [1 << mode, every, every ^ (1 << mode), (every ^ (1 << mode)) & 0x1E7]
    w = torch.ones(4, dtype=torch.float64, device="cuda")
    _, lp, status = ctx.grad(O, st["logdet"], pats, w)
    _, ref, good = ctx.grad(st["O"], st["logdet"], pats, w)
    lp, status, ref = lp.cpu().numpy(), status.cpu().numpy(), ref.cpu().numpy()
    assert (good.cpu().numpy() == 0).all()
    if bad == -1e300 and rows in ("x", "p"):  # finite and, with the other entry positive, positive definite: as the exact sum
        want = ctx.prob(O, st["logdet"], pats[:2], precision="dd")["status"].cpu().numpy()
        assert (status[:2] == want).all()
    else:
        assert status[:2].tolist() == [5, 5]
        assert np.isnan(lp[:2]).all()
    assert (status[2:] == 0).all() and np.array_equal(lp[2:], ref[2:])
