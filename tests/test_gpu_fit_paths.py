"""The sector fits' three paths (a warp on many sectors, clusters for the slow ones, supports smaller than
the order) give each pattern the same bits in any batch: alone (a sector a warp) and among others."""
import numpy as np
import pytest

import gbs_inputs as g

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


@pytest.mark.parametrize("order", [1, 2, 3, 4])
def test_batch_independent_fits(ctx, order):
    c = g.CONFIGS["m50_approx"]
    st = ctx.build_state(c.unitary(), c.squeezing(), c.eta)
    # 0..6 clicks (supports around the order), and the workload's sizes
    pats = np.concatenate([g.gen_patterns(70 + n, c.M, n, n, 3) for n in range(7)] + [c.patterns()[:60]])
    many = ctx.prob(st["O"], st["logdet"], np.concatenate([pats] * 3), order=order, precision="fp32")
    many = {k: v.cpu().numpy().reshape(3, -1) for k, v in many.items()}
    for k in ("logP", "status"):
        assert (many[k] == many[k][:1]).all()
    for i in list(range(3, 21)) + [21, 40, 60, 80]:
        one = ctx.prob(st["O"], st["logdet"], pats[i:i + 1], order=order, precision="fp32")
        assert one["logP"].cpu().numpy()[0] == many["logP"][0, i], i
        assert one["status"].cpu().numpy()[0] == many["status"][0, i]


def test_curves_follow_the_batch_kernels(ctx):
    # the curve kernel fits a warp a sector; its all-clicked column sums to the batch's estimate
    c = g.CONFIGS["m50_approx"]
    st = ctx.build_state(c.unitary(), c.squeezing(), c.eta)
    p = g.gen_patterns(9, c.M, 12, 12, 1)
    lp = ctx.prob(st["O"], st["logdet"], p, order=3, precision="ff")["logP"].cpu().numpy()[0]
    curves, lc, _ = ctx.approx_sector_curves(st["O"], st["logdet"], p, order=3, K=1000)
    assert lc.cpu().numpy()[0] == lp
    assert abs(np.log(curves[:, 12].sum().item()) - lp) < 1e-9
