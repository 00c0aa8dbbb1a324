"""Batches without a click: their sector tables are this call's, not an earlier one's."""
import numpy as np
import pytest
import torch

import gbs_inputs as g

pytestmark = pytest.mark.gpu
M = 12


@pytest.fixture()
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


@pytest.mark.parametrize("precision", ["ff", "fp64", "fp32"])
@pytest.mark.parametrize("order", [1, 2, 3, 4])
@pytest.mark.parametrize("pair_from", [80, 3])
def test_only_empty_patterns(ctx, precision, order, pair_from):
    U, r = g.haar_unitary(M, 3), g.squeezing(M, M // 2, 0.8, 1.2, 3)
    st = ctx.build_state(U, r, 0.5)
    if precision != "fp32":
        ctx.set_pair_from(pair_from)
    # leaves other numbers where the tables of the calls below lie
    ctx.prob(st["O"], st["logdet"], g.gen_patterns(1, M, 3, 8, 9), order=order, precision=precision)
    want = -0.5 * float(st["logdet"])
    for k in (1, 5):
        out = ctx.prob(st["O"], st["logdet"], np.zeros((k, 2), dtype=np.uint64), order=order, precision=precision)
        assert (out["status"] == 0).all()
        assert np.abs(out["logP"].cpu().numpy() - want).max() <= 1e-12
    # beside a pattern with clicks (of which every one is the pair kernel's, for the low limit)
    pats = g.gen_patterns(2, M, 4, 4, 3)
    pats[1] = 0
    out = ctx.prob(st["O"], st["logdet"], pats, order=order, precision=precision)
    alone = ctx.prob(st["O"], st["logdet"], pats[[0, 2]], order=order, precision=precision)
    assert abs(float(out["logP"][1]) - want) <= 1e-12
    assert torch.equal(out["logP"][[0, 2]], alone["logP"])


def test_gradient_of_empty_patterns(ctx):
    U, r = g.haar_unitary(M, 3), g.squeezing(M, M // 2, 0.8, 1.2, 3)
    st = ctx.build_state(U, r, 0.5)
    w = torch.ones(3, dtype=torch.float64, device="cuda")
    ctx.grad_approx(st["O"], st["logdet"], g.gen_patterns(1, M, 3, 8, 3), w, 2)
    d, lp, status = ctx.grad_approx(st["O"], st["logdet"], np.zeros((3, 2), dtype=np.uint64), w, 2)
    e, le, _ = ctx.grad(st["O"], st["logdet"], np.zeros((3, 2), dtype=np.uint64), w)
    assert (status == 0).all() and torch.allclose(lp, le, atol=1e-12, rtol=0)
    assert torch.allclose(d, e, rtol=1e-12, atol=1e-13)
