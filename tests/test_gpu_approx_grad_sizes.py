"""Gradient of the approximation at orders 1 and 2, where the diagonal blocks' groups go to 16 lanes and the
off-diagonal blocks to 32: click counts around these, against the oracle."""
import numpy as np
import pytest
import torch

import gbs_inputs as g
import oracle
from oracle import grad as og

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


@pytest.mark.parametrize("order", [1, 2])
@pytest.mark.parametrize("n", [1, 2, 7, 8, 9, 15, 16, 17, 20])
def test_low_orders(ctx, order, n):
    U, r, eta = g.haar_unitary(22, 9), g.squeezing(22, 11, 0.5, 1.0, 9), 0.5
    pats = g.gen_patterns(n, 22, n, n, 2)
    w = np.array([1.0, -0.7])
    st = ctx.build_state(U, r, eta)
    dsq, logP, status = ctx.grad_approx(st["O"], st["logdet"], pats, torch.as_tensor(w, device="cuda"), order)
    ref, ref_lp = og.grad_sigmaQ_approx(oracle.build_state(U, r, eta), pats, w, order)
    assert np.isin(status.cpu().numpy(), (0, 7)).all()
    # as for the other sizes: the forwards agree to 1e-9, the gradients to 1e-8 of their largest entry
    assert np.abs(logP.cpu().numpy() - ref_lp).max() < 1e-9
    assert np.abs(dsq.cpu().numpy() - ref).max() < 1e-8 * np.abs(ref).max()
