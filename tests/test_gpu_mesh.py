"""The mesh kernels at the edges of their split (eight CTAs of 1..16 columns, chunks of whole layers of
at most 512 cells) and the parameter chain, against numpy and the oracle."""
import numpy as np
import pytest

import gbs_inputs as g

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


@pytest.mark.parametrize("M", [2, 3, 5, 8, 9, 16, 17, 33, 46, 64, 65, 127, 128])
def test_mesh_and_chain(ctx, M):
    import torch
    from oracle import grad as og
    th, ph = g.clements_phases(M, 40 + M)
    r, eta = g.squeezing(M, max(1, M // 2), 0.4, 1.1, M), 0.7
    d = lambda a: torch.as_tensor(np.ascontiguousarray(a), device="cuda")  # noqa: E731
    U = g.clements_unitary(M, th, ph)
    Ud = ctx.clements_unitary(d(th), d(ph), M)
    # M layers of rotations
    assert np.abs(Ud.cpu().numpy().view(np.complex128) - U).max() <= 1e-15 * 8 * M
    rng = np.random.default_rng(M)
    dsq = rng.standard_normal((2 * M, 2 * M))
    dsq = dsq + dsq.T
    dU, dr, deta = ctx.grad_params(Ud, d(r), eta, d(dsq))
    rU, rr, re = og.chain_params(U, r, eta, dsq)
    # sums of 2M x 2M terms of size ~ e^{2.2}
    tol = 1e-13 * M
    scale = np.abs(rr).max()
    assert np.abs(dr.cpu().numpy() - rr).max() <= tol * scale
    assert abs(deta.item() - re) <= tol * max(scale, abs(re))
    dth, dph = ctx.clements_grad(d(th), d(ph), Ud, dU)
    rth, rph = og.chain_clements(M, th, ph, rU)
    assert np.abs(dth.cpu().numpy() - rth).max() <= tol * np.abs(rth).max()
    assert np.abs(dph.cpu().numpy() - rph).max() <= tol * max(np.abs(rph).max(), 1.0)
