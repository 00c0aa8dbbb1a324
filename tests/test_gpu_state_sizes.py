"""State build at the edges of its tiling: mode counts around the 8-row tile and the 8-CTA cluster,
the largest one, and a U whose storage is aligned to 8 bytes only."""
import numpy as np
import pytest

import gbs_inputs as g

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def reference(U, r, eta):
    M = len(r)
    R = np.block([[U.real, -U.imag], [U.imag, U.real]])
    s = eta * np.concatenate((np.exp(-2 * r), np.exp(2 * r))) / 2 + (1 - eta) / 2
    return (R * s) @ R.T, np.eye(2 * M) - (R / (s + 0.5)) @ R.T, np.log1p(eta * (2 - eta) * np.sinh(r) ** 2).sum()


@pytest.mark.parametrize("M", [1, 2, 3, 4, 5, 8, 9, 12, 31, 32, 33, 64, 65, 127, 128])
def test_state_against_numpy(ctx, M):
    import torch
    U, r = g.haar_unitary(M, 11), g.squeezing(M, max(1, M // 2), 0.3, 1.3, 11)
    sig, O, ld = reference(U, r, 0.7)
    flat = torch.zeros(2 * M * M + 1, dtype=torch.float64, device="cuda")
    flat[1:] = torch.as_tensor(U.view(np.float64).reshape(-1), device="cuda")
    Ud = flat[1:].view(M, 2 * M)  # data pointer at 8 modulo 16
    rd = torch.as_tensor(r, device="cuda")
    st = ctx.build_state(U, r, 0.7, want_sigma=True)
    O2, ld2 = torch.empty_like(st["O"]), torch.empty_like(st["logdet"])
    status = torch.ones(1, dtype=torch.int32, device="cuda")
    ctx.build_state_into(Ud, rd, 0.7, O2, ld2, status)
    # sums of 2M products of entries below 1 with weights below 4 e^{2.6}
    tol = 1e-15 * 2 * M * 14
    assert np.abs(st["sigma"].cpu().numpy() - sig).max() <= tol
    assert np.abs(st["O"].cpu().numpy() - O).max() <= tol
    assert abs(st["logdet"].item() - ld) <= 1e-14 * max(1, M)
    assert torch.equal(O2, st["O"]) and torch.equal(ld2, st["logdet"]) and status.item() == 0


@pytest.mark.parametrize("M,i,j", [(1, 0, 0), (8, 7, 0), (9, 8, 8), (33, 0, 32)])
def test_not_unitary_is_refused(ctx, M, i, j):
    from paper_2106_01445_gb300._lib import GbsError
    U, r = g.haar_unitary(M, 3), g.squeezing(M, M, 0.3, 0.9, 3)
    U[i, j] += 1e-6j * U[i, j] / abs(U[i, j]) + 1e-6
    with pytest.raises(GbsError):
        ctx.build_state(U, r, 0.7)
