"""Size bins of the click-number distribution whose terms differ by orders of magnitude: the small sizes keep
their last bits, which the alternating transform brings out."""
from decimal import Decimal, getcontext

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def distribution(M, t, eps):
    """log p(n) for pairs of modes with O = [[eps, t], [t, eps]] on x, [[eps, -t], [-t, eps]] on p: one mode's
    determinant is (1 - eps)^2, a pair's ((1 - eps)^2 - t^2)^2."""
    getcontext().prec = 90
    one, te, ee = Decimal(1), Decimal(t), Decimal(eps)
    d1, d2 = one / (one - ee), one / ((one - ee) ** 2 - te ** 2)
    # sum over the dark subsets: a mode clicks or is dark (weight of the included ones, minus)
    pair = [one, 2 * d1 - 2, d2 - 2 * d1 + one]  # 0, 1 and 2 clicks of the pair, x det(sigma_Q)^(1/2)
    p = [one]
    for _ in range(M // 2):
        q = [Decimal(0)] * (len(p) + 2)
        for i, a in enumerate(p):
            for j, b in enumerate(pair):
                q[i + j] += a * b
        p = q
    return np.array([float(x.ln()) for x in p])


@pytest.mark.parametrize("M", [8, 10, 16, 18])
def test_small_sizes_beside_large_terms(ctx, M):
    t, eps = float(np.sqrt(1 - 1 / 15.0)), 2.0 ** -66  # a pair's second determinant is 15^-2, near 2^-8
    O = np.zeros((2 * M, 2 * M))
    for a in range(0, M, 2):
        for s, off in ((t, 0), (-t, M)):
            O[a + off, a + 1 + off] = O[a + 1 + off, a + off] = s
    O[np.arange(2 * M), np.arange(2 * M)] = eps
    logp, kappa = ctx.click_distribution(torch.as_tensor(O, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda"))
    logp, kappa = logp.cpu().numpy(), kappa.cpu().numpy()
    want = distribution(M, t, eps)
    err = np.abs(logp - want) - 4e-15 * (1 + np.abs(want))
    assert kappa[1] > 1e19
    # one click: bins 0 and 1, whose terms are 1 and a single root; the bins to 2^-104, as double-double ones
    assert err[1] <= 2.0 ** -104 * kappa[1]
    # all: each term's chain of pivots to 2^-102 (a determinant of 15^-2 out of entries near 1, eight times)
    assert (err <= 2.0 ** -100 * kappa).all()
