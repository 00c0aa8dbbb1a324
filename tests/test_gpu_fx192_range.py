"""The 192-bit sweep's refusals: matrices that are not positive definite, and pivots below its range."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
OK, NONPOS, NOT_SPD, RANGE = 0, 4, 5, 8


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def prob(ctx, A, precision):
    M = len(A) // 2
    at = np.arange(2 * M).reshape(M, 2).T.ravel()
    O = torch.as_tensor((np.eye(2 * M) - A)[np.ix_(at, at)].copy(), device="cuda")
    pats = np.zeros((1, 2), dtype=np.uint64)
    pats[0, 0] = (1 << M) - 1
    out = ctx.prob(O, torch.zeros(1, dtype=torch.float64, device="cuda"), pats, precision=precision)
    return {k: v.cpu().numpy()[0] for k, v in out.items()}


@pytest.mark.parametrize("n,a", [(1, 0), (2, 0), (2, 1), (9, 0), (9, 8), (11, 0), (11, 1), (14, 0), (14, 1), (14, 3), (14, 7), (14, 13)])
@pytest.mark.parametrize("dx,dp", [(-0.4, -0.4), (0.4, -0.4), (-0.4, 0.4)])
def test_negative_entries(ctx, n, a, dx, dp):
    A = 0.3 * np.eye(2 * n)
    A[2 * a, 2 * a], A[2 * a + 1, 2 * a + 1] = dx, dp
    assert prob(ctx, A, "fx192")["status"] == NOT_SPD


def test_random_matrices(ctx):
    """What the 192-bit sweep answers, the double-double recursion answers too."""
    rng = np.random.default_rng(3)
    ok = 0
    for k in range(150):
        n = int(rng.integers(1, 15))
        A = rng.standard_normal((2 * n, 2 * n)) * 10.0 ** rng.uniform(-2.0, 0.0)
        A = np.clip((A + A.T) / 2, -3.9, 3.9)
        A[np.arange(2 * n), np.arange(2 * n)] = rng.uniform(-0.3 if k % 2 else 0.05, 1.5, 2 * n)
        one, two = prob(ctx, A, "fx192"), prob(ctx, A, "dd")
        if one["status"] == OK:
            ok += 1
            assert two["status"] == OK
            assert abs(one["logP"] - two["logP"]) <= 2 * two["err_bound"] + 1e-13 * (1 + abs(two["logP"]))
    assert ok >= 10


@pytest.mark.parametrize("lo", [1e-3, 2e-4, 1e-5, 1e-7])
@pytest.mark.parametrize("n,at", [(4, 0), (11, 0), (11, 5), (14, 0), (14, 2), (14, 9), (14, 13)])
def test_small_determinants(ctx, n, at, lo):
    """Positive definite with a pivot below the range: out of range, not 'not positive definite'."""
    rng = np.random.default_rng(7)
    Q = np.linalg.qr(rng.standard_normal((2 * n, 2 * n)))[0]
    A = (Q * rng.uniform(0.3, 0.9, 2 * n)) @ Q.T
    s = np.ones(2 * n)
    s[2 * at:2 * at + 2] = lo ** 0.5 / 0.6
    A = A * s[:, None] * s[None, :]
    assert prob(ctx, (A + A.T) / 2, "fx192")["status"] == RANGE


def pair(M, a, b, block):
    A = 0.3 * np.eye(2 * M)
    r = [2 * a, 2 * a + 1, 2 * b, 2 * b + 1]
    A[np.ix_(r, r)] = block
    return A


@pytest.mark.parametrize("n,a,b", [(2, 0, 1), (3, 1, 2), (8, 1, 5), (11, 0, 1), (11, 1, 6), (11, 0, 10), (14, 0, 1), (14, 0, 3),
                                   (14, 1, 13), (14, 2, 4), (14, 5, 6), (14, 12, 13)])
def test_large_rows(ctx, n, a, b):
    """Rows far beyond a positive definite matrix's; the second block's Schur complement is -41000 (2^16 more is positive)."""
    B = np.diag([0.09, 0.05, 5.0, 5.0])
    B[0, 2] = B[2, 0] = 3.9
    B[1, 2] = B[2, 1] = 2.14406
    assert prob(ctx, pair(n, a, b, B), "fx192")["status"] in (NOT_SPD, RANGE)
    B = np.zeros((4, 4))
    B[:2, :2] = [[2.5, (2.5 ** 2 - 0.0040) ** 0.5], [(2.5 ** 2 - 0.0040) ** 0.5, 2.5]]
    B[0, 2] = B[2, 0] = 4.0
    B[1, 2] = B[2, 1] = -4.0
    B[0, 3] = B[3, 0] = 4.0
    B[1, 3] = B[3, 1] = -4.0
    B[2, 2] = B[3, 3] = 5.0
    assert prob(ctx, pair(n, a, b, B), "fx192")["status"] in (NOT_SPD, RANGE)


@pytest.mark.parametrize("n,a", [(2, 0), (9, 3), (12, 0), (14, 1), (14, 9)])
def test_rows_beyond_two(ctx, n, a):
    """Positive definite with a diagonal entry of 4.9, so that a row goes beyond -2: its own value, or out of range."""
    A = 0.3 * np.eye(2 * n)
    b = a + 1 if a + 1 < n else a - 1
    lo, hi = min(a, b), max(a, b)
    A[2 * lo, 2 * lo], A[2 * hi, 2 * hi], A[2 * lo, 2 * hi], A[2 * hi, 2 * lo] = 1.0, 4.9, -2.15, -2.15
    one, two = prob(ctx, A, "fx192"), prob(ctx, A, "dd")
    assert (np.linalg.eigvalsh(A) > 0).all()
    assert one["status"] == RANGE or one["status"] == two["status"] == NONPOS or \
        (one["status"] == two["status"] == OK and abs(one["logP"] - two["logP"]) < 1e-12)
