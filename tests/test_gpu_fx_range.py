"""Matrices that are no state's, and states at the edge of the fixed-point range: the limb form's bounds hold for
positive definite A = I - O only, so what leaves them has to be seen, wherever its modes lie in the
recursion (prefix, sub-unit tree, levels, register bottom)."""
import numpy as np
import pytest
import torch

import gbs_inputs as g

pytestmark = pytest.mark.gpu
OK, NONPOS, NOT_SPD, RANGE = 0, 4, 5, 8


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


def prob(ctx, A, M, precision, modes=None):
    """A in mode order (x, p of mode 0, x, p of mode 1, ...); one pattern of these modes (all)."""
    at = np.arange(2 * M).reshape(M, 2).T.ravel()
    O = torch.as_tensor((np.eye(2 * M) - A)[np.ix_(at, at)].copy(), device="cuda")
    pats = np.zeros((1, 2), dtype=np.uint64)
    pats[0, 0] = sum(1 << m for m in (range(M) if modes is None else modes))
    out = ctx.prob(O, torch.zeros(1, dtype=torch.float64, device="cuda"), pats, precision=precision)
    return {k: v.cpu().numpy()[0] for k, v in out.items()}


def embed(M, a, b, block):
    """Modes a and b from the 4 x 4 block, the others 0.3 times the identity."""
    A = 0.3 * np.eye(2 * M)
    r = [2 * a, 2 * a + 1, 2 * b, 2 * b + 1]
    A[np.ix_(r, r)] = block
    return A


def indefinite():
    """Every |O| <= 4 and the first pivot positive; the Schur complement of x1 is 5 - 3.9^2 / 0.09 -
    2.14406^2 / 0.05 = -255.94, which an entry that is kept modulo 256 turns into 0.06."""
    B = np.diag([0.09, 0.05, 5.0, 5.0])
    B[0, 2] = B[2, 0] = 3.9
    B[1, 2] = B[2, 1] = 2.14406
    return B


# modes of an n-click pattern: n - 12 (n > 12) first ones fix the unit, three are the tree's, seven the levels', two the bottom
@pytest.mark.parametrize("n,a,b", [(2, 0, 1), (3, 0, 1), (3, 0, 2), (3, 1, 2), (8, 1, 5), (8, 2, 7), (11, 0, 1), (11, 1, 6),
                                   (11, 0, 10), (14, 0, 1), (14, 0, 3), (14, 1, 7), (14, 1, 13), (14, 2, 4), (14, 5, 6),
                                   (14, 12, 13)])
def test_indefinite_is_refused(ctx, n, a, b):
    A = embed(n, a, b, indefinite())
    assert prob(ctx, A, n, "dd")["status"] == NOT_SPD
    assert prob(ctx, A, n, "fx")["status"] in (NOT_SPD, RANGE)
    assert prob(ctx, A, n, "auto")["status"] == NOT_SPD


def test_random_indefinite(ctx):
    """Whatever the default precision answers for a matrix with |O| <= 4, the double-double recursion answers too."""
    rng = np.random.default_rng(1)
    ok = 0
    for k in range(120):
        n = int(rng.integers(2, 15))
        d = rng.uniform(0.02, 0.6, 2 * n) ** rng.integers(1, 3)
        A = rng.standard_normal((2 * n, 2 * n)) * 10.0 ** rng.uniform(-2.0, 0.0)
        A = np.clip((A + A.T) / 2, -3.9, 3.9)
        A[np.arange(2 * n), np.arange(2 * n)] = d
        one, two = prob(ctx, A, n, "auto"), prob(ctx, A, n, "dd")
        if one["status"] != two["status"]:
            assert one["status"] == NOT_SPD and two["status"] in (OK, NONPOS)  # a negative definite block in the levels
        elif one["status"] == OK:
            ok += 1
            assert abs(one["logP"] - two["logP"]) <= 2 * (one["err_bound"] + two["err_bound"]) + 1e-13 * (1 + abs(two["logP"]))
    assert ok >= 10


@pytest.mark.parametrize("n,a", [(14, 0), (14, 1), (14, 3), (13, 0), (11, 1), (14, 13), (2, 1)])
def test_negative_definite_block(ctx, n, a):
    """A block of positive determinant is accepted in the prefix, the tree and as the last mode."""
    A = 0.3 * np.eye(2 * n)
    A[2 * a, 2 * a] = A[2 * a + 1, 2 * a + 1] = -0.4
    one, two = prob(ctx, A, n, "auto"), prob(ctx, A, n, "dd")
    assert two["status"] == OK and one["status"] == OK
    # a product of one-mode factors: 0.3^-1 - 1 each, and 0.4^-1 - 1
    assert abs(two["logP"] - ((n - 1) * np.log(1 / 0.3 - 1) + np.log(1 / 0.4 - 1))) <= 1e-13 * n
    assert abs(one["logP"] - two["logP"]) <= 1e-13 * n


@pytest.mark.parametrize("lo", [1e-3, 2e-4, 1e-5, 1e-7])
@pytest.mark.parametrize("n,at", [(4, 0), (11, 0), (11, 5), (14, 0), (14, 2), (14, 9), (14, 13)])
def test_small_determinants_go_to_double_double(ctx, n, at, lo):
    """A positive definite matrix with a pivot below the range, coupled to the rest: never 'not positive definite'."""
    rng = np.random.default_rng(7)
    Q = np.linalg.qr(rng.standard_normal((2 * n, 2 * n)))[0]
    A = (Q * rng.uniform(0.3, 0.9, 2 * n)) @ Q.T
    s = np.ones(2 * n)
    s[2 * at:2 * at + 2] = lo ** 0.5 / 0.6
    A = A * s[:, None] * s[None, :]
    A = (A + A.T) / 2
    one, two = prob(ctx, A, n, "auto"), prob(ctx, A, n, "dd")
    assert prob(ctx, A, n, "fx")["status"] == RANGE
    assert two["status"] == OK and one["status"] == OK
    assert abs(one["logP"] - two["logP"]) <= 2 * (one["err_bound"] + two["err_bound"]) + 1e-13 * (1 + abs(two["logP"]))


def test_entries_beyond_four(ctx):
    """Positive definite with diagonal entries up to 90: out of range, not refused as indefinite."""
    n = 13
    A = 0.3 * np.eye(2 * n)
    for m in (0, 2, 6, 12):
        A[2 * m, 2 * m], A[2 * m + 1, 2 * m + 1] = 90.0, 0.2
        A[2 * m, 3], A[3, 2 * m] = 0.5, 0.5
    A[3, 3] = 1.0
    assert (np.linalg.eigvalsh(A) > 0).all()
    one, two = prob(ctx, A, n, "auto"), prob(ctx, A, n, "dd")
    assert prob(ctx, A, n, "fx")["status"] == RANGE
    assert two["status"] == one["status"] and two["status"] in (OK, NONPOS)
