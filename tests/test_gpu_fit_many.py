"""Sector fits with many trial points: thousands of them (each CTA takes one by itself) and a few (a cluster each), and
supports below the order beside larger ones, give each pattern the same bits in any batch."""
import numpy as np
import pytest

import gbs_inputs as g

pytestmark = pytest.mark.gpu
M = 8


@pytest.fixture(scope="module")
def ctx(cuda_ok):
    from paper_2106_01445_gb300.api import Context
    return Context(0)


@pytest.mark.parametrize("lo,hi,order,copies", [(5, 6, 4, 30), (2, 3, 2, 40), (1, 4, 4, 20)])
def test_many_slow_fits(ctx, lo, hi, order, copies):
    st = ctx.build_state(g.haar_unitary(M, 3), g.squeezing(M, M, 0.8, 1.2, 3), 1.0)
    base = g.gen_patterns(4, M, lo, hi, 10)
    few = ctx.prob(st["O"], st["logdet"], base, order=order, precision="fp64")
    many = ctx.prob(st["O"], st["logdet"], np.concatenate([base] * copies), order=order, precision="fp64")
    for k in ("logP", "status"):
        assert np.array_equal(many[k].cpu().numpy().reshape(copies, -1), np.tile(few[k].cpu().numpy(), (copies, 1)), equal_nan=k == "logP")
