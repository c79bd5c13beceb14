"""Batches of many LPs, whose control kernels take a warp per LP instead of a block,
against the persistent work-queue form of the same batch: the same sums in the same order
and the same decisions, so the same results bit for bit, over restarts, checks and
different ends.  (Not against smaller batches: a row longer than a tile is summed by
aligned groups of four, so its rounding depends on where the batch puts the LP.)"""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib, long_row_instance

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

FIELDS = ("status", "iterations", "accepted", "rejected", "restarts", "eps_p", "eps_d", "eps_g", "pobj", "dobj",
          "eta", "omega", "used_average")


def kinds():
    return [I.set_cover(m=20, n=50, seed=1), I.knapsack_cover(64, seed=2, per_col=4), I.packing_covering(40, 90, 3, seed=3),
            I.tiny_lp(4), I.mcf(nodes=8, avg_degree=3, commodities=3, seed=5), long_row_instance(seed=6),
            I.knapsack_cover(700, seed=7)]


def solve(batch, tol, limit):
    rs, _ = batch.solve(tol, limit)
    return [tuple(getattr(r, f) for f in FIELDS) for r in rs]


@pytest.mark.parametrize("precision,form", [(0, 1), (1, 1), (1, 3)])
@pytest.mark.parametrize("count", [458, 1001])
def test_many_lps_solve_as_in_the_persistent_form(count, precision, form):
    S = lib()
    few = kinds()
    insts = [few[i % len(few)] for i in range(count)]
    a, b = (S.Batch(insts, S.default_params(precision=precision, batch_launch=f)) for f in (form, 2))
    assert (a.info()[0], b.info()[0]) == (form, 2)
    for tol, limit in ((0.0, 1), (1e-4, 700), (0.0, 130)):  # the third from where the second ended
        ra, rb = solve(a, tol, limit), solve(b, tol, limit)
        for i in range(count):
            assert ra[i] == rb[i], i
    for i in list(range(14)) + list(range(count - 14, count)):
        np.testing.assert_array_equal(a.primal(i), b.primal(i))
        np.testing.assert_array_equal(a.dual(i), b.dual(i))
    a.close()
    b.close()
