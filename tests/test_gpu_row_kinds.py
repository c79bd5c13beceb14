"""The FP64 dual step takes one evaluation for a row with one bound or with equal bounds
and a second for a range, and the FP64 clamp compares bit patterns: fixed-step iterates
equal the oracle's (1e-9, the tolerance of the other fixed-step comparisons) with every
kind of row, with columns at zeros of both signs, and with rows split over lanes."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import compare_after, gpu_available

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def _kinds(m, n, per_col, order):
    inst = I.packing_covering(m, n, per_col, seed=m + per_col)
    mid = np.where(np.isfinite(inst.lo), inst.lo, inst.hi)
    w = 0.1 * np.abs(mid) + 0.01
    lo = [mid, mid - w, np.full(m, -np.inf), mid, np.full(m, -np.inf), np.full(m, -0.0)]
    hi = [np.full(m, np.inf), mid + w, mid, mid, np.full(m, np.inf), np.zeros(m)]
    k = np.arange(m) % 6 if order == "mixed" else np.sort(np.arange(m) % 6)
    inst.lo, inst.hi = np.choose(k, lo), np.choose(k, hi)
    inst.is_int[:] = 0
    j = np.arange(n)
    inst.l = np.where(j % 4 == 0, -0.0, np.where(j % 4 == 1, -5.0, np.where(j % 4 == 2, 0.0, -np.inf)))
    inst.u = np.where(j % 4 == 0, 0.0, np.where(j % 4 == 1, -0.0, np.where(j % 4 == 2, np.inf, 5.0)))
    return inst


@pytest.mark.parametrize("m,n,per_col", [(31, 40, 3), (257, 300, 9), (40, 700, 8)])
@pytest.mark.parametrize("order", ["mixed", "sorted"])
def test_fixed_step_iterates_with_every_row_kind(m, n, per_col, order):
    compare_after(_kinds(m, n, per_col, order), 24, replay=False, tol=1e-9, adaptive_step=False, restarts=False)
