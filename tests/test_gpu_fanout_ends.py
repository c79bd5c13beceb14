"""A fan-out whose last objectives end together inside a chunk, on a non-finite step, with
objective 0 finished long before: the attempt is counted, the finished objective keeps its
point, and the solve repeats bit for bit.

The LP has no costs and free rows, so target 0 (every column at its lower bound, where the
solve starts) is optimal at once, and the others (at the upper bounds, far away) take
growing steps until the squared step overflows, all at the same attempt."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("K", [2, 33, 64])
def test_objectives_that_end_together_on_an_overflow(K, precision):
    S = lib()
    inst = I.packing_covering(40, 90, 3, seed=5)
    inst.c, inst.is_int = np.zeros(inst.n), np.ones(inst.n, dtype=np.uint8)
    inst.lo, inst.hi = np.full(inst.m, -np.inf), np.full(inst.m, np.inf)
    inst.l, inst.u = np.zeros(inst.n), np.full(inst.n, 2.0 ** (70 if precision else 1000))
    lp = S.LP.from_instance(inst, S.default_params(precision=precision, aux_general_integers=0, step_growth_exp=0.02))
    targets = np.repeat(inst.u[:, None], K, axis=1)
    targets[:, 0] = 0.0
    f = S.Fanout(lp, targets)
    runs = []
    for _ in range(8):
        f.reset_state()
        rs, _ = f.solve(1e-9, 2000)
        assert rs[0].status == S.CONVERGED and rs[0].iterations == 0
        assert len({(r.status, r.iterations) for r in rs[1:]}) == 1 and rs[1].status == S.NUMERICAL
        assert 1 < rs[1].iterations < 2000
        np.testing.assert_array_equal(f.primal(0), np.zeros(inst.n))
        runs.append((rs[1].iterations, np.stack([f.primal(k) for k in range(K)]), np.stack([f.dual(k) for k in range(K)])))
        assert np.all(runs[-1][1][1:] == runs[-1][1][1])
    for r in runs[1:]:
        assert r[0] == runs[0][0]
        np.testing.assert_array_equal(r[1], runs[0][1])
        np.testing.assert_array_equal(r[2], runs[0][2])
    f.close()
    lp.close()
