"""An attempt whose step-size sums overflow ends a solve SCYLLA_NUMERICAL at the last
accepted point: the resident form of the attempts returns and keeps the point that the
launched form does.

The LP is unbounded: free rows, free columns and a cost so large that the squared step
overflows after some accepted attempts of the first chunk (no dual moves, so every
attempt is accepted and the step size grows by 1 + (k + 1)^-0.6 each time)."""
import numpy as np
import pytest

from tests.gpu_common import gpu_available, lib
from tests.test_gpu_resident import CASES, _same

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

# scope 1: one cluster, 2: one block per SM
SCOPES = {"one_tile": 1, "setcover": 1, "past_cluster": 2, "grid_full": 2, "grid_two_per_warp": 2}


def unbounded(name, precision):
    inst = CASES[name]()
    inst.lo, inst.hi = np.full(inst.m, -np.inf), np.full(inst.m, np.inf)
    inst.l, inst.u = np.full(inst.n, -np.inf), np.full(inst.n, np.inf)
    inst.is_int = np.zeros(inst.n, dtype=np.uint8)
    inst.c = np.random.default_rng(3).uniform(0.5, 1.0, inst.n) * ((1e150, 1e15)[precision])
    return inst


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(SCOPES))
def test_resident_form_keeps_the_last_accepted_point(name, precision):
    S = lib()
    inst = unbounded(name, precision)
    a, b = (S.LP.from_instance(inst, S.default_params(precision=precision, aux_general_integers=0, autotune=0,
                                                      use_graph=g)) for g in (1, 0))
    assert a.resident()[0] == SCOPES[name] and b.resident() == (0, 0)
    for first in (True, False):  # from the cold start, then from the point the first solve returned
        ra, rb = a.pdhg_solve(0.0, 64), b.pdhg_solve(0.0, 64)
        assert ra.status == rb.status == S.NUMERICAL
        assert ra.iterations == rb.iterations < 64 and (ra.accepted, ra.rejected) == (rb.accepted, rb.rejected)
        if first:
            assert ra.accepted > 1
        assert np.all(np.isfinite(b.primal())) and np.any(b.primal() != 0.0)
        _same([a.primal(), a.dual()] + [np.asarray(v) for v in a.get_state()],
              [b.primal(), b.dual()] + [np.asarray(v) for v in b.get_state()])
    a.close()
    b.close()
