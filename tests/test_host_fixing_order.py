"""Fix-and-propagate's fixing order on points whose distances to their rounding are mostly
equal (zero, or one of a few values), and on an assignment problem, where the propagation
fixes most columns before their turn: the oracle's point, domains, fixed columns in order
and ignored rows."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.test_host_fixprop import INSTANCES, assert_equals_oracle, harness, run_harness  # noqa: F401


def assignment(N):
    n = N * N
    q = np.arange(n)
    return I._from_coo("assignment", 2 * N, n, np.concatenate([q // N, N + q % N]), np.concatenate([q, q]),
                       np.ones(2 * n), np.ones(n), lo=np.ones(2 * N), hi=np.ones(2 * N), l=np.zeros(n), u=np.ones(n),
                       is_int=np.ones(n, dtype=np.uint8))


CASES = {"assignment": lambda: assignment(17),
         **{k: INSTANCES[k] for k in ("setcover", "packcover_gen_int", "mcf_small", "long_rows", "no_rows")}}


@pytest.mark.parametrize("name", list(CASES))
@pytest.mark.parametrize("distances", [(0.0,), (0.25,), (0.0, 0.001, 0.01, 0.5), (1e-9, 2e-9, -1e-9, 0.4)])
def test_equal_distances_keep_index_order(harness, tmp_path, name, distances):  # noqa: F811
    inst = CASES[name]()
    rng = np.random.default_rng(29)
    l = np.where(np.isfinite(inst.l), inst.l, -3.0)
    u = np.where(np.isfinite(inst.u), np.minimum(inst.u, l + 9.0), l + 9.0)
    xbar = np.floor(rng.uniform(l, u + 1.0)) + rng.choice(distances, inst.n)
    assert_equals_oracle(inst, xbar, run_harness(harness, inst, xbar, str(tmp_path / name)))
