"""Which LPs the resident form takes in which scope: the plan of every LP that the other
tests compare with the launched form, so that none of them compares that form with itself,
and the edges of the cluster scope (1, 4 and 8 or 16 blocks, up to 232 tiles a side in FP32
and 64 in FP64) with solves equal to the launched form's, bit for bit."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib
from tests.test_gpu_resident import CASES, _same, _solve

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

# scope in FP64 and FP32: 1 a cluster, 2 the grid
SCOPES = {"one_tile": (1, 1), "three_tiles": (1, 1), "setcover": (1, 1), "cluster_top": (2, 2), "past_cluster": (2, 2),
          "fp64_cluster": (2, 1), "fp64_past_cluster": (2, 1), "grid_full": (2, 2), "grid_two_per_warp": (2, 2),
          "open_bounds": (1, 1), "standard_form": (1, 1), "mcf": (2, 2), "long_rows": (1, 1), "long_rows_grid": (2, 2)}


def handle(inst, precision, **kw):
    S = lib()
    return S.LP.from_instance(inst, S.default_params(precision=precision, aux_general_integers=0, autotune=0, **kw))


@pytest.mark.parametrize("name", list(CASES))
def test_compared_lps_run_resident(name):
    got = []
    for precision in (0, 1):
        lp = handle(CASES[name](), precision)
        got.append(lp.resident()[0])
        lp.close()
    assert tuple(got) == SCOPES[name]


def circulant(tiles, seed):
    """16 entries in every row and column, so 16 of them to a tile of 256 entries."""
    m = 16 * tiles
    rng = np.random.default_rng(seed)
    steps = np.sort(rng.choice(m, 16, replace=False)) if m > 16 else np.arange(16)
    cols = np.sort((np.arange(m)[:, None] + steps) % m, axis=1)
    va = rng.uniform(0.5, 2.0, 16 * m)
    r = (va.reshape(m, 16) * rng.uniform(0.0, 2.0, m)[cols]).sum(axis=1)
    return I.Instance("circulant", m, m, (np.arange(m + 1) * 16).astype(np.int64), cols.ravel().astype(np.int32), va,
                      rng.normal(size=m), r - rng.uniform(0, 2, m), np.where(rng.random(m) < 0.5, np.inf, r + 1.0),
                      np.zeros(m), np.full(m, 3.0), np.zeros(m, dtype=np.uint8))


EDGES = [(0, 1, 1), (0, 2, 1), (0, 3, 4), (0, 8, 4), (0, 9, 16), (0, 63, 16), (0, 64, 16), (0, 65, None),
         (1, 2, 1), (1, 3, 4), (1, 8, 4), (1, 9, 8), (1, 231, 8), (1, 232, 8), (1, 233, None)]


@pytest.mark.parametrize("precision,tiles,blocks", EDGES)
def test_edges_of_the_cluster_scope(precision, tiles, blocks):
    inst = circulant(tiles, 3 * tiles + precision)
    a, b = handle(inst, precision), handle(inst, precision, use_graph=0)
    assert a.resident() == ((1, blocks) if blocks else (2, a.resident()[1])) and b.resident() == (0, 0)
    for k in (1, 65, 200):
        a.reset_state()
        b.reset_state()
        _same(_solve(a, k), _solve(b, k))
    _same(_solve(a, 130), _solve(b, 130))
    a.close()
    b.close()
