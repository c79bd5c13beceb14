"""The resident form of the per-attempt kernels (attempts between two checks in one
launch) against the launched form: the same arithmetic in the same order, so identical
points, step sizes, decisions and errors, at the edges of its deals (one tile, a tile
per warp, the cluster's and the grid's limits, several tiles per warp) and on rows
longer than a tile, empty rows, no rows and quadratic objectives."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I

pytestmark = pytest.mark.gpu


def _long_rows(m, n, seed):
    """A few rows of 300 to 900 entries among short and empty ones."""
    rng = np.random.default_rng(seed)
    counts = rng.integers(0, 6, size=m)
    counts[:: max(1, m // 7)] = rng.integers(300, 900, size=len(counts[:: max(1, m // 7)]))
    counts = np.minimum(counts, n)
    cols = [np.sort(rng.choice(n, size=int(k), replace=False)) for k in counts]
    rowptr = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    ci = np.concatenate(cols).astype(np.int32)
    va = rng.uniform(0.5, 2.0, size=len(ci)) * rng.choice([-1.0, 1.0], size=len(ci))
    x0 = rng.uniform(0.0, 4.0, n)
    r = np.array([va[rowptr[i]:rowptr[i + 1]] @ x0[ci[rowptr[i]:rowptr[i + 1]]] for i in range(m)])
    return I.Instance("long", m, n, rowptr, ci, va, rng.normal(size=n), r - rng.uniform(0, 1, m),
                      r + rng.uniform(0, 1, m), np.zeros(n), np.full(n, 5.0), np.zeros(n, dtype=np.uint8))


CASES = {
    "one_tile": lambda: I.packing_covering(4, 9, 2, seed=1),
    "three_tiles": lambda: I.packing_covering(40, 90, 3, seed=2),
    "setcover": lambda: I.set_cover(),
    "cluster_top": lambda: I.knapsack_cover(3712, 3),     # 232 tiles of the transpose
    "past_cluster": lambda: I.knapsack_cover(3728, 4),
    "fp64_cluster": lambda: I.knapsack_cover(1008, 5),    # 63 tiles
    "fp64_past_cluster": lambda: I.knapsack_cover(1100, 5),
    "grid_full": lambda: I.packing_covering(12_000, 40_001, 9, seed=6),
    "grid_two_per_warp": lambda: I.packing_covering(30_000, 70_003, 10, seed=7),
    "open_bounds": lambda: I.open_bounds_lp(900, 1500, 6, 3),
    "standard_form": lambda: I.standard_form_lp(400, 900, 6, 1),
    "mcf": lambda: I.mcf(nodes=60, commodities=40),
    "long_rows": lambda: _long_rows(700, 1200, 8),
    "long_rows_grid": lambda: _long_rows(20_000, 9000, 9),
}


def _solve(lp, k):
    r = lp.pdhg_solve(0.0, k)
    return [lp.primal(), lp.dual()] + [np.array([getattr(r, f) for f in
            ("iterations", "rejected", "restarts", "eta", "omega", "eps_p", "eps_d", "eps_g", "pobj", "dobj",
             "used_average")])]


def _pair(inst, precision, **kw):
    from paper_2307_03466_gb300 import scylla as S
    mk = lambda g: S.LP.from_instance(inst, S.default_params(precision=precision, aux_general_integers=0,  # noqa: E731
                                                             autotune=0, use_graph=g, trace_capacity=400, **kw))
    return mk(1), mk(0)


def _same(a, b):
    for u, v in zip(a, b):
        np.testing.assert_array_equal(u, v)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", list(CASES))
def test_resident_form_is_the_launched_one(name, precision):
    a, b = _pair(CASES[name](), precision)
    assert b.resident() == (0, 0)
    for k in (1, 3, 64, 65, 300):  # cold starts, then a warm one
        a.reset_state()
        b.reset_state()
        _same(_solve(a, k), _solve(b, k))
    _same(a.trace(), b.trace())
    _same(_solve(a, 100), _solve(b, 100))
    a.close()
    b.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_resident_scopes_are_taken(precision):
    """The plan takes the cluster, the grid and (beyond them) the launched form."""
    from paper_2307_03466_gb300 import scylla as S
    got = []
    for inst in (I.set_cover(), I.packing_covering(30_000, 70_000, 10), I.packing_covering(100_000, 200_000, 12)):
        lp = S.LP.from_instance(inst, S.default_params(precision=precision, aux_general_integers=0, autotune=0))
        got.append(lp.resident()[0])
        lp.close()
    assert got == [1, 2, 0]


def test_resident_form_without_rows():
    from paper_2307_03466_gb300 import scylla as S
    n = 9000
    rng = np.random.default_rng(1)
    c = rng.normal(size=n)
    lp = S.LP(np.zeros(1, dtype=np.int64), np.zeros(0, dtype=np.int32), np.zeros(0), c, np.zeros(0), np.zeros(0),
              np.zeros(n), np.ones(n), np.zeros(n, dtype=np.uint8), 0, n)
    assert lp.pdhg_solve(1e-9, 1000).status == S.CONVERGED
    np.testing.assert_allclose(lp.primal(), (c < 0).astype(float), atol=1e-8)
    lp.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", ["setcover", "grid_full"])
def test_resident_form_with_a_hessian(name, precision):
    inst = CASES[name]()
    a, b = _pair(inst, precision)
    q = np.random.default_rng(4).uniform(0.0, 2.0, inst.n)
    for lp in (a, b):
        lp.pdhg_solve(0.0, 10)
        lp.set_qp_objective(inst.c, q, 1.0)
    _same(_solve(a, 150), _solve(b, 150))
    a.close()
    b.close()


def test_resident_barrier_timeout_is_reported():
    """The grid scope's barrier waits are bounded by device_wait_limit_s."""
    from paper_2307_03466_gb300 import scylla as S
    lp = S.LP.from_instance(CASES["grid_full"](), S.default_params(aux_general_integers=0, device_wait_limit_s=1e-9))
    assert lp.resident()[0] == 2
    for _ in range(2):
        with pytest.raises(S.ScyllaError) as e:
            lp.pdhg_solve(1e-9, 5000)
        assert e.value.code == S.ERR_TIMEOUT
    lp.close()
