"""Rounds, screen and ends of the GPU bound propagation against the oracle's rounds, which
neither screen a row nor queue rounds ahead: equal domains, ignored rows, round and
conflict counts, bit for bit.

- Implication chains that need one round to many batches of rounds, cut at every
  max_rounds around the batches' ends (4, 12, 28, 44 rounds).
- Integer columns with fractional ends, which a row tightens by rounding alone however
  wide its slack.
- Rows whose slack equals their largest span, or differs from it by less and more than the
  screen's relative margin of 1e-6."""
import numpy as np
import pytest

from oracle import fixprop as F
from tests.gpu_common import gpu_available
from tests.test_gpu_propagate import as_instance, handle

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

INF = np.inf


def chain(K, top):
    """x_{k+1} >= x_k + 1 for k < K, x_0 >= 2, x in [0, top]."""
    n = K + 1
    dense = np.zeros((K + 1, n))
    for k in range(K):
        dense[k, k], dense[k, k + 1] = -1.0, 1.0
    dense[K, 0] = 1.0
    return as_instance(dense, np.array([1.0] * K + [2.0]), np.full(K + 1, INF), np.zeros(n), np.full(n, float(top)),
                       np.ones(n))


def compare(g, inst, dl, du, max_rounds=100000):
    got = g.propagate(dl, du, max_rounds)
    want = F.propagate_rounds(inst.rowptr, inst.cols, inst.vals, inst.lo, inst.hi, dl, du, inst.is_int, max_rounds)
    for a, b in zip(got[:3], want[:3]):
        np.testing.assert_array_equal(a, b)
    assert got[3:] == want[3:]
    return want[3]


@pytest.mark.parametrize("K", [0, 1, 2, 3, 4, 10, 26, 27, 42, 43, 60])
def test_chains_of_rounds_and_their_cuts(K):
    inst = chain(K, 300)
    g = handle(inst, aux_general_integers=0)
    rounds = compare(g, inst, inst.l, inst.u)
    assert rounds >= K
    for cut in (1, 2, 3, 4, 5, 11, 12, 13, 27, 28, 29, 44, 45):
        compare(g, inst, inst.l, inst.u, cut)
    g.close()


def test_a_chain_without_room_ends_in_conflicts_or_ignored_rows():
    inst = chain(40, 30)
    g = handle(inst, aux_general_integers=0)
    compare(g, inst, inst.l, inst.u)
    g.close()


@pytest.mark.parametrize("seed", range(6))
def test_fractional_ends_of_integer_columns(seed):
    rng = np.random.default_rng(seed)
    n, k = 60, 40
    l = rng.integers(-3, 1, n) + rng.choice([0.0, 0.3, 0.5], n)
    u = l + rng.integers(2, 6, n) + rng.choice([0.0, 0.2, 0.45], n)
    is_int = (rng.random(n) < 0.7).astype(np.uint8)
    # single-column rows a little outside the fractional ends: slack beyond the span, so
    # only the rounding tightens; and wide rows over several columns
    dense = np.zeros((2 * k, n))
    lo, hi = np.full(2 * k, -INF), np.full(2 * k, INF)
    for i in range(k):
        j = rng.integers(0, n)
        a = float(rng.choice([1.0, 2.0, -1.0]))
        dense[i, j] = a
        ends = sorted((a * (l[j] - 0.1), a * (u[j] + 0.1)))
        lo[i], hi[i] = ends
    for i in range(k, 2 * k):
        cs = rng.choice(n, 4, replace=False)
        dense[i, cs] = rng.integers(1, 4, 4) * rng.choice([-1.0, 1.0], 4)
        hi[i] = np.sum(np.where(dense[i] > 0, dense[i] * l, dense[i] * u)) + rng.uniform(3.0, 25.0)
    base = as_instance(dense, lo, hi, np.floor(l), np.ceil(u), is_int)
    g = handle(base, aux_general_integers=0)
    compare(g, base, l, u)  # the domains given are fractional, the LP's bounds are not
    compare(g, base, np.floor(l), np.ceil(u))  # a later call screens again
    g.close()


@pytest.mark.parametrize("scale", [1.0, 1e6])
@pytest.mark.parametrize("integer", [True, False])
def test_slacks_at_the_screens_margin(integer, scale):
    rng = np.random.default_rng(11)
    n = 80
    l = rng.integers(0, 3, n) * scale
    u = l + rng.integers(1, 5, n) * scale
    rows, lo, hi = [], [], []
    for d in (-0.3, -1e-3, -2e-6, -1e-6, -1e-9, 0.0, 1e-9, 0.9e-6, 1e-6, 1.1e-6, 2.0e-6, 4.0e-6, 1e-5, 1e-3, 0.3):
        for _ in range(6):
            a = np.zeros(n)
            cs = rng.choice(n, rng.integers(1, 5), replace=False)
            a[cs] = rng.integers(1, 6, len(cs)) * rng.choice([-1.0, 1.0], len(cs))
            minf = np.sum(np.where(a > 0, a * l, a * u))
            maxf = np.sum(np.where(a > 0, a * u, a * l))
            span = np.max(np.abs(a) * (u - l))
            up = rng.random() < 0.5
            rows.append(a)
            hi.append(minf + span * (1.0 + d) if up else INF)
            lo.append(-INF if up else maxf - span * (1.0 + d))
    inst = as_instance(np.array(rows), np.array(lo), np.array(hi), l, u, np.full(n, int(integer)))
    g = handle(inst, aux_general_integers=0)
    compare(g, inst, l, u)
    g.close()
