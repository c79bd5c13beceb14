"""Solves of several handles at the same time, from a thread each: a handle whose attempts
run resident on every SM launches them while others are solving, chunk by chunk, and its
results are those of a solve alone, bit for bit, whatever mix of the two it took."""
import threading

import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def outcome(lp, k):
    lp.reset_state()
    r = lp.pdhg_solve(0.0, k)
    x, y, eta, omega = lp.get_state()
    return x, y, np.array([eta, omega, r.iterations, r.rejected, r.restarts, r.eps_p, r.eps_d, r.eps_g])


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("hessian", [False, True])
def test_results_do_not_depend_on_other_solves(precision, hessian):
    S = lib()
    insts = [I.knapsack_cover(5000, 41), I.packing_covering(12_000, 40_001, 9, seed=42), I.set_cover(),
             I.packing_covering(30_000, 70_003, 10, seed=43)]
    mk = lambda i: S.LP.from_instance(i, S.default_params(precision=precision, aux_general_integers=0, autotune=0))  # noqa: E731
    lps = [mk(i) for i in insts]
    assert [lp.resident()[0] for lp in lps] == [2, 2, 1, 2]
    if hessian:  # drops the graphs that hold the LP's kernels
        for lp, i in zip(lps, insts):
            lp.pdhg_solve(0.0, 64)
            lp.set_qp_objective(i.c, np.full(i.n, 0.5), 0.0)
    budgets = [[700, 64, 1, 130, 2000], [300, 900, 65], [3000, 1000], [640, 200, 64]]
    alone = [[outcome(lp, k) for k in b] for lp, b in zip(lps, budgets)]
    together = [[] for _ in lps]

    def work(q):
        for _ in range(3):
            together[q].append([outcome(lps[q], k) for k in budgets[q]])

    threads = [threading.Thread(target=work, args=(q,)) for q in range(len(lps))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    for q in range(len(lps)):
        assert len(together[q]) == 3
        for rep in together[q]:
            for got, want in zip(rep, alone[q]):
                for a, b in zip(got, want):
                    np.testing.assert_array_equal(a, b)
    for lp in lps:
        lp.close()


def test_a_batch_and_a_fanout_beside_a_resident_solve():
    S = lib()
    inst = I.packing_covering(12_000, 40_001, 9, seed=42)
    lp = S.LP.from_instance(inst, S.default_params(precision=1, aux_general_integers=0, autotune=0))
    base = I.fanout_base(4000, 9000, 6)
    host = S.LP.from_instance(base, S.default_params(precision=1, aux_general_integers=0))
    fan = S.Fanout(host, I.fanout_targets(base, np.zeros(base.n), 8))
    batch = S.Batch([I.knapsack_cover(300, s) for s in range(6)], S.default_params(precision=1))
    want = outcome(lp, 1500)
    fan.solve(0.0, 200)
    batch.solve(0.0, 200)
    xf, xb = fan.primal(3), batch.primal(3)
    got = []

    def others():
        for _ in range(4):
            fan.reset_state()
            fan.solve(0.0, 200)
            batch.reset_state()
            batch.solve(0.0, 200)

    t = threading.Thread(target=others)
    t.start()
    for _ in range(6):
        got.append(outcome(lp, 1500))
    t.join()
    for g in got:
        for a, b in zip(g, want):
            np.testing.assert_array_equal(a, b)
    np.testing.assert_array_equal(fan.primal(3), xf)
    np.testing.assert_array_equal(batch.primal(3), xb)
    for h in (fan, batch, lp, host):
        h.close()
