"""The create-time choice of the per-attempt kernels' forms in the handles that launch
them: launch modes other than the chunk graphs on LPs that the chunk graphs run resident,
and LPs that stay in L2 but do not fit the resident form.

Sizes are used by no other test of this process: a choice is kept per matrix shape, and
only the first handle of a shape times the forms."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def handle(inst, precision, **kw):
    S = lib()
    return S.LP.from_instance(inst, S.default_params(precision=precision, aux_general_integers=0, **kw))


def check_choice(lp, precision):
    """Each kernel's form is the fastest of its timings unless the rule's is within 3%."""
    forms, rule, ms = lp.kernel_form()
    assert rule == 4  # the 32-row plain form
    timed = (4, 2, 5) if precision else (4, 2)
    for side in (0, 1):
        t = {f: ms[2 * q + side] for q, f in enumerate(timed)}
        assert all(v > 0 for v in t.values())
        best = min(t, key=t.get)
        assert forms[side] == (best if t[best] < 0.97 * t[rule] else rule)
    return forms


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("use_graph", [0, 2, 3])
def test_modes_that_launch_attempts_keep_the_choice(use_graph, precision):
    inst = I.packing_covering(1500 + 10 * use_graph + precision, 3100, 4, seed=31)
    lp = handle(inst, precision, use_graph=use_graph)
    assert lp.resident() == (0, 0)
    check_choice(lp, precision)
    lp.close()


@pytest.mark.parametrize("precision", [0, 1])
def test_persistent_mode_that_runs_as_chunk_graphs_is_resident(precision):
    """use_graph = 3 with infeasibility detection runs as 1: the same attempts, the same
    results."""
    inst = I.packing_covering(1557, 3201, 4, seed=32)
    a, b = (handle(inst, precision, use_graph=g, infeasibility_checks=1) for g in (3, 1))
    assert a.resident() == b.resident() and a.resident()[0] != 0
    ra, rb = a.pdhg_solve(0.0, 200), b.pdhg_solve(0.0, 200)
    assert (ra.iterations, ra.rejected, ra.rel_kkt) == (rb.iterations, rb.rejected, rb.rel_kkt)
    np.testing.assert_array_equal(a.primal(), b.primal())
    np.testing.assert_array_equal(a.dual(), b.dual())
    a.close()
    b.close()


# past the resident form's limit, within the L2 rule's
PAST = {0: (60_000, 140_001, 11), 1: (100_000, 200_001, 12)}


@pytest.mark.parametrize("precision", [0, 1])
def test_l2_sized_lps_past_the_resident_form_are_tuned(precision):
    """The wide tiles are built after the other arrays here: the choice is the timings',
    a solve is that of a handle with the form forced (whose wide tiles come with the
    arrays), and a later handle of the shape keeps the choice."""
    inst = I.packing_covering(*PAST[precision], seed=33)
    a = handle(inst, precision)
    assert a.resident() == (0, 0)
    forms = check_choice(a, precision)
    b = handle(inst, precision, prefetch=forms[0], dual_form=forms[1])
    assert b.kernel_form()[0] == forms
    ra, rb = a.pdhg_solve(0.0, 130), b.pdhg_solve(0.0, 130)
    assert (ra.iterations, ra.rejected, ra.restarts, ra.eta) == (rb.iterations, rb.rejected, rb.restarts, rb.eta)
    np.testing.assert_array_equal(a.primal(), b.primal())
    np.testing.assert_array_equal(a.dual(), b.dual())
    b.close()
    c = handle(inst, precision)
    assert c.kernel_form()[0] == forms and not np.any(c.kernel_form()[2])
    a.close()  # the first handle's late tiles go; the later one's stay
    c.pdhg_solve(0.0, 10)
    d = handle(inst, precision, prefetch=forms[0], dual_form=forms[1])
    d.pdhg_solve(0.0, 10)
    np.testing.assert_array_equal(c.primal(), d.primal())
    c.close()
    d.close()
