"""Reads of a point on both sides of the size up to which the unscaling kernel writes
pinned host memory (4096 entries): the values are the state's, whatever the destination,
from a handle, a batch and a fan-out, and a reset handle repeats its solve."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

SIZES = [64, 4095, 4096, 4097]
KW = dict(precision=0, aux_general_integers=0, n_check=8)


def _inst(n):
    return I.packing_covering(n, n, 2, seed=n)


def _shifted(n):
    """Its start point is the lower bounds: l / C * C, two roundings."""
    inst = _inst(n)
    inst.is_int[:] = 0
    inst.l = 1.0 + np.arange(n)
    inst.u = inst.l + 10.0
    return inst


@pytest.mark.parametrize("n", SIZES)
def test_reads_equal_the_device_copy(n):
    import torch
    S = lib()
    lp = S.LP.from_instance(_inst(n), S.default_params(**KW))
    lp.reset_state()
    r0 = lp.pdhg_solve(0.0, 24)
    dev = torch.empty(lp.n, dtype=torch.float64, device="cuda")
    lp.primal_device(dev.data_ptr())
    want = dev.cpu().numpy()
    assert np.array_equal(lp.primal(), want)
    pinned = torch.empty(lp.n, dtype=torch.float64, pin_memory=True).numpy()
    lp.primal(out=pinned)
    assert np.array_equal(pinned, want)
    y = lp.dual()
    assert y.any()
    lp.reset_state()
    assert not lp.dual().any()
    r1 = lp.pdhg_solve(0.0, 24)
    assert np.array_equal(lp.primal(), want) and np.array_equal(lp.dual(), y)
    assert (r0.eta, r0.omega, r0.iterations) == (r1.eta, r1.omega, r1.iterations)
    lp.close()


def test_batch_reads():
    S = lib()
    insts = [_shifted(n) for n in SIZES]
    B = S.Batch(insts, S.default_params(**KW))
    B.reset_state()
    for k, inst in enumerate(insts):
        np.testing.assert_allclose(B.primal(k), inst.l, rtol=1e-15)
        assert not B.dual(k).any() and B.dual(k).shape == (inst.m,)
    B.close()


@pytest.mark.parametrize("n", SIZES)
def test_fanout_reads(n):
    S = lib()
    inst = _shifted(n)
    inst.is_int[:3] = 1
    lp = S.LP.from_instance(inst, S.default_params(**KW))
    fan = S.Fanout(lp, np.stack([inst.l, inst.l, inst.l], axis=1))
    fan.reset_state()
    for k in range(3):
        np.testing.assert_allclose(fan.primal(k), inst.l, rtol=1e-15)
        assert fan.dual(k).shape == (inst.m,)
    fan.close()
    lp.close()
