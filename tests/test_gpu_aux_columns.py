"""Auxiliary distance columns of an LP large enough to be gathered and copied by several
host threads (slices of 65,536 columns and 262,144 nonzeros): the iterated LP's pattern,
bounds and objective are those of the definition, at every slice's ends."""
import numpy as np
import pytest
import scipy.sparse as sp

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


@pytest.mark.parametrize("m,n,per_col", [(300, 700, 4), (40_000, 131_072, 5), (70_000, 200_003, 4)])
def test_auxiliary_columns_follow_the_general_integers(m, n, per_col):
    S = lib()
    inst = I.packing_covering(m, n, per_col, seed=n)
    rng = np.random.default_rng(n)
    inst.is_int = (rng.random(n) < 0.5).astype(np.uint8)
    inst.l, inst.u = np.zeros(n), rng.integers(1, 4, n).astype(float)  # width 1: a binary, without an auxiliary column
    for j in (0, 65_535, 65_536, 66_667, 66_668, n - 1):
        if j < n:
            inst.is_int[j], inst.u[j] = 1, 3.0
    gen = np.nonzero((inst.is_int == 1) & (inst.u != 1.0))[0]
    lp = S.LP.from_instance(inst)
    na = len(gen)
    assert (lp.n_aux, lp.n_total, lp.m_total, lp.nnz_total) == (na, n + na, m + 2 * na, len(inst.cols) + 4 * na)
    A = sp.csr_matrix((np.ones(len(inst.cols)), inst.cols, inst.rowptr), shape=(m, n))
    t = np.arange(na)
    aux = sp.csr_matrix((np.ones(4 * na), (np.repeat(np.arange(2 * na), 2),
                                           np.stack([gen, n + t, gen, n + t], 1).ravel())), shape=(2 * na, n + na))
    full = sp.vstack([sp.hstack([A, sp.csr_matrix((m, na))]), aux]).tocsc()
    full.sort_indices()
    colptr, rows, vals = lp.transpose()
    np.testing.assert_array_equal(colptr, full.indptr)
    np.testing.assert_array_equal(rows, full.indices)
    # the values are those of A under the reported scaling, and -1, 1, 1, 1 in the rows of
    # an auxiliary column (products of two rounded factors: two roundings)
    R, C = lp.scaling()
    A.data = inst.vals
    aux.data = np.tile([-1.0, 1.0, 1.0, 1.0], na)
    full = sp.vstack([sp.hstack([A, sp.csr_matrix((m, na))]), aux]).tocsc()
    full.sort_indices()
    want = full.data * R[full.indices] * np.repeat(C, np.diff(full.indptr))
    np.testing.assert_allclose(vals, want, rtol=4 * np.finfo(float).eps, atol=0.0)
    lp.close()
