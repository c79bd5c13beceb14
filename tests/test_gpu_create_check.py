"""scylla_lp_create validates large LPs on the device: every kind of malformed input is
refused with the host check's code and message, the first and the last entry included,
and well-formed LPs with empty rows pass."""
import numpy as np
import pytest

from paper_2307_03466_gb300 import instances as I
from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]

BASE = I.packing_covering(9000, 20_000, 11, seed=3)  # 220k nonzeros
NAN, INF = np.nan, np.inf


def _set(field, index, value):
    def f(d):
        d[field][index] = value
    return f


def _swap(k):
    """Two neighbouring entries of the row that holds entry k exchanged."""
    def f(d):
        i = int(np.searchsorted(d["rowptr"], k, side="right")) - 1
        a = int(d["rowptr"][i])
        d["cols"][[a, a + 1]] = d["cols"][[a + 1, a]]
    return f


def _repeat(k):
    def f(d):
        i = int(np.searchsorted(d["rowptr"], k, side="right")) - 1
        a = int(d["rowptr"][i])
        d["cols"][a + 1] = d["cols"][a]
    return f


J = int(np.nonzero(BASE.is_int)[0][5])
BAD = {
    "column -1": (_set("cols", 0, -1), "column index"),
    "column n": (_set("cols", -1, 20_000), "column index"),
    "order": (_swap(100_000), "not strictly increasing"),
    "repeat": (_repeat(0), "not strictly increasing"),
    "value nan": (_set("vals", 12_345, NAN), "matrix value"),
    "value inf": (_set("vals", -1, INF), "matrix value"),
    "lo nan": (_set("lo", 0, NAN), "row bounds"),
    "hi nan": (_set("hi", 8999, NAN), "row bounds"),
    "lo inf": (_set("lo", 77, INF), "row bounds"),
    "cost": (_set("c", 19_999, -INF), "objective"),
    "crossed": (_set("l", 4, 1e6), "column bounds"),
    "upper -inf": (_set("u", 0, -INF), "column bounds"),
    "flag": (_set("is_int", 3, 2), "is_integer"),
    "fractional": (_set("u", J, 2.5), "fractional"),
}


def _create(d):
    S = lib()
    return S.LP(d["rowptr"], d["cols"], d["vals"], d["c"], d["lo"], d["hi"], d["l"], d["u"], d["is_int"], 9000, 20_000,
                S.default_params(aux_general_integers=0))


def _copy():
    return {k: getattr(BASE, k).copy() for k in ("rowptr", "cols", "vals", "c", "lo", "hi", "l", "u", "is_int")}


@pytest.mark.parametrize("name", list(BAD))
def test_malformed_large_lp_is_refused(name):
    S = lib()
    d = _copy()
    BAD[name][0](d)
    with pytest.raises(S.ScyllaError) as e:
        _create(d)
    assert e.value.code == S.ERR_INVALID_ARG and BAD[name][1] in str(e.value)


def test_large_lp_with_empty_rows_and_infinite_bounds_passes():
    d = _copy()
    # every third row's entries to the row before it
    rp = d["rowptr"].copy()
    keep = np.ones(len(d["cols"]), dtype=bool)
    for i in range(0, 3000, 3):
        keep[rp[i]:rp[i + 1]] = False
    counts = np.diff(rp)
    counts[0:3000:3] = 0
    d["rowptr"] = np.concatenate([[0], np.cumsum(counts)]).astype(np.int64)
    d["cols"], d["vals"] = d["cols"][keep], d["vals"][keep]
    d["l"][::7] = -INF
    d["u"][::11] = INF
    d["l"][BASE.is_int == 1] = 0.0
    lp = _create(d)
    assert lp.nnz_total == int(keep.sum())
    lp.close()
