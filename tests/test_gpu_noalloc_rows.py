"""scylla_primal_residual_noalloc at the edges of its deal: one block of 256 rows (read
in aligned groups of four, or entry by entry from unaligned arrays) and several blocks,
rows of every length, empty ones among them."""
import numpy as np
import pytest

from tests.gpu_common import gpu_available, lib

pytestmark = [pytest.mark.gpu, pytest.mark.skipif(not gpu_available(), reason="needs a CUDA GPU")]


def _counts(kind, m, rng):
    k = rng.integers(0, 41, size=m)
    if kind == "empty":
        k[:] = 0
    elif kind == "one_long":
        k[m // 2] = 65
    elif kind == "long":
        k[::3] = rng.integers(500, 700, size=len(k[::3]))
    elif kind == "huge":
        k[m // 3] = 9000
        k[m - 1] = 8193
    elif kind == "limits":
        k[:] = rng.choice([0, 1, 8, 63, 64], size=m)
    return k


@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("m", [1, 255, 256, 257, 1000])
@pytest.mark.parametrize("kind", ["short", "empty", "one_long", "long", "huge", "limits"])
def test_residual_of_rows_of_every_length(kind, m, shift):
    import torch

    S = lib()
    rng = np.random.default_rng(m)
    n = 10_000
    k = _counts(kind, m, rng)
    rowptr = np.concatenate([[0], np.cumsum(k)]).astype(np.int64)
    nnz = int(rowptr[-1])
    cols = rng.integers(0, n, size=max(nnz, 1)).astype(np.int32)
    vals = rng.normal(size=max(nnz, 1))
    x = rng.normal(size=n)
    prod = vals[:nnz] * x[cols[:nnz]]
    ax = np.array([np.sum(prod[a:b]) for a, b in zip(rowptr[:-1], rowptr[1:])])
    mag = np.array([np.sum(np.abs(prod[a:b])) for a, b in zip(rowptr[:-1], rowptr[1:])])
    lo = np.where(rng.random(m) < 0.3, -np.inf, ax + rng.normal(size=m))
    hi = np.where(rng.random(m) < 0.3, np.inf, np.where(np.isfinite(lo), lo, ax) + rng.random(m))
    pad = lambda a: torch.tensor(np.concatenate([a[:shift], a]), device="cuda")[shift:]  # noqa: E731
    d = [torch.tensor(rowptr, device="cuda"), pad(cols), pad(vals)] + [torch.tensor(a, device="cuda") for a in (x, lo, hi)]
    out = torch.full((2,), -1.0, dtype=torch.float64, device="cuda")
    r = np.linalg.norm(ax - np.clip(ax, lo, hi))
    b = np.maximum(np.where(np.isfinite(lo), np.abs(lo), 0.0), np.where(np.isfinite(hi), np.abs(hi), 0.0))
    for _ in range(2):
        S.primal_residual_noalloc(m, *[t.data_ptr() for t in d], out.data_ptr(),
                                  torch.cuda.current_stream().cuda_stream)
        torch.cuda.synchronize()
        got = out.cpu().numpy()
        # either side's row sum is within (length) eps of the terms' magnitudes, the
        # norms of m terms within m eps
        tol = 2.0 * (9000 * np.linalg.norm(mag) + (m + 4) * (r + 1e-300)) * np.finfo(float).eps
        assert abs(got[0] - r) <= tol
        assert abs(got[1] - r / (1.0 + np.linalg.norm(b))) <= tol
