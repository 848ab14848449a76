"""The allocation-free product over row lengths and row counts on both sides of its choice of
lanes per row (square root of the mean length; wider while few threads would run), with
empty and very long rows, in the caller's row order.

Tolerance: both sums of the product run in FP64 over at most 2,048 terms; the reference sums
the same products in another order: 1e-13 of the result's norm, as in test_zz_no_alloc.py.
"""
import numpy as np
import pytest
import scipy.sparse as sp
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,per_row", [(1, 1, 1), (40, 7, 2), (1023, 1024, 17), (32769, 500, 3), (8192, 8191, 4),
                                         (70000, 20000, 9), (5000, 4000, 40), (3000, 2048, 700)])
def test_noalloc_product_lanes(m, n, per_row):
    import paper_2107_09006_gb300 as L

    rng = np.random.default_rng(m + n)
    rows = np.repeat(np.arange(m), rng.integers(0, 2 * per_row + 1, m))
    A = sp.csr_matrix((rng.standard_normal(rows.size), (rows, rng.integers(0, n, rows.size))), shape=(m, n))
    A.sum_duplicates()
    A.sort_indices()
    T = A.tocsc()
    T.sort_indices()
    dev = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")  # noqa: E731
    p = rng.standard_normal(n)
    w = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    L.ls_normal_product_noalloc(m, n, dev(A.indptr, torch.int64), dev(A.indices, torch.int32), dev(A.data, torch.float64),
                                dev(T.indptr, torch.int64), dev(T.indices, torch.int32), dev(T.data, torch.float64),
                                A.nnz, dev(p, torch.float64), w, torch.cuda.current_stream().cuda_stream)
    ref = A.T @ (A @ p)
    assert np.linalg.norm(w.cpu().numpy() - ref) <= 1e-13 * max(np.linalg.norm(ref), np.linalg.norm(np.abs(A).T @ (np.abs(A) @ np.abs(p))))
