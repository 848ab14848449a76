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


def _product(A, repeats=0):
    """w = A^T (A p) by the call, its reference and norm bound, and us a call (repeats > 0)"""
    import paper_2107_09006_gb300 as L

    A = A.tocsr()
    A.sort_indices()
    T = A.tocsc()
    T.sort_indices()
    m, n = A.shape
    dev = lambda a, dt: torch.as_tensor(np.ascontiguousarray(a), dtype=dt, device="cuda")  # noqa: E731
    p = np.random.default_rng(1).standard_normal(n)
    w = torch.full((n,), np.nan, dtype=torch.float64, device="cuda")
    args = (m, n, dev(A.indptr, torch.int64), dev(A.indices, torch.int32), dev(A.data, torch.float64),
            dev(T.indptr, torch.int64), dev(T.indices, torch.int32), dev(T.data, torch.float64), A.nnz,
            dev(p, torch.float64), w, torch.cuda.current_stream().cuda_stream)
    L.ls_normal_product_noalloc(*args)
    out = w.cpu().numpy()
    B = abs(A)
    us = None
    if repeats:
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(repeats):
            L.ls_normal_product_noalloc(*args)
        e1.record()
        torch.cuda.synchronize()
        us = e0.elapsed_time(e1) / repeats * 1000.0
    return out, A.T @ (A @ p), float(np.linalg.norm(B.T @ (B @ np.abs(p)))), us


def _even(m, n, k, seed=0):
    rng = np.random.default_rng(seed)
    return sp.csr_matrix((rng.standard_normal(m * k), (np.repeat(np.arange(m), k), rng.integers(0, n, m * k))),
                         shape=(m, n))


@pytest.mark.parametrize("per_row,m,n", [(1, 40000, 40000), (5, 40000, 10000), (17, 4000, 4000), (70, 3000, 3000),
                                         (300, 3000, 2500)])
def test_noalloc_product_with_long_rows_among_short_ones(per_row, m, n):
    """Rows on both sides of the length from which the whole warp takes a row (16 entries per
    lane, for every number of lanes), several of them in one warp, the first and the last row,
    and a full column: chains of at most 40,000 / 32 additions, each within eps."""
    rng = np.random.default_rng(per_row)
    A = _even(m, n, per_row).tolil()
    for r in (0, 1, 2, 37, 38, m // 2, m - 1):
        for length in (15, 16, 17, 31, 32, 33, 63, 64, 65, 127, 128, 129, 255, 256, 257, n):
            q = (r + length) % m if r not in (0, m - 1) else r
            c = rng.choice(n, min(length, n), replace=False)
            A[q, c] = rng.standard_normal(c.size)
    A[:, n // 3] = rng.standard_normal((m, 1))
    out, ref, bound, _ = _product(A)
    assert np.linalg.norm(out - ref) <= 2.3e-16 * 1300 * bound


def test_noalloc_product_time_with_a_full_row():
    """One full row in 400,000 of six entries: a chain of 100,000 entries on a few lanes would
    take 90 (eight lanes) to 230 (two) times the rest; on a warp it takes about 23 times."""
    even = _even(400000, 100000, 6)
    full = sp.vstack([even, sp.csr_matrix(np.random.default_rng(2).standard_normal((1, 100000)))])
    t0, t1 = _product(even, 50)[3], _product(full, 20)[3]
    assert t1 <= 60.0 * t0, (t0, t1)
