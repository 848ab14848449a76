"""Subdomains whose factor has very wide block rows, and very many subdomains.

A column that couples with the far end of its subdomain makes a block row of all its tiles.
From 363 tiles (11,616 columns) on, the pairs of block rows below a column of the Cholesky
no longer fit one dimension of a launch.  Checked against SciPy's sparse LU of the same local
matrices: with one level the preconditioner apply is sum_i R_i^T (C_ii + delta I)^{-1} R_i r.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a GPU", allow_module_level=True)

import scipy.sparse as sp  # noqa: E402
import scipy.sparse.linalg as spl  # noqa: E402

import paper_2107_09006_gb300 as L  # noqa: E402


def chain(n, cuts, wide, seed=0):
    """A: a scaled identity over random rows of three neighbouring columns, and for every
    subdomain of `wide` one row that couples its first column with its last; subdomains are
    the column ranges between the cuts."""
    rng = np.random.default_rng(seed)
    j = np.arange(n - 2)
    neigh = sp.csr_matrix((rng.uniform(-1, 1, 3 * (n - 2)), (np.repeat(j, 3), (j[:, None] + [0, 1, 2]).ravel())),
                          shape=(n - 2, n))
    rows = [sp.identity(n, format="csr") * 2.0, neigh]
    for i in wide:
        rows.append(sp.csr_matrix(([1.0, 0.5], ([0, 0], [cuts[i], cuts[i + 1] - 1])), shape=(1, n)))
    A = sp.vstack(rows).tocsr()
    A.sort_indices()
    part = np.repeat(np.arange(len(cuts) - 1), np.diff(cuts)).astype(np.int32)
    return A, part


def one_level(A, part, N, r, delta):
    """sum_i R_i^T (A(:, Omega_i)^T A(:, Omega_i) + delta I)^{-1} R_i r"""
    AT = A.T.tocsr()
    z = np.zeros(A.shape[1])
    Ac = A.tocsc()
    for i in range(N):
        rows = np.unique(AT[np.flatnonzero(part == i)].indices)
        om = np.unique(A[rows].indices)
        Ai = Ac[:, om]
        z[om] += spl.spsolve((Ai.T @ Ai + delta * sp.identity(len(om))).tocsc(), r[om])
    return z


@pytest.mark.parametrize("prec,tol", [("f64", 1e-9), ("f32", 1e-5)])
@pytest.mark.parametrize("tiles,narrow", [(362, 0), (363, 0), (420, 40)])
def test_wide_block_rows(tiles, narrow, prec, tol):
    """Both sides of the launch limit, alone and among subdomains of a few tiles; the tolerances
    are those of the parity tests."""
    cuts = np.concatenate([[0, 32 * tiles], 32 * tiles + 60 * np.arange(1, narrow + 1)]).astype(int)
    A, part = chain(int(cuts[-1]), cuts, [0])
    N = len(cuts) - 1
    S = L.Solver(A.shape[0], A.shape[1], A.indptr, A.indices, A.data, part, N, coarse=0, factor_prec=prec)
    r = np.random.default_rng(1).standard_normal(A.shape[1])
    z = S.apply_preconditioner(r, 1).cpu().numpy()
    zo = one_level(A, part, N, r, S.info()["delta"])
    assert np.linalg.norm(z - zo) <= tol * np.linalg.norm(zo)
    S.close()


@pytest.mark.parametrize("prec,tol", [("f64", 1e-9), ("f32", 1e-5)])
def test_more_subdomains_than_a_launch_dimension_holds(prec, tol):
    """65,600 subdomains of two columns: the single-vector path over superblocks against the
    32-row sweeps, which are forced, and two right-hand sides of the block path against it."""
    N = 65600
    A, part = chain(2 * N, 2 * np.arange(N + 1), [])
    args = (A.shape[0], A.shape[1], A.indptr, A.indices, A.data, part, N)
    rng = np.random.default_rng(1)
    r = rng.standard_normal(A.shape[1])
    z, x = {}, {}
    b = rng.standard_normal((2, A.shape[0]))
    for config in (0, 1):
        S = L.Solver(*args, coarse=0, factor_prec=prec, local_config=config, spmv=2)
        assert S.info()["local_config"] == (4 if config == 0 else 1)
        z[config] = S.apply_preconditioner(r, 1).cpu().numpy()
        x[config] = S.solve(b, rtol=1e-9)[0].cpu().numpy() if config == 0 else \
            np.stack([S.solve(v, rtol=1e-9)[0].cpu().numpy() for v in b])
        S.close()
    assert np.linalg.norm(z[0] - z[1]) <= tol * np.linalg.norm(z[1])
    # two solutions to residuals of 1e-9; C >= 4 I and ||A^T b|| <= sqrt(||C||) ||b||
    assert np.linalg.norm(x[0] - x[1]) <= 1e-7 * np.linalg.norm(x[1])
