"""The projected eigenproblems of the local eigensolves on a pair of CTAs: the smallest basis
(48), the usual one (58), the largest (160), subdomains smaller than the basis and of odd
size.  Eigenvalues against the oracle's dense solver, with the bound of the parity tests, and
the preconditioner with the coarse space they select."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2107_09006_gb300 as L  # noqa: E402
import oracle as O  # noqa: E402
from workloads import make_grid_ls, block_partition  # noqa: E402


@pytest.mark.parametrize("W,H,piece,nev", [(30, 30, 15, 4), (30, 30, 15, 16), (40, 24, 20, 67), (15, 9, 5, 6), (7, 7, 3, 3)])
def test_projected_eigenproblem(W, H, piece, nev):
    m, n, rp, c, v, b, _ = make_grid_ls(W, H, 4, 6, 2, 11)
    part = block_partition(W, H, piece, piece)
    N = int(part.max()) + 1
    S = L.Solver(m, n, rp, c, v, part, N, nev_max=nev)
    M = O.build_two_level(O.schwarz.as_csr(m, n, rp, c, v), part, N, tau=0.0, nev_max=nev)
    for i in range(N):
        lg = S.eigvals(i)
        lo = M.lams[i][: len(lg)]
        assert np.max(np.abs(lg - lo)) <= 1e-10 * max(1.0, np.abs(lo).max())
    r = np.random.default_rng(3).standard_normal(n)
    z, ref = S.apply_preconditioner(r, 0).cpu().numpy(), M.apply(r)
    assert np.linalg.norm(z - ref) <= 1e-9 * np.linalg.norm(ref)
    S.close()


@pytest.mark.parametrize("nev", [16, 32, 67])
def test_two_setups_of_a_matrix_give_the_same_bits(nev):
    """Bases of 58, 90 and 160: the rotations of a round are made by one, two and three warps,
    and the order in which the warps run must not show."""
    W = 64
    m, n, rp, c, v, b, _ = make_grid_ls(W, W, 4, 8, 3, 2)
    part = block_partition(W, W, 16, 16)
    r = np.random.default_rng(3).standard_normal(n)
    out = []
    for _ in range(4):
        S = L.Solver(m, n, rp, c, v, part, 16, nev_max=nev, spmv=2)
        out.append((np.concatenate([S.eigvals(i) for i in range(16)]), S.apply_preconditioner(r, 0).cpu().numpy()))
        S.close()
    for lam, z in out[1:]:
        assert np.array_equal(lam, out[0][0])
        assert np.array_equal(z, out[0][1])


@pytest.mark.parametrize("W,piece,nev", [(36, 2, 1), (60, 3, 2), (56, 4, 3), (72, 5, 4), (84, 6, 4)])
def test_many_tiny_subdomains(W, piece, nev):
    """196 to 400 subdomains of 2.6 to 6 block rows, on both sides of the rule that gives each a
    CTA for the whole iteration.  Eigenvalues of C v = lambda B v, B = C~ + s I, from Cholesky
    factors of B carry errors of eps cond(B) lambda, and cond(B) <= ||C~|| / s = 1e8 with the
    default shift: 1e-8 of the largest (pieces of 2 x 2 and 3 x 3 columns have lambda up to 2e5)
    and a converged solve; from 4 x 4 on lambda <= 43, and the bounds of the parity tests hold."""
    m, n, rp, c, v, b, _ = make_grid_ls(W, W, 4, 6, 2, 11)
    part = block_partition(W, W, piece, piece)
    N = int(part.max()) + 1
    S = L.Solver(m, n, rp, c, v, part, N, nev_max=nev)
    M = O.build_two_level(O.schwarz.as_csr(m, n, rp, c, v), part, N, tau=0.0, nev_max=nev)
    tol = 1e-10 if piece >= 4 else 1e-8
    for i in range(N):
        lg = S.eigvals(i)
        lo = M.lams[i][: len(lg)]
        assert np.max(np.abs(lg - lo)) <= tol * max(1.0, np.abs(lo).max())
    x, info = S.solve(b, rtol=1e-9)
    assert info["relres_true"] <= 1e-9
    if piece >= 4:
        r = np.random.default_rng(3).standard_normal(n)
        z, ref = S.apply_preconditioner(r, 0).cpu().numpy(), M.apply(r)
        assert np.linalg.norm(z - ref) <= 1e-9 * np.linalg.norm(ref)
    S.close()
