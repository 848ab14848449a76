"""GMRES and LSQR at fixed step counts around the widths of their device passes (the
Gram-Schmidt pass takes eight basis vectors at a time; a restart in mid-run; LSQR's two
scalar states in turn), against the oracle's loop with the device's own preconditioner, so
that only rounding differs: FP64 sums of n < 3,200 terms, a factor of kappa^2 < 1e3 and a
few steps keep that below 1e-10."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a GPU", allow_module_level=True)

import paper_2107_09006_gb300 as L  # noqa: E402
import oracle as O  # noqa: E402
from workloads import make_grid_ls, bisection_partition  # noqa: E402


@pytest.fixture(scope="module")
def prob():
    m, n, rp, c, v, b, _ = make_grid_ls(60, 52, 4, 6, 2, 5)
    part = bisection_partition(60, 52, 700, 9)
    return dict(a=(m, n, rp, c, v, part, int(part.max()) + 1), A=O.schwarz.as_csr(m, n, rp, c, v), b=b)


def rel(a, b):
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def run(prob, **kw):
    S = L.Solver(*prob["a"], nev_max=8, **kw)
    x, info = S.solve(prob["b"], rtol=1e-8)
    x = x.cpu().numpy()
    assert info["iters"] == kw["fixed_iters"]
    return S, x, lambda r: S.apply_preconditioner(r, 0).cpu().numpy()


@pytest.mark.parametrize("steps,restart", [(1, 30), (7, 30), (8, 30), (9, 30), (12, 12), (13, 5)])
def test_gmres_steps(prob, steps, restart):
    S, x, apply = run(prob, solver=2, fixed_iters=steps, restart=restart)
    xo, _ = O.fgmres(prob["A"], prob["b"], apply, fixed_iters=steps, restart=restart)
    assert rel(x, xo) < 1e-10
    S.close()


@pytest.mark.parametrize("steps", [1, 2, 3, 8])
def test_lsqr_steps(prob, steps):
    S, x, apply = run(prob, solver=1, fixed_iters=steps)
    xo, _ = O.preconditioned_lsqr(prob["A"], prob["b"], apply, fixed_iters=steps)
    assert rel(x, xo) < 1e-10
    S.close()
