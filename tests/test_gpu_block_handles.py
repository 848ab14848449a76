"""Two handles of the tcgen05 block local solve in one process: the one with the wider window
(more shared memory) still solves after the other has been set up and has solved."""
import numpy as np
import pytest

from workloads.grid import block_partition, make_grid_ls

pytestmark = pytest.mark.gpu


def test_wide_handle_solves_after_a_narrow_one():
    import paper_2107_09006_gb300 as L

    def handle(W, block):
        m, n, rp, col, val, b, _ = make_grid_ls(W, W, 4, 8, 3, 5, nrhs=3)
        part = block_partition(W, W, block, block)
        return L.Solver(m, n, rp, col, val, part, int(part.max()) + 1, nev_max=4, factor_prec="f32", block_kernel=2), b

    wide, bw = handle(96, 48)
    narrow, bn = handle(32, 8)
    for S, b in ((narrow, bn), (wide, bw), (narrow, bn)):
        X, info = S.solve(b, rtol=1e-9)
        assert info["local_kernel"] == 2 and info["relres_true"] <= 1e-9
        assert np.isfinite(X.cpu().numpy()).all()
    wide.close()
    narrow.close()
