"""Waits of the superblock local solve that run out are reported, not hung on.

The option test_stall selects the 32-row kernels, so the waits of the default kernel are made
to run out in the bounds-checked build (ls_debug_stall): 1 the producer warp issues no copies
(FP64 factors), 2 the last CTA of every cluster sends no messages.  A solve, a block solve or
the eigensolves of setup must then return LS_ERR_DEVICE_TIMEOUT within seconds, with every CTA
of a cluster past its barriers, and the context must stay usable: without the hook the same
call gives the answer.  Each case runs in a child process that loads that build.
"""
import os
import subprocess
import sys

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():  # pragma: no cover - CPU containers
    pytest.skip("needs a GPU", allow_module_level=True)

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import ctypes, sys, time
import numpy as np
sys.path.insert(0, ROOT)
import torch
import paper_2107_09006_gb300 as L
from workloads import make_grid_ls, block_partition
assert L.LIBRARY_PATH.endswith("libls_schwarz_dbg.so"), L.LIBRARY_PATH
stall = ctypes.CDLL(L.LIBRARY_PATH).ls_debug_stall
stall.restype = None
stall.argtypes = [ctypes.c_int]
W, P = WIDTH, PIECE
m, n, rp, c, v, b, _ = make_grid_ls(W, W, 4, 8, 3, 0, nrhs=8)
part = block_partition(W, W, P, P)
N = int(part.max()) + 1
def make(**kw):
    return L.Solver(m, n, rp, c, v, part, N, nev_max=4, spmv=2, **kw)
def timed_out(call):
    t0 = time.time()
    try:
        call()
    except L.LSError as e:
        assert e.status == L.LS_ERR_DEVICE_TIMEOUT, e
    else:
        raise AssertionError("the call did not time out")
    assert time.time() - t0 < 60.0
    torch.cuda.synchronize()
'''


def _child(width, piece, body):
    import importlib.util
    spec = importlib.util.spec_from_file_location("_ls_build_s", os.path.join(ROOT, "paper_2107_09006_gb300",
                                                                              "_build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.build(debug_bounds=True)
    code = CHILD.replace("ROOT", repr(ROOT)).replace("WIDTH", str(width)).replace("PIECE", str(piece))
    p = subprocess.run([sys.executable, "-c", code + body + "\nprint('child done')\n"], capture_output=True, text=True,
                       env=dict(os.environ, LS_SCHWARZ_BOUNDS="1"), timeout=300)
    assert p.returncode == 0 and "child done" in p.stdout, p.stderr[-3000:]


@pytest.mark.parametrize("prec,width,piece,mode", [
    ("f64", 60, 20, 1),    # 9 subdomains: clusters of 8
    ("f64", 60, 20, 2),
    ("f32", 96, 32, 2),    # 9 subdomains of 8.5 tiles a block row: a pair of CTAs each
    ("bf16", 96, 32, 2),
    ("f32", 128, 64, 2),   # 4 subdomains of 14 tiles a block row: clusters of 4
])
def test_single_vector_solve(prec, width, piece, mode):
    _child(width, piece, f"""
S = make(factor_prec={prec!r})
assert S.info()["local_config"] == 4
stall({mode})
timed_out(lambda: S.solve(b[0], rtol=1e-8))
stall(0)
S.close()
S = make(factor_prec={prec!r})
x, info = S.solve(b[0], rtol=1e-8)
assert info["relres_true"] <= 1e-8
S.close()
""")


@pytest.mark.parametrize("prec,width,piece,mode", [
    ("f64", 96, 32, 1),
    ("f64", 60, 20, 2),  # (of 32 x 32 pieces a cluster's vectors for four right-hand sides do not fit)
    ("f32", 96, 32, 2),
    ("bf16", 96, 32, 2),
])
def test_block_solve(prec, width, piece, mode):
    _child(width, piece, f"""
S = make(factor_prec={prec!r})
stall({mode})
timed_out(lambda: S.solve(b, rtol=1e-8))
stall(0)
S.close()
S = make(factor_prec={prec!r})
X, info = S.solve(b, rtol=1e-8)
assert info["local_kernel"] == 0 and (S.batch_stats(8)[1] <= 1e-8).all()
S.close()
""")


@pytest.mark.parametrize("mode", [1, 2])
def test_eigensolves_of_setup(mode):
    _child(60, 20, f"""
stall({mode})
timed_out(lambda: make())
stall(0)
S = make()
assert S.solve(b[0], rtol=1e-8)[1]["relres_true"] <= 1e-8
S.close()
""")
