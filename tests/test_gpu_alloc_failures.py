"""Calls that meet a device out-of-memory error, and the calls after them.

The bounds-checked build refuses a chosen allocation of the library on the host
(ls_debug_alloc).  A child process that loads it refuses, one after the other, every
allocation that a call makes.  The call must succeed or return LS_ERR_OOM, and the same call
on the same handle, with nothing refused, must then give the answer: nothing that the failed
call left half built may be used.  Nothing here makes the GPU itself run out of memory.
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
import ctypes, sys
import numpy as np
sys.path.insert(0, ROOT)
import torch
import paper_2107_09006_gb300 as L
from workloads import make_grid_ls, block_partition
assert L.LIBRARY_PATH.endswith("libls_schwarz_dbg.so"), L.LIBRARY_PATH
hook = ctypes.CDLL(L.LIBRARY_PATH).ls_debug_alloc
hook.restype = None
hook.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p]

def refuse(fail_at=0, capacity=0):
    """(allocations, peak bytes) since the last call; then refuse as given."""
    seen, peak = ctypes.c_int64(), ctypes.c_int64()
    hook(fail_at, capacity, ctypes.byref(seen), ctypes.byref(peak))
    return seen.value, peak.value

W, H = 40, 36
m, n, rp, c, v, b, _ = make_grid_ls(W, H, 3, 6, 2, 5, nrhs=12)
part = block_partition(W, H, 12, 14)
N = int(part.max()) + 1
b = np.asarray(b)

def make(**opt):
    return L.Solver(m, n, rp, c, v, part, N, nev_max=6, spmv=2, **opt)

def solve(S, R):
    return S.solve(b[:R], rtol=1e-9)[0].cpu().numpy()

ref = None

def check(x, R):
    global ref
    if ref is None:
        S = make()
        ref = np.stack([S.solve(b[k], rtol=1e-11)[0].cpu().numpy() for k in range(12)])
        S.close()
    assert np.isfinite(x).all()
    # residuals of 1e-9 and 1e-11 of ||A^T b||; ||A^T b|| / (lambda_min(C) ||x||) <= 14 here
    assert np.linalg.norm(x - ref[:R]) <= 1e-7 * np.linalg.norm(ref[:R])

def refused_one_by_one(opt, R, before=(), after=None, lasting=True):
    """Every allocation of solve(R) refused in turn (lasting: and all after it), each on a fresh
    handle (`before`: widths solved first; `after`: the width solved after the failed call,
    default R)."""
    k, failed = 1, 0
    while True:
        S = make(**opt)
        for w in before:
            check(solve(S, w), w)
        refuse(fail_at=-k if lasting else k)
        ok = True
        try:
            x = solve(S, R)
        except L.LSError as e:
            assert e.status == L.LS_ERR_OOM, e
            ok = False
            failed += 1
        seen, _ = refuse()
        if ok:
            check(x, R)
        for w in (after or R, R):
            check(solve(S, w), w)
        S.close()
        if seen < k:
            assert ok and k > 1
            return failed
        k += 1

'''


def _child(body):
    import importlib.util
    spec = importlib.util.spec_from_file_location("_ls_build_a", os.path.join(ROOT, "paper_2107_09006_gb300",
                                                                              "_build.py"))
    mod = importlib.util.module_from_spec(spec)
    spec.loader.exec_module(mod)
    mod.build(debug_bounds=True)
    code = CHILD.replace("ROOT", repr(ROOT)) + body + "\nprint('child done')\n"
    p = subprocess.run([sys.executable, "-c", code], capture_output=True, text=True,
                       env=dict(os.environ, LS_SCHWARZ_BOUNDS="1"), timeout=900)
    assert p.returncode == 0 and "child done" in p.stdout, p.stderr[-3000:]


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_block_solve_after_out_of_memory(prec):
    """The superblock storage of the block path is made by the first block solve: an error on
    the way must not leave a plan that names storage which is not there."""
    _child(f"assert refused_one_by_one(dict(factor_prec={prec!r}), 3) > 0")


@pytest.mark.parametrize("opt", ["dict(factor_prec='f32', block_kernel=1)", "dict(factor_prec='f32', block_kernel=2)",
                                 "dict(factor_prec='f64', block_kernel=1)"])
def test_block_kernel_copies_after_out_of_memory(opt):
    """The factor copies of the two tensor-core kernels (and the CUDA-core kernel, which
    makes none)."""
    _child(f"assert refused_one_by_one({opt}, 3) > 0")


@pytest.mark.parametrize("opt", ["dict(factor_prec='f64')", "dict(factor_prec='f32', block_kernel=1)"])
def test_narrow_block_solve_after_a_wider_one_ran_out_of_memory(opt):
    """A wider block solve replaces the work vectors of a narrower one; after an error on the
    way the narrower solve must not use those that went."""
    _child(f"assert refused_one_by_one({opt}, 5, before=(2,), after=2) > 0")


@pytest.mark.parametrize("opt", ["dict(factor_prec='f64')", "dict(factor_prec='f32')", "dict(factor_prec='bf16')",
                                 "dict(factor_prec='f32', block_kernel=2)"])
def test_block_solve_makes_room(opt):
    """One refusal: the superblock copies of the factor are for speed only, so the call goes
    without them instead of failing."""
    _child(f"assert refused_one_by_one({opt}, 3, lasting=False) == 0")


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_block_solve_below_its_superblock_storage(prec):
    """A ceiling just below what the solve takes with its superblock storage: the 32-row kernels
    run, and so they do in the solves after it."""
    _child(f"""
S = make(factor_prec={prec!r})
refuse()
check(solve(S, 3), 3)
_, full = refuse()
S.close()
S = make(factor_prec={prec!r})
refuse(capacity=full - 1)
check(solve(S, 3), 3)
_, peak = refuse()
assert peak < full
check(solve(S, 3), 3)
check(S.solve(b[0], rtol=1e-9)[0].cpu().numpy()[None], 1)
g = np.random.default_rng(2).standard_normal((3, n))
gb, gv, _ = S.backward(b[:3], ref[:3], g, rtol=1e-10)
S.close()
S = make(factor_prec={prec!r}, local_config=1, block_kernel=1)
ob = np.stack([S.backward(b[k], ref[k], g[k], rtol=1e-10)[0].cpu().numpy() for k in range(3)])
assert np.linalg.norm(gb.cpu().numpy() - ob) <= 1e-7 * np.linalg.norm(ob)
S.close()
""")


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
def test_setup_without_room_for_the_superblock_copies(prec):
    """Every allocation of setup refused once, and a ceiling just below its peak: setup goes
    without the copies (the 32-row kernels, one CTA per subdomain in the eigensolves)."""
    _child(f"""
check(np.stack([make(factor_prec={prec!r}).solve(b[0], rtol=1e-9)[0].cpu().numpy()]), 1)
import gc; gc.collect()
refuse()
S = make(factor_prec={prec!r})
assert S.info()["local_config"] == 4
count, full = refuse()
lam = S.eigvals(0)
S.close()
for k in list(range(1, count + 1, 7)) + [0]:
    refuse(fail_at=k, capacity=0 if k else full - 1)
    S = make(factor_prec={prec!r})
    _, peak = refuse()
    assert S.info()["local_config"] in (1, 2, 3), k
    assert k or peak < full
    assert np.max(np.abs(S.eigvals(0) - lam)) <= 1e-10 * max(1.0, np.abs(lam).max())
    check(S.solve(b[0], rtol=1e-9)[0].cpu().numpy()[None], 1)
    check(solve(S, 3), 3)
    S.close()
refuse(fail_at=-1)
try:
    make(factor_prec={prec!r})
    raise AssertionError("setup without any memory")
except L.LSError as e:
    assert e.status == L.LS_ERR_OOM
refuse()
S = make(factor_prec={prec!r})
assert S.info()["local_config"] == 4
S.close()
""")


def test_backward_and_value_update_after_out_of_memory():
    _child("""
g = np.random.default_rng(2).standard_normal(n)
outs = []
for k in (0, 1, 2, 4, 6, -1, -3, -6):
    S = make(factor_prec='f32')
    x = S.solve(b[0], rtol=1e-9)[0]
    check(x.cpu().numpy()[None], 1)
    refuse(fail_at=k)
    try:
        S.backward(b[0], x, g, rtol=1e-10)
        assert k >= 0
    except L.LSError as e:
        assert k < 0 and e.status == L.LS_ERR_OOM
    refuse(fail_at=k)
    try:
        S.update_values(v)
    except L.LSError as e:
        assert k < 0 and e.status == L.LS_ERR_OOM
    refuse()
    S.update_values(v)
    gb, gv, _ = S.backward(b[0], x, g, rtol=1e-10)
    outs.append((gb.cpu().numpy(), gv.cpu().numpy()))
    S.close()
for gb, gv in outs[1:]:
    assert np.linalg.norm(gb - outs[0][0]) <= 1e-7 * np.linalg.norm(outs[0][0])
    assert np.linalg.norm(gv - outs[0][1]) <= 1e-6 * np.linalg.norm(outs[0][1])
""")
