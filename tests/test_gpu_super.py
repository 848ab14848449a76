"""The superblock local solve (the default configuration 4) against the 32-row sweeps
(configuration 1, which test_gpu_parity.py holds to the oracle), in every launch shape the
rule picks: one CTA per subdomain, clusters of 2, 4 and 8, two CTAs per SM, last
superblocks of one to four block rows, subdomains of a single block row, envelopes that
start inside a superblock, block rows wider and narrower than the warps deal at once.

Tolerances: both configurations evaluate the same operator in different summation orders
(BF16: from the same rounded factors), so they differ by a small multiple of kappa(C_ii)
times the unit roundoff of the arithmetic: 1e-12 (FP64) and 1e-5 (FP32 sums), as between
the other configurations in test_gpu_parity.py.
"""
import numpy as np
import pytest
import torch

from workloads.grid import bisection_partition, block_partition, make_grid_ls, strip_partition

pytestmark = pytest.mark.gpu

# name: W, H, rows of the matrix (k, radius), partition
SHAPES = {
    "one-row": (4, 5, (4, 2), lambda W, H: np.zeros(W * H, np.int32)),
    "strips": (32, 32, (4, 2), lambda W, H: strip_partition(W, H, 4)),
    "blocks8": (24, 24, (8, 3), lambda W, H: block_partition(W, H, 8, 8)),
    "blocks32-ragged": (90, 75, (8, 3), lambda W, H: block_partition(W, H, 32, 32)),
    "bisect30": (100, 60, (6, 2), lambda W, H: bisection_partition(W, H, 300, 5)),
    "n100": (60, 60, (6, 2), lambda W, H: block_partition(W, H, 6, 6)),
    "n169": (65, 65, (6, 2), lambda W, H: block_partition(W, H, 5, 5)),
    "n400": (80, 80, (8, 3), lambda W, H: block_partition(W, H, 4, 4)),
    "wide": (128, 128, (8, 3), lambda W, H: block_partition(W, H, 64, 64)),
    "scattered": (40, 30, (6, 2), lambda W, H: (np.arange(W * H) % 3).astype(np.int32)),
}


@pytest.mark.parametrize("prec", ["f64", "f32", "bf16"])
@pytest.mark.parametrize("name", sorted(SHAPES))
def test_super_matches_row_sweeps(name, prec):
    import paper_2107_09006_gb300 as L

    W, H, (k, radius), split = SHAPES[name]
    m, n, rp, col, val, b, _ = make_grid_ls(W, H, 4, k, radius, 7)
    part = split(W, H)
    r = torch.from_numpy(np.random.default_rng(2).standard_normal(n)).cuda()
    z = {}
    for config in (0, 1):
        S = L.Solver(m, n, rp, col, val, part, int(part.max()) + 1, nev_max=4, factor_prec=prec, local_config=config)
        assert S.info()["local_config"] == (4 if config == 0 else 1)
        z[config] = S.apply_preconditioner(r, 1)
        # both levels: the coarse correction runs beside the local solves
        both = S.apply_preconditioner(r, 0)
        apart = z[config] + S.apply_preconditioner(r, 2)
        assert float((both - apart).norm() / apart.norm()) < 1e-13
        if config == 0:
            x, info = S.solve(b, rtol=1e-9)
            assert info["relres_true"] <= 1e-9
        S.close()
    tol = 1e-12 if prec == "f64" else 1e-5
    assert float((z[0] - z[1]).norm() / z[1].norm()) < tol


@pytest.mark.parametrize("prec,R", [("f64", 2), ("f64", 5), ("f32", 3), ("f32", 8), ("f32", 19), ("bf16", 4), ("bf16", 7)])
@pytest.mark.parametrize("name", ["strips", "blocks8", "blocks32-ragged", "n100", "n400"])
def test_super_many_right_hand_sides(name, prec, R):
    """Three fixed iterations of R right-hand sides (one to three groups of four or eight,
    full and partial) against the same operator elsewhere: FP64 and BF16 the single-vector
    path's, to 1e-10 and 1e-4 (the block path keeps its coarse basis in FP32); FP32 the
    tensor-core kernel with the same TF32-rounded factor, to 1e-4."""
    import paper_2107_09006_gb300 as L

    W, H, (k, radius), split = SHAPES[name]
    m, n, rp, col, val, b, _ = make_grid_ls(W, H, 4, k, radius, 7, nrhs=R)
    part = split(W, H)
    mk = lambda **o: L.Solver(m, n, rp, col, val, part, int(part.max()) + 1, nev_max=4, factor_prec=prec,  # noqa: E731
                              fixed_iters=3, **o)
    S = mk()
    X, info = S.solve(b)
    groups, sms = -(-R // 8), torch.cuda.get_device_properties(0).multi_processor_count
    wide = prec == "f32" and groups > 2 and groups * (int(part.max()) + 1) > 3 * sms  # a tensor-core kernel's ground
    assert (info["local_kernel"] == 0) != wide
    if prec == "f32":
        S2 = mk(block_kernel=2)
        ref, info = S2.solve(b)
        assert info["local_kernel"] == 2
        S2.close()
    else:
        ref = torch.stack([S.solve(b[q])[0] for q in range(R)])
    S.close()
    tol = 1e-10 if prec == "f64" else 1e-4
    for q in range(R):
        assert float((X[q] - ref[q]).norm() / ref[q].norm()) < tol, q


# the rest of the rule: name -> as above, here with the counts that select the shape
SHAPES.update({
    "n64": (128, 128, (6, 2), lambda W, H: block_partition(W, H, 16, 16)),
    "n100-32": (320, 320, (8, 3), lambda W, H: block_partition(W, H, 32, 32)),
})


def _rule(name, prec):
    """(subdomains, mean width of a block row in tiles, SMs)"""
    import paper_2107_09006_gb300 as L

    W, H, (k, radius), split = SHAPES[name]
    m, n, rp, col, val, _, _ = make_grid_ls(W, H, 4, k, radius, 7)
    part = split(W, H)
    S = L.Solver(m, n, rp, col, val, part, int(part.max()) + 1, coarse=0, factor_prec=prec)
    st = S.storage()
    S.close()
    return (int(part.max()) + 1, st["fac_elems"] / 1024 / st["total_blocks"],
            torch.cuda.get_device_properties(0).multi_processor_count)


def test_super_pair_of_ctas_in_double():
    N, _, sms = _rule("n64", "f64")
    assert 2 * N <= sms < 4 * N
    test_super_matches_row_sweeps("n64", "f64")


@pytest.mark.parametrize("prec", ["f32", "bf16"])
def test_super_one_cta_of_24_warps(prec):
    N, width, sms = _rule("n100-32", prec)
    assert N <= sms < 2 * N and width >= 8.0
    test_super_matches_row_sweeps("n100-32", prec)


def test_super_many_right_hand_sides_on_a_pair_in_double():
    N, _, sms = _rule("n64", "f64")
    assert 2 * N <= sms < 4 * N
    test_super_many_right_hand_sides("n64", "f64", 3)


@pytest.mark.parametrize("prec,tol", [("f64", 1e-10), ("f32", 1e-4), ("bf16", 1e-4)])
def test_super_timed_choice_for_wide_block_solves(prec, tol):
    """1,024 subdomains of 4 x 4 columns: with several groups of right-hand sides the superblocks
    can be the slower kernel, and the first solve of a width times both.  Whichever ran, three
    iterations agree with the 32-row kernel's (tolerances as above), also when the widths
    alternate, and the solve is not slower than that one's by more than the spread of timing
    (it was up to 2.9 times slower with BF16 factors, 1.5 with FP64)."""
    import time

    import paper_2107_09006_gb300 as L

    m, n, rp, col, val, b, _ = make_grid_ls(128, 128, 4, 6, 2, 7, nrhs=32)
    b = torch.as_tensor(np.asarray(b), device="cuda")
    part = block_partition(128, 128, 4, 4)
    mk = lambda **o: L.Solver(m, n, rp, col, val, part, 1024, coarse=0, factor_prec=prec, fixed_iters=3,  # noqa: E731
                              spmv=2, **o)
    S, S1 = mk(), mk(block_kernel=1)
    out = {}
    for R in (32, 12, 32, 8, 12):
        X, X1 = S.solve(b[:R])[0], S1.solve(b[:R])[0]
        assert float((X - X1).norm() / X1.norm()) < tol, R
        assert R not in out or torch.equal(out[R], X)
        out[R] = X

    def seconds(solver, R):
        best = 1e9
        for _ in range(7):
            torch.cuda.synchronize()
            t = time.perf_counter()
            solver.solve(b[:R])
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        return best

    for R in (12, 32):
        assert seconds(S, R) <= 1.25 * seconds(S1, R), R
    S.close()
    S1.close()
