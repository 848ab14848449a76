"""The calls of this framework that are timed, over the range of sizes and options it is used with.

Every case is one call a user's program makes: the normal-equations product on its own, a
solve on a handle that is kept, a solve of many right-hand sides or of many problems, a
training step through the autograd function, or the whole way from a new matrix to its
solution.  The matrices are drawn like those of workloads/grid.py (random rows of k entries in
a window of the grid plus 1e-2 I rows), on the device, so that making them costs little.

Fields of a case:
  call       "product" | "solve" | "train" | "batch" | "oneshot"
  W, H       the grid (n = W H columns); batch: the smallest and largest side of the problems
  k, radius  entries of a random row and the radius of their window (4 n such rows)
  part       "block" | "strip" | "bisect", and piece: edge of a block, grid rows of a strip,
             most columns of a piece of the bisection
  zero_sum   the values of every random row sum to zero (the case the coarse space is for)
  col_scale  columns scaled by 10^U(-3, 3), with the option equilibrate
  prec, nev, rtol, nrhs, variant, solver   options of the solver
  problems   batch: how many problems one handle holds
"""
import math

import numpy as np
import torch

import paper_2107_09006_gb300 as L

_BASE = {"k": 8, "radius": 3, "part": "block", "piece": 64, "zero_sum": False, "col_scale": False, "prec": "f64",
         "nev": 16, "rtol": 1e-8, "nrhs": 1, "variant": 0, "solver": 0, "problems": 1}


def _case(call, W, H, **kw):
    return {"call": call, "W": W, "H": H, **_BASE, **kw}


def listed():
    def c(name, call, W, H, **kw):
        return {"name": name, **_case(call, W, H, **kw)}

    return [
        # w = A^T (A p) inside a caller's own loop: the smallest problem of the test suite
        # (latency and launches) and the benchmark's matrix (bandwidth)
        c("product-32x32", "product", 32, 32, k=4, radius=2),
        c("product-1024x1024", "product", 1024, 1024),
        # the smallest solve: default options (FP64 factors) on the 1,024-column test problem
        c("solve-tiny-f64", "solve", 32, 32, k=4, radius=2, part="strip", piece=4),
        # an ordinary small solve with odd sides and uneven subdomains, FP32 factors, the
        # near-singular matrix that needs its coarse space
        c("solve-ragged-f32", "solve", 211, 173, part="bisect", piece=1100, zero_sum=True, prec="f32"),
        # the plain FP64 form at an ordinary size: the benchmark's subdomains, a quarter of its grid side
        c("solve-256x256-f64", "solve", 256, 256, piece=32),
        # the benchmark: a million columns, 256 subdomains, FP32 factors in flexible PCG
        c("solve-1024x1024-f32", "solve", 1024, 1024, prec="f32", nev=32),
        # the paper's practical pairing: GMRES with RAS and the deflated second level
        c("gmres-384x384-f32", "solve", 384, 384, piece=48, zero_sum=True, prec="f32", variant=2, solver=2),
        # the paper's LSQR with the balanced second level, BF16 factors
        c("lsqr-200x200-bf16", "solve", 200, 200, piece=40, zero_sum=True, prec="bf16", variant=1, solver=1),
        # several right-hand sides on one matrix
        c("rhs8-256x256-f32", "solve", 256, 256, piece=32, prec="f32", nrhs=8),
        # independent problems that share a handle, 32 right-hand sides each
        c("batch8x32-f32", "batch", 64, 160, k=6, radius=2, part="bisect", piece=1500, prec="f32", nrhs=32, problems=8),
        # a training step: values in, solution out, gradients of values and right-hand side back
        c("train-320x320-f32", "train", 320, 320, piece=40, prec="f32", rtol=1e-10),
        # a new matrix solved once: setup (index sets, factors, eigensolves, coarse operator) and solve
        c("oneshot-128x128-f64", "oneshot", 128, 128, piece=32),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["product", "product", "solve", "solve", "solve", "solve", "solve", "batch", "train", "oneshot"])
    radius = rng.choice([2, 3])
    kw = {"radius": radius, "k": rng.choice([4, 5, 6]) if radius == 2 else rng.choice([6, 8, 9])}
    if call == "product":
        return _case(call, _log(rng, 32, 1023), _log(rng, 32, 1023), **kw)
    kw["prec"] = rng.choice(["f64", "f32", "f32", "bf16"])
    kw["rtol"] = rng.choice([1e-8, 1e-8, 1e-10])
    kw["zero_sum"] = rng.random() < 0.4
    if call == "batch":
        lo = _log(rng, 32, 100)
        return _case(call, lo, lo + rng.randint(0, 60), part="bisect", piece=rng.randint(500, 1500),
                     nrhs=rng.randint(2, 32), problems=rng.randint(2, 8), **kw)
    W, H = _log(rng, 32, 256), _log(rng, 32, 256)
    kw["part"] = rng.choice(["block", "block", "bisect"])
    kw["piece"] = rng.randint(20, 40) if kw["part"] == "block" else rng.randint(400, 1600)
    if call == "solve":
        shape = rng.choice(["one", "one", "many", "lsqr", "gmres"])
        kw["col_scale"] = shape == "one" and not kw["zero_sum"] and rng.random() < 0.2
        if shape == "many":
            kw["nrhs"] = rng.randint(2, 32)
        elif shape == "lsqr":
            kw.update(solver=1, variant=rng.choice([0, 1]))
        elif shape == "gmres":
            kw.update(solver=2, variant=rng.choice([0, 2]))
    if call == "train":
        kw["rtol"] = 1e-10
    return _case(call, W, H, **kw)


# ---- inputs ------------------------------------------------------------------------------


def _grid_matrix(W, H, c, gen):
    """CSR arrays of one grid problem on the device: 4 n random rows, then n rows 1e-2 e_j."""
    dev, n, k, rad = "cuda", W * H, c["k"], c["radius"]
    mr, w = 4 * n, 2 * rad + 1
    cx = torch.randint(0, W, (mr,), device=dev, generator=gen)
    cy = torch.randint(0, H, (mr,), device=dev, generator=gen)
    cell = torch.arange(w * w, device=dev)
    dx, dy = cell % w - rad, cell // w - rad
    cols = torch.empty((mr, k), dtype=torch.int64, device=dev)
    for s in range(0, mr, 1 << 20):
        e = min(mr, s + (1 << 20))
        gx, gy = cx[s:e, None] + dx, cy[s:e, None] + dy
        keys = torch.rand((e - s, w * w), device=dev, generator=gen)
        keys[(gx < 0) | (gx >= W) | (gy < 0) | (gy >= H)] = 2.0
        pick = torch.topk(keys, k, dim=1, largest=False).indices
        cols[s:e] = torch.sort(gy.gather(1, pick) * W + gx.gather(1, pick), dim=1).values
    vals = torch.randn((mr, k), dtype=torch.float64, device=dev, generator=gen)
    if c["zero_sum"]:
        vals = vals - vals.mean(dim=1, keepdim=True)
    row_ptr = torch.cat([torch.arange(mr + 1, device=dev) * k, mr * k + torch.arange(1, n + 1, device=dev)])
    col = torch.cat([cols.reshape(-1), torch.arange(n, device=dev)]).to(torch.int32)
    val = torch.cat([vals.reshape(-1), torch.full((n,), 1e-2, dtype=torch.float64, device=dev)])
    if c["col_scale"]:
        u = torch.rand(n, dtype=torch.float64, device=dev, generator=gen) * 6.0 - 3.0
        val = val * torch.pow(10.0, u)[col.long()]
    return mr + n, n, row_ptr, col, val


def _partition(W, H, c, seed):
    """Subdomain of every column of one grid."""
    j = np.arange(W * H)
    gx, gy = j % W, j // W
    if c["part"] == "strip":
        return (gy // c["piece"]).astype(np.int32)
    if c["part"] == "block":
        p = c["piece"]
        return ((gy // p) * -(-W // p) + gx // p).astype(np.int32)
    rng, part, todo, count = np.random.default_rng(seed), np.empty((H, W), np.int32), [(0, W, 0, H)], 0
    while todo:
        x0, x1, y0, y1 = todo.pop()
        if (x1 - x0) * (y1 - y0) <= c["piece"]:
            part[y0:y1, x0:x1] = count
            count += 1
            continue
        f = rng.uniform(0.35, 0.65)
        if x1 - x0 >= y1 - y0:
            cut = min(max(x0 + int(round(f * (x1 - x0))), x0 + 1), x1 - 1)
            todo += [(cut, x1, y0, y1), (x0, cut, y0, y1)]
        else:
            cut = min(max(y0 + int(round(f * (y1 - y0))), y0 + 1), y1 - 1)
            todo += [(x0, x1, cut, y1), (x0, x1, y0, cut)]
    return part.reshape(-1)


def _sides(c):
    """Grid sides of the problems: of a batch spread evenly over their logarithm."""
    if c["call"] != "batch":
        return [(c["W"], c["H"])]
    q = c["problems"]
    return [(s, s) for s in (int(round(c["W"] * (c["H"] / c["W"]) ** (i / max(q - 1, 1)))) for i in range(q))]


def _inputs(c, seed):
    """The matrix (block diagonal for a batch), its partition, the right-hand sides and the
    vectors that the calls take, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    rps, cols, vals, parts, m_off, n_off, nparts, nnz = [], [], [], [], [0], [0], 0, 0
    for q, (W, H) in enumerate(_sides(c)):
        m, n, rp, col, val = _grid_matrix(W, H, c, gen)
        if c["call"] != "product":
            p = _partition(W, H, c, seed + 7919 * q)
            parts.append(p + nparts)
            nparts += int(p.max()) + 1
        rps.append(rp[1:] + nnz if q else rp)
        cols.append(col + n_off[-1])
        vals.append(val)
        nnz += val.numel()
        m_off.append(m_off[-1] + m)
        n_off.append(n_off[-1] + n)
    m, n, R = m_off[-1], n_off[-1], c["nrhs"]
    s = {"m": m, "n": n, "row_ptr": torch.cat(rps), "col": torch.cat(cols).to(torch.int32), "val": torch.cat(vals),
         "nparts": nparts, "m_off": m_off, "n_off": n_off}
    if parts:
        s["part"] = torch.from_numpy(np.concatenate(parts).astype(np.int32)).cuda()
    s["b"] = torch.randn((m,) if R == 1 and c["call"] != "batch" else (R, m), dtype=torch.float64, device="cuda", generator=gen)
    s["v"] = torch.randn(n, dtype=torch.float64, device="cuda", generator=gen)
    return s


def _transpose(s):
    """The CSC arrays of A (rows ascending in every column)."""
    rows = torch.repeat_interleave(torch.arange(s["m"], device="cuda"), torch.diff(s["row_ptr"]))
    order = torch.sort(s["col"], stable=True).indices
    ptr = torch.zeros(s["n"] + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.bincount(s["col"], minlength=s["n"]).cumsum(0)
    return ptr, rows[order].to(torch.int32), s["val"][order]


def _solver(c, s):
    problems = (s["m_off"], s["n_off"]) if c["call"] == "batch" else None
    return L.Solver(s["m"], s["n"], s["row_ptr"], s["col"], s["val"], s["part"], s["nparts"], problems=problems,
                    nev_max=c["nev"], factor_prec=c["prec"], variant=c["variant"], solver=c["solver"],
                    equilibrate=int(c["col_scale"]))


def prepare(case, seed):
    c, s = case, _inputs(case, seed)
    s["case"] = c
    if c["call"] == "product":
        s["col_ptr"], s["row"], s["cval"] = _transpose(s)
        s["w"] = torch.empty(s["n"], dtype=torch.float64, device="cuda")
    elif c["call"] != "oneshot":
        s["solver"] = _solver(c, s)
    if c["call"] == "train":
        s["val"].requires_grad_(True)
        s["b"].requires_grad_(True)
    return s


def run(state):
    s, c = state, state["case"]
    if c["call"] == "product":
        L.ls_normal_product_noalloc(s["m"], s["n"], s["row_ptr"], s["col"], s["val"], s["col_ptr"], s["row"], s["cval"],
                                    s["val"].numel(), s["v"], s["w"], stream=torch.cuda.current_stream().cuda_stream)
        return s["w"]
    if c["call"] == "oneshot":
        solver = _solver(c, s)
        x, _ = solver.solve(s["b"], rtol=c["rtol"])
        solver.close()
        return x
    if c["call"] == "train":
        x = L.LSSolve.apply(s["val"], s["b"], s["solver"], c["rtol"])
        gv, gb = torch.autograd.grad(x, (s["val"], s["b"]), s["v"])
        return x.detach(), gv, gb
    x, _ = s["solver"].solve(s["b"], rtol=c["rtol"])
    return x


def work(case):
    """The matrix, the right-hand sides and the vectors read once, the results written once, and
    the multiplications and additions of one product with A^T A for each right-hand side."""
    c = case
    n = sum(W * H for W, H in _sides(c))
    m, nnz, R = 5 * n, (4 * c["k"] + 1) * n, c["nrhs"]
    a = 12 * nnz + 8 * (m + 1)
    if c["call"] == "product":
        return {"bytes": 2 * a + 16 * n, "flops": 4 * nnz}
    if c["call"] == "train":  # values, b and the gradient in; x and the gradients of values and b out
        return {"bytes": a + 8 * nnz + 8 * (2 * m + 2 * n), "flops": 12 * nnz}
    return {"bytes": a + 8 * R * (m + n), "flops": 4 * nnz * R}


def _csr(ptr, idx, val, rows, cols):
    return torch.sparse_csr_tensor(ptr, idx.long(), val, size=(rows, cols), dtype=torch.float64, device="cuda")


def exact(case, seed):
    """The least-squares solution (and the gradients) by plain conjugate gradients on the
    column-scaled normal equations in 64 bits, run until it no longer improves, twice (the second
    time on the residual of the first)."""
    c, s = case, _inputs(case, seed)
    ptr, row, cval = _transpose(s)
    if c["call"] == "product":
        A, At = _csr(s["row_ptr"], s["col"], s["val"], s["m"], s["n"]), _csr(ptr, row, cval, s["n"], s["m"])
        return At @ (A @ s["v"])
    n, col = s["n"], s["col"].long()
    sc = torch.zeros(n, dtype=torch.float64, device="cuda").index_add_(0, col, s["val"] ** 2).rsqrt()
    A = _csr(s["row_ptr"], col, s["val"] * sc[col], s["m"], n)
    At = _csr(ptr, row, cval * torch.repeat_interleave(sc, torch.diff(ptr)), n, s["m"])

    def cg(g):  # (A S)^T (A S) y = g, a column for each right-hand side
        y, r = torch.zeros_like(g), g.clone()
        p, rr = r.clone(), (r * r).sum(0)
        stop = 1e-30 * rr
        for it in range(20000):
            w = At @ (A @ p)
            a = rr / (p * w).sum(0).clamp_min(1e-300)
            y += a * p
            r -= a * w
            new = (r * r).sum(0)
            p = r + (new / rr.clamp_min(1e-300)) * p
            rr = new
            if it % 16 == 0 and bool((rr <= stop).all()):
                break
        return y

    def normal_solve(g):  # C x = g for g already scaled by S
        y = cg(g)
        y += cg(g - At @ (A @ y))
        return y

    b = s["b"].reshape(-1, s["m"]).T.contiguous()
    x = normal_solve(At @ b)
    y = x + cg(At @ (b - A @ x))  # the residual of the least-squares problem itself
    x = sc[:, None] * y
    if c["call"] == "train":
        ly = normal_solve((sc * s["v"])[:, None])
        mu, rho = (A @ ly)[:, 0], (b - A @ y)[:, 0]
        rows = torch.repeat_interleave(torch.arange(s["m"], device="cuda"), torch.diff(s["row_ptr"]))
        lam = sc * ly[:, 0]
        return x[:, 0], rho[rows] * lam[col] - mu[rows] * x[col, 0], mu
    return x[:, 0] if s["b"].dim() == 1 else x.T.contiguous()
