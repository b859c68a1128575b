"""The work whose speed counts: what a user of the library has it do, through its public
entry points, over the sizes, value types, numberings, basis loops and options it serves.

The problems are parallel-beam tomography (the library's workload) at the sizes of
tomo.CONFIGS, of the batch generators and of the tests, and at odd sizes between them.
The rays start a quarter of an angle step off the axes, so none runs along a grid line,
and the projector is built on the GPU (tomo.siddon_csr takes minutes at 512 x 512).  A
scanner's geometry stays while its scans change: a program keeps one handle per geometry,
so the handles are kept here too, and a seed draws the phantom and the noise of a scan.

The FP32 and FP64 recurrences amplify rounding about a hundredfold every two or three
iterations once it reaches the pivots, so beyond the first iterations two correct
summation orders differ by per cents: exact() gives a value where one exists (FP64, or
few iterations) and None elsewhere.
"""
from __future__ import annotations

import ctypes
import functools
import math
import types

import numpy as np
import torch

from paper_2409_05239_gb300 import lslu, tomo

VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2}


def listed():
    return [
        # one product in each direction on the smallest workload: what a caller that runs
        # its own iteration pays per step (launch latency)
        {"name": "products_32_f64", "kind": "products", "side": 32, "angles": 45, "rays": 46,
         "values": "f64"},
        # the projected problem alone, on device buffers and without allocation, at a
        # size where a stopping rule would end a solve
        {"name": "projected_60", "kind": "projected", "k": 60, "rule": "gcv"},
        # the smallest workload in the reference precision, in the loop meant for it
        {"name": "cluster_32_f64", "kind": "solve", "side": 32, "angles": 45, "rays": 46, "K": 50,
         "values": "f64", "order": "natural", "loop": "cluster", "rule": "gcv"},
        # the same workload in FP32 as a first user calls it: host arrays, default loop,
        # the lambda and residual of every iteration
        {"name": "history_32_f32", "kind": "host", "side": 32, "angles": 45, "rays": 46, "K": 50,
         "values": "f32", "order": "natural", "rule": "wgcv", "histories": True},
        # a matrix met for the first time, in host arrays: what its handle costs, with one
        # product in each direction
        {"name": "setup_128_f32", "kind": "setup", "side": 128, "angles": 120, "rays": 181,
         "K": 30, "values": "f32"},
        # the 256 x 256 workload (the paper's image size), renumbered as the benchmark does
        {"name": "solve_256_f32", "kind": "solve", "side": 256, "angles": 180, "rays": 362,
         "K": 200, "values": "f32", "order": "tiles", "loop": "graph", "rule": "gcv"},
        # the paper's stopping rule at that size, BF16 values, matrix as numbered
        {"name": "stopping_256_bf16", "kind": "stopping", "side": 256, "angles": 180, "rays": 362,
         "K": 200, "values": "bf16", "order": "natural", "rule": "wgcv"},
        # independent problems of uneven size in one launch sequence
        {"name": "batch_16_f32", "kind": "batch", "count": 16, "side_lo": 64, "side_hi": 256,
         "angles_lo": 30, "angles_hi": 180, "sizes_seed": 4000, "K": 60, "values": "f32",
         "rule": "gcv"},
        # sixteen scans of one scanner at once
        {"name": "shared_16_256_f32", "kind": "shared", "nrhs": 16, "side": 256, "angles": 180,
         "rays": 362, "K": 50, "values": "f32", "order": "tiles", "rule": "gcv"},
        # a training step through the solve: forward, loss, backward to the data and lambda
        {"name": "gradient_128_f32", "kind": "gradient", "side": 128, "angles": 180, "rays": 181,
         "K": 12, "values": "f32", "order": "natural", "lam": 0.5},
        # FP64 with histories and posterior variances afterwards, matrix as numbered
        {"name": "uq_160_f64", "kind": "uq", "side": 160, "angles": 180, "rays": 226, "K": 40,
         "values": "f64", "order": "natural", "rule": "gcv"},
        # the benchmark workload
        {"name": "solve_512_f32", "kind": "solve", "side": 512, "angles": 360, "rays": 724,
         "K": 300, "values": "f32", "order": "tiles", "loop": "graph", "rule": "gcv"},
    ]


def draw(rng):
    """A case of the ranges above, sizes spread over their logarithm."""

    def log_int(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    def geometry(lo, hi):
        side = log_int(lo, hi)
        return {"side": side, "angles": max(12, int(round(side * rng.uniform(0.7, 1.4)))),
                "rays": int(round(1.41 * side)) + rng.randint(0, 3)}

    kind = rng.choice(["products", "projected", "solve", "solve", "host", "setup", "stopping",
                       "batch", "shared", "gradient", "uq"])
    rule = rng.choice(["gcv", "wgcv"])
    order = rng.choice(["natural", "tiles"])
    if kind == "products":
        return {"kind": kind, **geometry(32, 300), "values": rng.choice(["f64", "f32", "bf16"])}
    if kind == "projected":
        return {"kind": kind, "k": log_int(8, 200), "rule": rule}
    if kind == "solve":
        if rng.random() < 0.3:  # sizes that the cluster loop holds in shared memory
            return {"kind": kind, **geometry(20, 34), "K": log_int(10, 50),
                    "values": rng.choice(["f64", "f32"]), "order": order, "loop": "cluster",
                    "rule": rule}
        return {"kind": kind, **geometry(40, 360), "K": log_int(20, 200),
                "values": rng.choice(["f32", "f32", "bf16", "f64"]), "order": order,
                "loop": "graph", "rule": rule}
    if kind == "host":
        return {"kind": kind, **geometry(24, 96), "K": log_int(10, 60),
                "values": rng.choice(["f64", "f32", "bf16"]), "order": order, "rule": rule,
                "histories": rng.random() < 0.5}
    if kind == "setup":
        return {"kind": kind, **geometry(24, 128), "K": log_int(8, 40),
                "values": rng.choice(["f64", "f32", "bf16"])}
    if kind == "stopping":
        return {"kind": kind, **geometry(40, 256), "K": log_int(60, 200),
                "values": rng.choice(["f32", "bf16", "f64"]), "order": order, "rule": rule}
    if kind == "batch":
        lo = log_int(32, 100)
        return {"kind": kind, "count": log_int(4, 24), "side_lo": lo, "side_hi": 2 * lo,
                "angles_lo": 30, "angles_hi": 180, "sizes_seed": rng.randint(1, 10**6),
                "K": log_int(20, 80), "values": rng.choice(["f32", "bf16"]), "rule": rule}
    if kind == "shared":
        return {"kind": kind, "nrhs": rng.randint(2, 16), **geometry(48, 200), "K": log_int(15, 60),
                "values": rng.choice(["f32", "bf16"]), "order": order, "rule": rule}
    if kind == "gradient":
        side = log_int(32, 140)
        return {"kind": kind, "side": side, "angles": int(round(1.4 * side)),
                "rays": int(round(1.41 * side)), "K": log_int(5, 12),
                "values": rng.choice(["f32", "f64"]), "order": order, "lam": 0.5}
    return {"kind": kind, **geometry(40, 160), "K": log_int(10, 40),
            "values": rng.choice(["f64", "f32"]), "order": order, "rule": rule}


# ---- problems -----------------------------------------------------------------------


def projector(side, angles, rays):
    """CSR of the ray-pixel intersection lengths (row_ptr int64, columns int32, values
    FP64, on the GPU); pixels row by row, rays angle by angle, columns sorted."""
    dev = torch.device("cuda")
    f64 = dict(dtype=torch.float64, device=dev)
    half = 0.5 * side
    grid = torch.arange(side + 1, **f64) - half
    s = torch.arange(rays, **f64) - 0.5 * (rays - 1)
    step = max(1, (1 << 24) // (rays * (2 * side + 2)))
    counts, cols, vals = [], [], []
    for a0 in range(0, angles, step):
        a = torch.arange(a0, min(angles, a0 + step), **f64)
        th = (a + 0.25) * (math.pi / angles)
        c, sn = torch.cos(th)[:, None, None], torch.sin(th)[:, None, None]
        px, py = -s[None, :, None] * sn, s[None, :, None] * c
        tx, ty = (grid - px) / c, (grid - py) / sn
        lo = torch.maximum(torch.minimum(tx[..., :1], tx[..., -1:]),
                           torch.minimum(ty[..., :1], ty[..., -1:]))
        hi = torch.minimum(torch.maximum(tx[..., :1], tx[..., -1:]),
                           torch.maximum(ty[..., :1], ty[..., -1:]))
        t = torch.cat([tx, ty], -1)
        t = torch.minimum(torch.maximum(t, lo), hi).sort(-1).values
        seg, mid = t[..., 1:] - t[..., :-1], 0.5 * (t[..., 1:] + t[..., :-1])
        ix = torch.floor(px + mid * c + half).long()
        iy = torch.floor(py + mid * sn + half).long()
        keep = (seg > 1e-10) & (ix >= 0) & (ix < side) & (iy >= 0) & (iy < side) & (hi > lo)
        ray = torch.arange(keep.shape[0] * rays, device=dev).view(-1, rays, 1)
        key, at = (ray * (side * side) + iy * side + ix)[keep].sort(stable=True)
        counts.append(torch.bincount(key // (side * side), minlength=keep.shape[0] * rays))
        cols.append((key % (side * side)).int())
        vals.append(seg[keep][at])
    row_ptr = torch.zeros(angles * rays + 1, dtype=torch.int64, device=dev)
    row_ptr[1:] = torch.cumsum(torch.cat(counts), 0)
    return row_ptr, torch.cat(cols), torch.cat(vals)


def product(row_ptr, cols, vals, x):
    """A x in FP64, each row summed in one order whatever the run."""
    return torch.segment_reduce(vals * x[cols.long()], "sum", lengths=row_ptr.diff(), unsafe=True)


@functools.lru_cache(maxsize=1)
def geometry(side, angles, rays):
    A = projector(side, angles, rays)
    return types.SimpleNamespace(N=side, n_ang=angles, p=rays, m=angles * rays, n=side * side, A=A)


def scan(g, rng, ellipses=5):
    """A phantom and its noisy data (FP64 on the GPU; read out in FP32 as a detector's)."""
    x_true = torch.from_numpy(tomo.ellipse_phantom(g.N, ellipses, rng)).cuda()
    clean = product(*g.A, x_true)
    e = torch.from_numpy(rng.standard_normal(g.m)).cuda()
    b = clean + rng.uniform(0.005, 0.02) * clean.norm() / e.norm() * e
    return x_true, b.float().double()


def orders(g, order, device):
    if order != "tiles":
        return None
    return [torch.from_numpy(o).cuda() if device else o for o in tomo.locality_order(g)]


def batch_sizes(case):
    rng = np.random.default_rng(case["sizes_seed"])
    sides = rng.integers(case["side_lo"], case["side_hi"] + 1, case["count"])
    angles = rng.integers(case["angles_lo"], case["angles_hi"] + 1, case["count"])
    return [(int(s), int(a), int(round(1.41 * s))) for s, a in zip(sides, angles)]


def shape_of(case):
    return case["side"], case["angles"], case["rays"]


def zero_free_memory():
    """Device memory comes back from cudaMalloc as its last owner left it.  A handle is
    created on zeroed memory, so that its results cannot depend on what ran before: blocks
    of every size that the driver carves out of its pools are taken, zeroed and given back."""
    torch.cuda.synchronize()
    lib, held = lslu.load(), []
    for log2_size, count in ((21, 32), (20, 64), (18, 64), (16, 128), (14, 128), (12, 256), (9, 512)):
        for _ in range(count):
            p = ctypes.c_void_p()
            if lib.cudaMalloc(ctypes.byref(p), ctypes.c_size_t(1 << log2_size)) == 0:
                lib.cudaMemset(p, 0, ctypes.c_size_t(1 << log2_size))
                held.append(p)
    torch.cuda.synchronize()
    for p in held:
        lib.cudaFree(p)


@functools.lru_cache(maxsize=1)
def single_handle(shape, values, K, order, loop):
    g = geometry(*shape)
    o = orders(g, order, True) or (None, None)
    zero_free_memory()
    s = lslu.Solver(g.m, g.n, *g.A, value_type=values, max_iter=K, row_order=o[0], col_order=o[1])
    if loop != "graph":
        s.set_loop(loop)
    return g, s


def host_csr(g):
    return (g.m, g.n, *(t.cpu().numpy() for t in g.A))


@functools.lru_cache(maxsize=1)
def batch_handle(shapes, values, K):
    gs = [geometry.__wrapped__(*shape) for shape in shapes]
    zero_free_memory()
    return gs, lslu.BatchedSolver([host_csr(g) for g in gs], value_type=values, max_iter=K)


@functools.lru_cache(maxsize=1)
def shared_handle(shape, values, K, nrhs, order):
    g = geometry(*shape)
    zero_free_memory()
    return g, lslu.BatchedSolver(host_csr(g), value_type=values, max_iter=K, nrhs=nrhs,
                                 orders=orders(g, order, False))


def prepare(case, seed):
    rng = np.random.default_rng(seed)
    kind, K = case["kind"], case.get("K")
    st = {"kind": kind, "K": K, "rule": case.get("rule"), "case": case}
    dev = dict(device="cuda")
    if kind == "projected":
        # H of a basis built on the 32 x 32 workload, as a solve hands it over
        k = case["k"]
        g = geometry(32, 45, 46)
        _, b = scan(g, rng)
        basis = reference_basis(reference_operator(g, "f64", torch.float64), b, k)
        st |= {"H": basis["H"].t().contiguous().t(), "beta": float(basis["beta"]), "m": g.m}
        for name, size in (("y", k), ("sigma", k), ("c", k + 1), ("lam", 1), ("resid", 1)):
            st[name] = torch.empty(size, dtype=torch.float64, **dev)
        return st
    if kind in ("batch", "shared"):
        if kind == "batch":
            gs, st["solver"] = batch_handle(tuple(batch_sizes(case)), case["values"], K)
        else:
            g, st["solver"] = shared_handle(shape_of(case), case["values"], K, case["nrhs"],
                                            case["order"])
            gs = [g] * case["nrhs"]
        st["b"] = torch.cat([scan(g, rng)[1] for g in gs])
        P = len(gs)
        st["x"] = torch.empty(sum(g.n for g in gs), dtype=torch.float64, **dev)
        st["gp"] = torch.empty(P, K, dtype=torch.int32, **dev)
        st["tp"] = torch.empty(P, K + 1, dtype=torch.int32, **dev)
        st["k_done"] = torch.empty(P, dtype=torch.int32, **dev)
        st["status"] = torch.empty(P, dtype=torch.int32, **dev)
        return st
    basis = torch.float64 if case["values"] == "f64" else torch.float32
    if kind in ("products", "setup"):
        g = geometry(*shape_of(case))
        st["x"] = torch.from_numpy(rng.standard_normal(g.n)).to(basis).cuda()
        st["d"] = torch.from_numpy(rng.standard_normal(g.m)).to(basis).cuda()
        st["u"] = torch.empty(g.m, dtype=basis, **dev)
        st["q"] = torch.empty(g.n, dtype=basis, **dev)
        if kind == "setup":
            return st | {"A": host_csr(g), "values": case["values"]}
    g, st["solver"] = single_handle(shape_of(case), case["values"], K or 8,
                                    case.get("order", "natural"), case.get("loop", "graph"))
    if kind == "products":
        return st
    x_true, b = scan(g, rng, 20 if case["side"] >= 512 else 5)
    if kind in ("host", "stopping", "uq"):
        st["b"] = b.cpu().numpy()
        st["histories"] = kind == "uq" or bool(case.get("histories"))
    elif kind == "gradient":
        st |= {"b": b.to(basis), "x_true": x_true,
               "log_lam": torch.tensor(math.log(case["lam"]), dtype=basis, **dev)}
    else:
        st |= {"b": b, "x": torch.empty(g.n, dtype=torch.float64, **dev),
               "gp": torch.empty(K, dtype=torch.int32, **dev),
               "tp": torch.empty(K + 1, dtype=torch.int32, **dev)}
    return st


def run(st):
    kind, K, rule = st["kind"], st["K"], st["rule"]
    if kind == "products":
        st["solver"].spmv(0, st["x"], st["u"])
        st["solver"].spmv(1, st["d"], st["q"])
        return {"u": st["u"], "q": st["q"]}
    if kind == "projected":
        lslu.projected_noalloc(st["H"], st["beta"], rule, 0.0, st["m"], st["y"], st["sigma"],
                               st["c"], st["lam"], st["resid"])
        return {k: st[k] for k in ("y", "sigma", "c", "lam", "resid")}
    if kind == "solve":
        st["solver"].solve_device(st["b"], st["x"], K, rule, gp=st["gp"], tp=st["tp"])
        return {k: st[k] for k in ("x", "gp", "tp")}
    if kind in ("batch", "shared"):
        st["solver"].solve_device(st["b"], st["x"], K, rule, gp=st["gp"], tp=st["tp"],
                                  k_done=st["k_done"], status=st["status"])
        return {k: st[k] for k in ("x", "gp", "tp", "k_done", "status")}
    if kind == "host":
        r = st["solver"].solve(st["b"], K, rule, histories=st["histories"])
        return {k: r[k] for k in ("x", "gp", "tp", "lam_hist", "res_hist", "k_done")}
    if kind == "setup":
        with lslu.Solver(*st["A"], value_type=st["values"], max_iter=K) as s:
            s.spmv(0, st["x"], st["u"])
            s.spmv(1, st["d"], st["q"])
        return {"u": st["u"], "q": st["q"]}
    if kind == "stopping":
        return st["solver"].solve_stopping(st["b"], K, rule, tol=1e-6)
    if kind == "gradient":
        b = st["b"].detach().requires_grad_()
        log_lam = st["log_lam"].detach().requires_grad_()
        x = lslu.hybrid_lslu(st["solver"], b, log_lam, K)
        loss = (x - st["x_true"]).square().sum()
        db, dlog = torch.autograd.grad(loss, (b, log_lam))
        return {"x": x.detach(), "loss": loss.detach(), "db": db, "dlog_lam": dlog}
    r = st["solver"].solve(st["b"], K, rule, histories=True)
    v = st["solver"].uq(1e-4, max(float(r["lam_hist"][-1]), 1e-3))
    return {**{k: r[k] for k in ("x", "gp", "tp", "lam_hist", "res_hist")}, **v}


# ---- what a pass cannot do without --------------------------------------------------


def solve_work(m, n, nnz, K, values, nrhs=1):
    """K iterations: A and its transpose read once each (a value and a 2-byte column
    per non-zero) and every earlier basis vector read once, per iteration."""
    s = 8 if values == "f64" else 4
    eliminated = n * K * (K - 1) / 2 + m * K * (K + 1) / 2
    return {"bytes": 2 * K * nnz * (VALUE_BYTES[values] + 2) + nrhs * s * (
                eliminated + (4 * K + 1) * (m + n)),
            "flops": nrhs * (4.0 * K * nnz + 2 * eliminated)}


def work(case):
    kind, K, values = case["kind"], case.get("K"), case.get("values")
    if kind == "projected":  # H once, the results once; the bidiagonalisation's operations
        return {"bytes": 8 * (case["k"] * (case["k"] + 4)), "flops": 8 / 3 * case["k"] ** 3}

    def size(side, angles, rays):  # a ray crosses 4/pi pixels per unit length on average
        return angles * rays, side * side, 4 / math.pi * angles * side * side

    if kind == "batch":
        parts = [solve_work(*size(*s), K, values) for s in batch_sizes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    m, n, nnz = size(*shape_of(case))
    if kind in ("products", "setup"):
        s = 8 if values == "f64" else 4
        products = 2 * nnz * (VALUE_BYTES[values] + 2) + 2 * s * (m + n)
        # a new handle: the caller's CSR read once, both stored matrices written once
        return {"bytes": products * (2 if kind == "setup" else 1) + (
                    12 * nnz + 8 * m if kind == "setup" else 0), "flops": 4 * nnz}
    if kind == "stopping":  # the rule ends these problems after 20 to 40 iterations
        K = min(K, 30)
    w = solve_work(m, n, nnz, K, values, case.get("nrhs", 1))
    if kind == "gradient":  # the reverse sweep: the same products and passes, transposed
        w = {k: 2 * v for k, v in w.items()}
    return w


# ---- the method in 64 bits, in plain torch and numpy --------------------------------


def reference_operator(g, values, dtype):
    """(x -> A x, d -> A^T d) with A's values as the handle stores them."""
    row_ptr, cols, vals = g.A
    if values != "f64":
        vals = vals.float().to(torch.bfloat16 if values == "bf16" else torch.float32).to(dtype)
    A = torch.sparse_csr_tensor(row_ptr, cols.long(), vals, (g.m, g.n))
    rows = torch.repeat_interleave(torch.arange(g.m, device="cuda"), row_ptr.diff())
    at = torch.sort(cols, stable=True).indices
    ptr = torch.zeros(g.n + 1, dtype=torch.int64, device="cuda")
    ptr[1:] = torch.cumsum(torch.bincount(cols, minlength=g.n), 0)
    At = torch.sparse_csr_tensor(ptr, rows[at], vals[at], (g.n, g.m))

    class Product(torch.autograd.Function):
        @staticmethod
        def forward(ctx, x, adjoint):
            ctx.adjoint = adjoint
            return (At if adjoint else A) @ x

        @staticmethod
        def backward(ctx, y_bar):
            return (A if ctx.adjoint else At) @ y_bar, None

    return lambda x: Product.apply(x, False), lambda d: Product.apply(d, True)


def reference_basis(operator, b, K):
    """The two bases with pivoting: A L = D H, A^T D = L W."""
    forward, adjoint = operator

    def step(q, B, piv):
        """Remove the earlier vectors from q at their pivots, then scale by the pivot."""
        if piv:
            at = torch.tensor(piv, device="cuda")
            basis = torch.stack(B, 1)
            c = torch.linalg.solve_triangular(basis[at], q[at][:, None], upper=False,
                                              unitriangular=True)[:, 0]
            q = q - basis @ c
            q = q.index_fill(0, at, 0.0)
        else:
            c = q[:0]
        i = int(torch.argmax(q.detach().abs()))
        return q / q[i], i, torch.cat([c, q[i:i + 1]])

    d, i, beta = step(b, [], [])
    D, t, L, g, H, W = [d], [i], [], [], [], []
    for k in range(K):
        l, i, w = step(adjoint(D[k]), L, g)
        L.append(l)
        g.append(i)
        W.append(torch.cat([w, w.new_zeros(K - k - 1)]))
        d, i, h = step(forward(l), D, t)
        D.append(d)
        t.append(i)
        H.append(torch.cat([h, h.new_zeros(K - k - 1)]))
    return {"L": torch.stack(L, 1), "D": torch.stack(D, 1), "H": torch.stack(H, 1),
            "W": torch.stack(W, 1), "beta": beta[0]}


def reference_projected(H, beta, rule, m):
    """y, sigma, |c|, lambda and the residual of min ||beta e1 - H y||^2 + lambda^2 ||y||^2,
    lambda the minimiser of the (weighted) GCV function."""
    k = H.shape[1]
    U, s, Vt = np.linalg.svd(H, full_matrices=True)
    c = beta * U[0]
    omega = (k + 1) / m if rule == "wgcv" else 1.0

    def parts(mu):
        f = mu / (s * s + mu)
        df = s * s / (s * s + mu) ** 2
        num = np.sum((f * c[:k]) ** 2) + c[k] ** 2
        den = 1.0 + np.sum(((1.0 - omega) * s * s + mu) / (s * s + mu))
        return num / den**2, np.sum(2 * f * df * c[:k] ** 2) * den - 2 * num * omega * np.sum(df)

    grid = s[0] * 10.0 ** (-14.0 + 0.0625 * np.arange(257))
    best = int(np.argmin([parts(lam * lam)[0] for lam in grid]))
    lam = grid[best]
    if 0 < best < 256:
        lo, hi = np.log(grid[best - 1]), np.log(grid[best + 1])
        if parts(np.exp(2 * lo))[1] < 0 < parts(np.exp(2 * hi))[1]:
            for _ in range(64):
                mid = 0.5 * (lo + hi)
                lo, hi = (mid, hi) if parts(np.exp(2 * mid))[1] < 0 else (lo, mid)
            lam = np.exp(0.5 * (lo + hi))
    f = lam * lam / (s * s + lam * lam)
    y = Vt.T @ (s * c[:k] / (s * s + lam * lam))
    return y, s, np.abs(c), lam, math.sqrt(np.sum((f * c[:k]) ** 2) + c[k] ** 2)


#: Iterations up to which rounding has not reached the pivots.
STABLE = {"f64": 16, "f32": 6, "bf16": 6}


def stable(case):
    """Twice as many rays as pixels damp the recurrence on the smallest images."""
    small = case["side"] <= 34 and case["angles"] * case["rays"] >= 1.9 * case["side"] ** 2
    return case["K"] <= (50 if small else STABLE[case["values"]])


def exact(case, seed):
    kind, K, values, rule = case["kind"], case.get("K"), case.get("values"), case.get("rule")
    f64 = torch.float64
    if kind == "projected":
        st = prepare(case, seed)
        y, s, c, lam, resid = reference_projected(st["H"].cpu().numpy(), st["beta"], rule, st["m"])
        return {"y": y, "sigma": s, "c": c, "lam": np.array([lam]), "resid": np.array([resid])}
    if kind in ("products", "setup"):
        st = prepare(case, seed)
        forward, adjoint = reference_operator(geometry(*shape_of(case)), values, f64)
        return {"u": forward(st["x"].to(f64)), "q": adjoint(st["d"].to(f64))}
    if kind == "gradient":
        st = prepare(case, seed)
        b = st["b"].to(f64).requires_grad_()
        log_lam = st["log_lam"].to(f64).requires_grad_()
        basis = reference_basis(reference_operator(geometry(*shape_of(case)), values, f64), b, K)
        H = basis["H"]
        rhs = basis["beta"] * H[0]
        M = H.t() @ H + torch.exp(2 * log_lam) * torch.eye(K, dtype=f64, device="cuda")
        x = basis["L"] @ torch.linalg.solve(M, rhs)
        loss = (x - st["x_true"]).square().sum()
        db, dlog = torch.autograd.grad(loss, (b, log_lam))
        return {"x": x.detach(), "loss": loss.detach(), "db": db, "dlog_lam": dlog}
    if kind not in ("solve", "host", "uq") or not stable(case):
        return None
    st = prepare(case, seed)
    g = geometry(*shape_of(case))
    b = torch.as_tensor(st["b"], dtype=f64, device="cuda")
    basis = reference_basis(reference_operator(g, values, f64), b, K)
    H, beta = basis["H"].cpu().numpy(), float(basis["beta"])
    per_k = range(1, K + 1) if st.get("histories") else [K]
    solved = [reference_projected(H[:k + 1, :k], beta, rule, g.m) for k in per_k]
    out = {"x": basis["L"] @ torch.from_numpy(solved[-1][0]).cuda(), "gp": None, "tp": None}
    if kind == "host":
        hist = st["histories"]
        out |= {"lam_hist": np.array([r[3] for r in solved]) if hist else None,
                "res_hist": np.array([r[4] for r in solved]) if hist else None, "k_done": None}
    if kind == "uq":
        out |= {"lam_hist": np.array([r[3] for r in solved]),
                "res_hist": np.array([r[4] for r in solved]), "var_diag": None, "var_sum": None}
    return out
