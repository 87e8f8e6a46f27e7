"""The work that the library's users have it do, as cases to measure.

Each case goes through the public entry points (the Python binding of the C
ABI): the fused product y = A x, d = Q^H y in its three forms, fixed numbers
of iterations of the unpreconditioned method, whole preconditioned solves
(natural-order and multicolour ILU(0), FP64 and FP32-refined, scalar and
3x3-block storage), and a batch of uneven systems.

What the outputs can be held to decides how a solve is cut off.  Without a
preconditioner the iterates of the log-normal systems depend on the order of
the sums after a few dozen iterations (a relative change of 1e-16 in b grows
to 1e-11 within 12 iterations and to order one within 40), so those solves
run a fixed 8 to 16 iterations: block 0 of the method and the blocks after
it, the same passes that a whole solve of thousands of iterations repeats.
The preconditioned solves run to their tolerance.

The matrices are those of paper_1106_3678_gb300.workloads; right-hand sides,
solutions and shadow vectors are drawn from the seed.
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_1106_3678_gb300 import mlbicgstab as M
from paper_1106_3678_gb300 import workloads as W

PRECOND = {"none": M.MLB_PRECOND_NONE, "jacobi": M.MLB_PRECOND_JACOBI, "ilu0": M.MLB_PRECOND_ILU0,
           "ilu0_mc": M.MLB_PRECOND_ILU0_MC}


def listed():
    return [
        # The smallest call: a 2-D system of 1,024 rows, one product whose
        # inner products come back to the host.  Latency alone.
        {"name": "product_2d_sync", "do": "product", "entry": "sync", "matrix": "cd2d", "m": 32, "n": 4,
         "dtype": "f64"},
        # The fused product of the 128^3 convection-diffusion system in FP64
        # with 4 shadow vectors, pipelined by its caller.
        {"name": "product_3d_f64", "do": "product", "entry": "async", "matrix": "lognormal", "m": 128, "sigma": 2.0,
         "n": 4, "dtype": "f64"},
        # The same on the FP32 copies of a refined handle, with 8 shadow
        # vectors: columns beyond those fused into the product's epilogue.
        {"name": "product_3d_f32_n8", "do": "product", "entry": "async", "matrix": "lognormal", "m": 128,
         "sigma": 2.0, "n": 8, "dtype": "f32"},
        # The allocation-free product on the caller's own CSR arrays, at a
        # size that no tile divides.
        {"name": "product_noalloc", "do": "product", "entry": "noalloc", "matrix": "lognormal", "m": 101,
         "sigma": 2.0, "n": 8, "dtype": "f64"},
        # A whole small solve from host arrays: the 32x32 system to 1e-10,
        # about a hundred iterations on one CTA.
        {"name": "solve_2d_small", "do": "converge", "matrix": "cd2d", "m": 32, "n": 4, "dtype": "f64",
         "precond": "none", "refined": False, "tol": 1e-10, "host": True, "iters": 104},
        # A system whose vectors stay in L2: the cost of a pass's
        # synchronisation shows.
        {"name": "solve_3d_64", "do": "iterate", "matrix": "lognormal", "m": 64, "sigma": 1.0, "n": 4,
         "dtype": "f64", "iters": 12},
        # The headline system: vectors stream from HBM.
        {"name": "solve_3d_128", "do": "iterate", "matrix": "lognormal", "m": 128, "sigma": 2.0, "n": 4,
         "dtype": "f64", "iters": 12},
        # The complex Helmholtz system with 8 shadow vectors.
        {"name": "solve_helmholtz_c128", "do": "iterate", "matrix": "helmholtz", "m": 128, "mz": 32, "n": 8,
         "dtype": "c128", "iters": 16},
        # Multicolour ILU(0), the fastest way to a solution of the 3-D system.
        {"name": "solve_ilu0_mc_96", "do": "converge", "matrix": "lognormal", "m": 96, "sigma": 2.0, "n": 4,
         "dtype": "f64", "precond": "ilu0_mc", "refined": False, "tol": 1e-12, "host": False, "iters": 200},
        # The paper's own preconditioner: natural-order ILU(0), one barrier
        # per wavefront of the triangular solves.
        {"name": "solve_ilu0_48", "do": "converge", "matrix": "lognormal", "m": 48, "sigma": 2.0, "n": 4,
         "dtype": "f64", "precond": "ilu0", "refined": False, "tol": 1e-12, "host": False, "iters": 65},
        # The 3x3-block reservoir system in FP32 inside FP64 refinement.
        {"name": "solve_reservoir_refined", "do": "converge", "matrix": "reservoir", "m": 64, "mz": 32, "n": 8,
         "dtype": "f64", "precond": "ilu0_mc", "refined": True, "tol": 1e-12, "host": False, "iters": 16},
        # Many systems of 1e3 to 1e5 rows in one launch.
        {"name": "batch_uneven", "do": "batch", "count": 96, "mat_seed": 5, "n_max": 1e5, "n": 4, "iters": 12},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    do = rng.choice(["product", "product", "iterate", "iterate", "converge", "batch"])
    n = rng.choice([1, 2, 3, 4, 4, 5, 8])
    if do == "product":
        entry = rng.choice(["sync", "async", "noalloc"])
        dtype = rng.choice(["f64", "f64", "c128"] if entry != "async" else ["f64", "f32", "c128"])
        n = rng.choice([1, 2, 3, 4, 8, 12, 16])
        if dtype == "c128":
            return {"do": do, "entry": entry, "matrix": "helmholtz", "m": _log_int(rng, 16, 120),
                    "mz": _log_int(rng, 8, 32), "n": n, "dtype": dtype}
        if rng.random() < 0.4:
            return {"do": do, "entry": entry, "matrix": "cd2d", "m": _log_int(rng, 24, 1000), "n": n, "dtype": dtype}
        return {"do": do, "entry": entry, "matrix": "lognormal", "m": _log_int(rng, 12, 120), "sigma": 2.0, "n": n,
                "dtype": dtype}
    if do == "iterate":
        if rng.random() < 0.25:
            return {"do": do, "matrix": "helmholtz", "m": _log_int(rng, 40, 128), "mz": _log_int(rng, 12, 32),
                    "n": rng.choice([4, 8]), "dtype": "c128", "iters": 12}
        return {"do": do, "matrix": "lognormal", "m": _log_int(rng, 32, 120), "sigma": 1.0, "n": n, "dtype": "f64",
                "iters": 12 if n > 2 else 7}
    if do == "converge":
        m = _log_int(rng, 14, 64)
        pc = rng.choice(["ilu0", "ilu0_mc", "ilu0_mc"])
        if pc == "ilu0":
            m = min(m, 40)
        return {"do": do, "matrix": "lognormal", "m": m, "sigma": 1.0, "n": n, "dtype": "f64", "precond": pc,
                "refined": rng.random() < 0.3, "tol": 1e-12, "host": rng.random() < 0.3,
                "iters": int((1.2 if pc == "ilu0" else 2.0) * m)}
    return {"do": do, "count": _log_int(rng, 8, 96), "mat_seed": rng.randrange(1 << 20),
            "n_max": float(_log_int(rng, 4000, 100000)), "n": rng.choice([1, 4, 4, 8]), "iters": 9}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=16)
def _built(kind, m, mz, sigma):
    if kind == "cd2d":
        return W.cd2d(m)
    if kind == "lognormal":
        return W.cd3d_lognormal(m, sigma=sigma)
    if kind == "reservoir":
        return W.reservoir_bsr3(m, m, mz)
    return W.helmholtz3d_c(m, m, mz)


def _matrix(case):
    return _built(case["matrix"], case["m"], case.get("mz", 0), case.get("sigma", 0.0))


@functools.lru_cache(maxsize=4)
def _systems(count, mat_seed, n_max):
    return [A for A, _ in W.batch_cd(count, seed=mat_seed, n_max=n_max)]


def _scalar_csr(A):
    """(row pointers, columns, values) of a CSR or BSR(3) matrix, scalar."""
    if A.val.ndim == 3:
        A = W.bsr3_to_csr(A)
    return A.row_ptr, A.col, A.val


def _on_gpu(A):
    rp, ci, v = _scalar_csr(A)
    return torch.sparse_csr_tensor(torch.from_numpy(rp).cuda(), torch.from_numpy(ci.astype(np.int64)).cuda(),
                                   torch.from_numpy(v).cuda(), size=(A.n_rows, A.n_rows))


@functools.lru_cache(maxsize=2)
def _on_gpu_built(kind, m, mz, sigma):
    return _on_gpu(_built(kind, m, mz, sigma))


def _operator(case):
    return _on_gpu_built(case["matrix"], case["m"], case.get("mz", 0), case.get("sigma", 0.0))


def _random(N, cols, cplx, seed, normal):
    """`cols` columns of N random values on the GPU, one after another:
    N(0, 1) or U[-1, 1] (real and imaginary parts)."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    shape = (cols, N, 2) if cplx else (cols, N)
    t = torch.randn(shape, dtype=torch.float64, device="cuda", generator=g) if normal else \
        torch.rand(shape, dtype=torch.float64, device="cuda", generator=g) * 2.0 - 1.0
    return torch.view_as_complex(t) if cplx else t


def _shadow(N, n, cplx, seed):
    """Q ~ N(0, 1), as rows on the GPU."""
    return _random(N, n, cplx, 4 * seed + 1, True)


def _handle(A, Q, **opt):
    return M.mlbicgstab_create(A, n=int(Q.shape[0]), Q=Q.cpu().numpy().T, **opt)


def prepare(case, seed):
    if case["do"] == "batch":
        systems = _systems(case["count"], case["mat_seed"], case["n_max"])
        sizes = [A.n_rows for A in systems]
        b = _random(sum(sizes), 1, False, 4 * seed, False)[0]
        x = torch.zeros_like(b)
        hs = [_handle(A, _shadow(A.n_rows, case["n"], False, 1000 * seed + s)) for s, A in enumerate(systems)]
        return {"case": case, "hs": hs, "b": list(b.split(sizes)), "x": x, "xs": list(x.split(sizes)),
                "tols": [0.0] * len(hs), "maxits": [case["iters"]] * len(hs)}
    A = _matrix(case)
    N, n, cplx = A.n_rows, case["n"], case["dtype"] == "c128"
    Q = _shadow(N, n, cplx, seed)
    v = _random(N, 1, cplx, 4 * seed, case["do"] == "product")[0]
    if case["do"] == "product":
        if case["dtype"] == "f32":
            v = v.float()
        y = torch.empty_like(v)
        st = {"case": case, "x": v, "y": y}
        if case["entry"] == "noalloc":
            st["csr"] = [torch.from_numpy(a).cuda() for a in (A.row_ptr, A.col, A.val)]
            st["Q"] = Q
            st["d"] = torch.empty(n, dtype=v.dtype, device="cuda")
        else:
            st["h"] = _handle(A, Q, precision=M.MLB_PREC_FP32_REFINED if case["dtype"] == "f32" else M.MLB_PREC_FP64)
            st["d"] = torch.empty(n * (2 if cplx else 1) + 1, dtype=torch.float64, device="cuda")
        return st
    if case["do"] == "iterate":
        h = _handle(A, Q)
        return {"case": case, "h": h, "b": v, "x": torch.zeros_like(v)}
    # a whole solve: b = A x* for a random x*
    b = _operator(case) @ v
    h = _handle(A, Q, precond=PRECOND[case["precond"]],
                precision=M.MLB_PREC_FP32_REFINED if case["refined"] else M.MLB_PREC_FP64)
    x = torch.zeros_like(b)
    if case["host"]:
        b, x = b.cpu().numpy(), x.cpu().numpy()
    return {"case": case, "h": h, "b": b, "x": x}


def run(state):
    case = state["case"]
    if case["do"] == "product":
        x, y = state["x"], state["y"]
        if case["entry"] == "sync":
            return {"y": y, "d": M.mlbicgstab_spmv_qdot(state["h"], x, y)}
        d = state["d"]
        if case["entry"] == "noalloc":
            M.mlbicgstab_spmv_qdot_noalloc(*state["csr"], x, state["Q"], y, d)
            return {"y": y, "d": d}
        M.mlbicgstab_spmv_qdot_async(state["h"], x, y, d)
        # sums of FP32 products, kept no wider than their inputs
        return {"y": y, "d": d.to(x.dtype) if x.dtype == torch.float32 else d}
    x = state["x"]
    if isinstance(x, np.ndarray):
        x[:] = 0.0
    else:
        x.zero_()
    if case["do"] == "batch":
        res = M.mlbicgstab_solve_batch(state["hs"], state["b"], state["xs"], state["tols"], state["maxits"])
        return {"x": x, "iter": np.array([r.iter for r in res])}
    if case["do"] == "iterate":
        res, _ = M.mlbicgstab_solve(state["h"], state["b"], x, 0.0, case["iters"])
        return {"x": x, "iter": int(res.iter)}
    res, _ = M.mlbicgstab_solve(state["h"], state["b"], x, case["tol"], 20000)
    return {"x": x, "flag": int(res.flag)}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _iteration_work(N, nnz, entry_bytes, vs, n, iters, cplx, ilu, resident):
    """Bytes and operations of `iters` iterations (Algorithm 7.1).  Per block
    of n iterations: n + 1 products; n updates of x and r; the sweeps, whose
    step i reads the columns i.. of w and g of the last block and ..i of g
    of this one and writes two; one omega step.  Every vector of a step
    counts once.  A system whose matrix and vectors fit in L2 (resident)
    moves them from HBM once for all iterations."""
    k = iters / n
    product = nnz * entry_bytes + 3 * N * vs
    sweeps = sum((3 + 2 * (n - i)) + (i if i else 0) + (n - i) + (i if i else 0) for i in range(n))
    vectors = k * (n * 7 + 6 + sweeps) * N * vs
    flops = k * ((n + 1) * 2 * nnz + (n * 8 + 8 + sum(2 * (3 * (n - i) + 2 * i + 2) for i in range(n))) * N)
    bytes_ = k * (n + 1) * product + vectors
    if ilu:
        bytes_ += k * (n + 1) * (nnz * 12 + 3 * N * vs)
        flops += k * (n + 1) * 2 * nnz
    if resident:
        bytes_ = nnz * entry_bytes * (2 if ilu else 1) + (4 * n + 4) * N * vs
    return bytes_, flops * (4 if cplx else 1)


def work(case):
    if case["do"] == "batch":
        by = fl = 0.0
        for A in _systems(case["count"], case["mat_seed"], case["n_max"]):
            # all systems' matrices and vectors exceed L2 from about 8 large ones on
            b, f = _iteration_work(A.n_rows, A.nnz, 12, 8, case["n"], case["iters"], False, False,
                                   case["count"] * case["n_max"] < 1e6)
            by, fl = by + b, fl + f
        return {"bytes": by, "flops": fl}
    A = _matrix(case)
    N, n, cplx = A.n_rows, case["n"], case["dtype"] == "c128"
    nnz = A.nnz
    vs = {"f64": 8, "f32": 4, "c128": 16}[case["dtype"]]
    if case["do"] == "product":
        rp = 8 * N if case["entry"] == "noalloc" else N // 4
        return {"bytes": nnz * (vs + 4) + rp + (2 + n) * N * vs,
                "flops": (2 * nnz + 2 * n * N) * (4 if cplx else 1)}
    blocked = case["matrix"] == "reservoir"
    if case.get("refined"):
        vs = 4
    entry = vs + 4 / 3 if blocked else vs + 4
    resident = nnz * entry + (4 * n + 4) * N * vs < 100e6
    by, fl = _iteration_work(N, nnz, entry, vs, n, case["iters"], cplx,
                             case.get("precond", "none").startswith("ilu0"), resident)
    return {"bytes": by, "flops": fl}


# ---------------------------------------------------------------------------
# the same results in 64 bits, in plain torch
# ---------------------------------------------------------------------------

def _adjoint(A):
    return A.to_sparse_coo().transpose(0, 1).conj().resolve_conj().coalesce().to_sparse_csr()


def _method(A, b, q, iters):
    """x after `iters` iterations of Algorithm 7.1 with M = I from x = 0;
    q: the shadow vectors as rows."""
    n = q.shape[0]
    AH = _adjoint(A)
    f = [AH @ q[s] for s in range(n - 1)]
    dot = torch.vdot
    x, r = torch.zeros_like(b), b.clone()
    g, w, c = [None] * n, [None] * n, [None] * n
    g[0] = r.clone()
    w[0] = A @ g[0]
    c[0] = dot(q[0], w[0])
    e = dot(q[0], r)
    done, first, omega = 0, True, None
    while True:
        for i in range(1, n):
            alpha = e / c[i - 1]
            x, r = x + alpha * g[i - 1], r - alpha * w[i - 1]
            done += 1
            if done == iters:
                return x
            e = dot(q[i], r)
            if first:
                new = r + (-(dot(f[0], r) / c[0])) * g[0]
                start = 1
            else:
                beta = -(e / c[i])
                zw, zg = r + beta * w[i], beta * g[i]
                for s in range(i + 1, n):
                    beta = -(dot(q[s], zw) / c[s])
                    zw, zg = zw + beta * w[s], zg + beta * g[s]
                new = zw - zg / omega
                start = 0
            for s in range(start, i):
                new = new + (-(dot(f[s], new) / c[s])) * g[s]
            g[i] = new
            w[i] = A @ new
            c[i] = dot(q[i], w[i])
        alpha = e / c[n - 1]
        x, u = x + alpha * g[n - 1], r - alpha * w[n - 1]
        z = A @ u
        omega = dot(z, u) / dot(z, z).real
        x, r = x + omega * u, u - omega * z
        done += 1
        if done == iters:
            return x
        e = dot(q[0], r)
        beta = -(e / c[0])
        zw, zg = r + beta * w[0], beta * g[0]
        for s in range(1, n):
            beta = -(dot(q[s], zw) / c[s])
            zw, zg = zw + beta * w[s], zg + beta * g[s]
        g[0] = zw - zg / omega
        w[0] = A @ g[0]
        c[0] = dot(q[0], w[0])
        first = False


def exact(case, seed):
    if case["do"] == "batch":
        systems = _systems(case["count"], case["mat_seed"], case["n_max"])
        sizes = [A.n_rows for A in systems]
        b = _random(sum(sizes), 1, False, 4 * seed, False)[0].split(sizes)
        xs = [_method(_on_gpu(A), b[s], _shadow(A.n_rows, case["n"], False, 1000 * seed + s), case["iters"])
              for s, A in enumerate(systems)]
        return {"x": torch.cat(xs), "iter": None}
    A = _matrix(case)
    N, n, cplx = A.n_rows, case["n"], case["dtype"] == "c128"
    v = _random(N, 1, cplx, 4 * seed, case["do"] == "product")[0]
    if case["do"] == "converge":
        return {"x": v.cpu().numpy() if case["host"] else v, "flag": None}
    Q = _shadow(N, n, cplx, seed)
    if case["do"] == "iterate":
        return {"x": _method(_operator(case), v, Q, case["iters"]), "iter": None}
    A = _operator(case)
    if case["dtype"] == "f32":
        v, Q = v.float().double(), Q.float().double()
        A = torch.sparse_csr_tensor(A.crow_indices(), A.col_indices(), A.values().float().double(), size=A.shape)
    y = A @ v
    d = torch.stack([torch.vdot(q, y) for q in Q])
    if case["entry"] == "async":   # real parts and imaginary parts in turn, then the status word
        d = torch.view_as_real(d).reshape(-1) if cplx else d
        d = torch.cat([d, d.new_zeros(1)])
    elif case["entry"] == "sync":
        d = d.cpu().numpy()
    return {"y": y, "d": d}
