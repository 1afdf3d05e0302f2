"""The performance cases of the rpCholesky-QR library: what its users have it factor, from the smallest
call to the largest, in every mode, through the public entry points of ``paper_2406_11751_gb300``.

A case is one factorisation (or one batch) with its plan and output buffers in hand, as a Krylov or
LOBPCG program holds them: the plan, Q, R and info live across calls, the matrix changes.  Matrices are
A = G diag(sigma) V^T with G an m x n Gaussian matrix scaled by 1/sqrt(m) (orthonormal up to a factor
(1 +- sqrt(n/m)), so incoherent), V a random orthogonal matrix and sigma log-spaced from 1 to 1/kappa.
Q is determined by A only up to about eps * kappa, so kappa stays at 1e5 in FP64 and at 10 in FP32:
beyond that, two correct programs give different digits.  No kernel's work depends on kappa.
"""
import math

import torch

import paper_2406_11751_gb300 as rq

_MODES = {"fp64": rq.FP64, "split": rq.SPLIT64, "fp32": rq.FP32}
_SMOOTH = {"none": rq.SMOOTH_NONE, "wht": rq.SMOOTH_WHT, "dct": rq.SMOOTH_DCT}


def _factor(mode, m, n, c=3, pad=0, smooth="none", host=False, **more):
    """One matrix, s = c n sampled rows, leading dimensions n + pad."""
    return dict(more, kind="factor", mode=mode, m=m, n=n, s=c * n, pad=pad, smooth=smooth, host=host)


def _batch(mode, count, m_max, pick, **more):
    """`count` matrices of uneven size: m log-uniform in [4096, m_max], n from {8, 16, 32, 64, 128}."""
    return dict(more, kind="batch", mode=mode, count=count, m_max=m_max, pick=pick)


def listed():
    return [
        # the documented first example: one small block, all latency
        _factor("fp64", 10000, 50, name="fp64 10000x50"),
        # the standard tall block of the library's benchmark, in plain FP64
        _factor("fp64", 1 << 20, 128, name="fp64 1048576x128"),
        # a wide block of odd size in plain FP64 (blocked solves, separate Gram matrix)
        _factor("fp64", 200003, 300, name="fp64 200003x300"),
        # the size of the paper's experiments with the split mode: a small block again
        _factor("split", 6000, 100, name="split 6000x100"),
        # the standard tall block in the split (tensor-core) mode, the one a user of large blocks picks
        _factor("split", 1 << 20, 128, name="split 1048576x128"),
        # an odd row count, a width between two paddings, a leading dimension wider than the block
        _factor("split", 400009, 200, pad=3, name="split 400009x200"),
        # the large single-GPU problem: rows cut so that several fit the device
        _factor("split", 1 << 21, 512, name="split 2097152x512"),
        # the widest figures of the paper: few rows, many columns, so the small factors carry the cost
        _factor("split", 6000, 1000, name="split 6000x1000"),
        # single-precision Krylov users
        _factor("fp32", 1 << 20, 128, name="fp32 1048576x128"),
        # blocks of uneven size from a block-Krylov solver, one persistent launch
        _batch("fp64", 32, 1 << 20, 17, name="batch fp64 32"),
        # coherent or unknown inputs: rows are mixed before sampling
        _factor("split", 1 << 18, 100, smooth="wht", name="smoothed 262144x100"),
        # a matrix that lives in host memory, copied in and out around the factorisation
        _factor("split", 1 << 19, 96, host=True, name="host 524288x96"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: every mode, sizes over the logarithm of their range, odd ones included."""
    what = rng.choice(["fp64", "fp64", "split", "split", "split", "fp32", "fp32", "batch", "smooth", "host"])
    if what == "batch":
        return _batch(rng.choice(["fp64", "split"]), rng.randint(8, 32), _log(rng, 1 << 15, 1 << 18),
                      rng.randrange(1 << 20))
    n_max, cost = {"fp64": (512, 5e10), "split": (1024, 1.5e12), "fp32": (512, 5e11), "smooth": (128, 3e10),
                   "host": (128, 3e10)}[what]
    while True:
        n = _log(rng, 8, n_max)
        m = _log(rng, 4096, 1 << 20)
        c = rng.choice([3, 3, 3, 10])
        if m >= 2 * c * n and 3.0 * m * n * n <= cost:
            break
    if what == "host":
        return _factor("split", m, n, c, host=True)
    if what == "smooth":
        return _factor(rng.choice(["fp64", "split"]), m, n, c, smooth=rng.choice(["wht", "dct"]))
    return _factor(what, m, n, c, pad=rng.choice([0, 0, 1, 4, 24]))


def _sizes(case):
    """(m, n, s) of every matrix of a case."""
    if case["kind"] == "factor":
        return [(case["m"], case["n"], case["s"])]
    g = torch.Generator().manual_seed(case["pick"])
    out = []
    for _ in range(case["count"]):
        u = float(torch.rand((), generator=g, dtype=torch.float64))
        n = (8, 16, 32, 64, 128)[int(torch.randint(5, (), generator=g))]
        out.append((int(4096 * (case["m_max"] / 4096) ** u), n, 3 * n))
    return out


def _matrix(m, n, gen, dtype):
    """A = G diag(sigma) V^T on the GPU."""
    kappa = 10.0 if dtype == torch.float32 else 1e5
    g = torch.randn((m, n), generator=gen, dtype=dtype, device="cuda").mul_(1.0 / math.sqrt(m))
    v, _ = torch.linalg.qr(torch.randn((n, n), generator=gen, dtype=torch.float64, device="cuda"))
    sigma = kappa ** -(torch.arange(n, dtype=torch.float64, device="cuda") / max(1, n - 1))
    return g @ (sigma[:, None] * v.T).to(dtype)


def _inputs(case, seed):
    """The matrices of a case, from the seed alone."""
    gen = torch.Generator(device="cuda").manual_seed(seed)
    dtype = torch.float32 if case["mode"] == "fp32" else torch.float64
    return [_matrix(m, n, gen, dtype) for m, n, _ in _sizes(case)]


def _padded(a, pad):
    """The same matrix with a leading dimension `pad` wider, as a block of a larger array."""
    if not pad:
        return a
    wide = torch.zeros((a.shape[0], a.shape[1] + pad), dtype=a.dtype, device=a.device)
    wide[:, :a.shape[1]] = a
    return wide[:, :a.shape[1]]


def _views(sizes):
    """One buffer cut into the matrices of a batch: (buffer, views)."""
    flat = torch.zeros(sum(r * c for r, c in sizes), dtype=torch.float64, device="cuda")
    views, at = [], 0
    for r, c in sizes:
        views.append(flat[at:at + r * c].view(r, c))
        at += r * c
    return flat, views


def prepare(case, seed):
    mode, sizes, As = _MODES[case["mode"]], _sizes(case), _inputs(case, seed)
    max_m, max_n, max_s = (max(x[i] for x in sizes) for i in range(3))
    st = {"case": case, "seed": seed}
    if case["kind"] == "batch":
        st["ss"] = [s for _, _, s in sizes]
        st["seeds"] = [seed + i for i in range(len(sizes))]
        st["Q"], st["Qs"] = _views([(m, n) for m, n, _ in sizes])
        st["R"], st["Rs"] = _views([(n, n) for _, n, _ in sizes])
        st["As"] = As
        st["info"] = torch.zeros(2 * len(sizes), dtype=torch.int32, device="cuda")
        if mode == rq.FP64:
            st["plan"] = rq.rpcholqr_plan_create(0, max_m, max_n, max_s, mode=mode)
            rq.rpcholqr_plan_set_option(st["plan"], rq.OPT_BATCH_CAPACITY, len(sizes))
            st["arrays"] = rq.BatchArrays(As, st["ss"], st["seeds"], st["Qs"], st["Rs"])
        else:
            # the slot plans of the batch, its work captured once and replayed per step
            st["batch"] = rq.rpcholqr_batch_create(0, max_m, max_n, max_s, slots=4, mode=mode)
            stream = torch.cuda.Stream()
            stream.wait_stream(torch.cuda.current_stream())
            with torch.cuda.stream(stream):
                rq.rpcholqr_batch_capture(st["batch"], As, st["ss"], st["seeds"], st["Qs"], st["Rs"], st["info"],
                                          stream=stream)
            torch.cuda.current_stream().wait_stream(stream)
        return st
    m, n, s = sizes[0]
    dtype = As[0].dtype
    st["plan"] = rq.rpcholqr_plan_create(0, max_m, max_n, max_s, mode=mode)
    if case["smooth"] != "none":
        rq.rpcholqr_plan_set_smoothing(st["plan"], _SMOOTH[case["smooth"]])
    if case["host"]:
        st["A"] = torch.empty((m, n), dtype=dtype, pin_memory=True)
        st["A"].copy_(As[0])
        st["Q"] = torch.empty((m, n), dtype=dtype, pin_memory=True)
        st["R"] = torch.empty((n, n), dtype=dtype, pin_memory=True)
    else:
        st["A"] = _padded(As[0], case["pad"])
        st["Q"] = torch.zeros((m, n + case["pad"]), dtype=dtype, device="cuda")[:, :n]
        st["R"] = torch.zeros((n, n), dtype=dtype, device="cuda")
        st["info"] = torch.zeros(2, dtype=torch.int32, device="cuda")
    return st


def run(st):
    case = st["case"]
    if case["kind"] == "batch":
        if "plan" in st:
            rq.rpcholqr_factor_batched(st["plan"], st["As"], st["ss"], st["seeds"], st["Qs"], st["Rs"], st["info"],
                                       arrays=st["arrays"])
        else:
            rq.rpcholqr_batch_replay(st["batch"])
        return {"Q": st["Q"], "R": st["R"], "info": st["info"]}
    if case["host"]:
        Q, R, status, pivot = rq.rpcholqr_factor_host(st["plan"], st["A"], case["s"], st["seed"], st["Q"], st["R"])
        return {"Q": Q, "R": R, "info": [status, pivot]}
    call = rq.rpcholqr_factor_f32 if case["mode"] == "fp32" else rq.rpcholqr_factor
    Q, R, info = call(st["plan"], st["A"], case["s"], st["seed"], st["Q"], st["R"], st["info"])
    return {"Q": Q, "R": R, "info": info}


def work(case):
    """A read and Q written once; the method's operations, 3 m n^2 for the passes over the rows (row solve,
    Gram matrix, row solve), 2 s n^2 - 2 n^3 / 3 for the sample's QR, n^3 / 3 each for Cholesky and R1 Rs."""
    size = 4 if case["mode"] == "fp32" else 8
    total = {"bytes": 0.0, "flops": 0.0}
    for m, n, s in _sizes(case):
        total["bytes"] += size * (2.0 * m * n + n * n)
        total["flops"] += 3.0 * m * n * n + 2.0 * s * n * n
    return total


def _thin_qr(a):
    """The thin QR factors with a positive diagonal, in FP64: Cholesky-QR three times (kappa is at most 1e5)."""
    q, r = a, None
    for _ in range(3):
        ri = torch.linalg.cholesky(q.T @ q).T
        q = torch.linalg.solve_triangular(ri, q, upper=True, left=False)
        r = ri if r is None else ri @ r
    return q, torch.triu(r)


def exact(case, seed):
    out = [_thin_qr(a.double()) for a in _inputs(case, seed)]
    if case["kind"] == "batch":
        return {"Q": torch.cat([q.reshape(-1) for q, _ in out]), "R": torch.cat([r.reshape(-1) for _, r in out]),
                "info": None}
    return {"Q": out[0][0], "R": out[0][1], "info": [None, None] if case["host"] else None}
