"""The work that a user of this framework has it do, as cases that can be measured.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes
what a program has in hand before the call (matrices, right-hand sides, the handle it keeps),
``run`` is one pass through the public entry points, ``work`` counts what the path cannot do
without, and ``exact`` gives the outputs in float64 by plain torch: a Householder QR of A^*
and three refinement passes whose residuals are summed from exact products of short pieces.

Kinds of case:
  step    a new preconditioner (sketch, pivoted QR, Gram, factors) and one apply with it
  apply   one apply with a preconditioner that is kept
  ipm     one iteration of an interior-point loop: new column scalings, then a step
  layer   the projection as a differentiable layer: a new A, forward and backward
  batch   many small instances of uneven sizes, one step of all of them by graph replay
  sparse  a sparse (optionally plus low rank) A: a step, or an apply with what is kept
"""
import math

import numpy as np
import torch

import workloads
from paper_0912_1135_gb300 import Projector, SparseProjector
from paper_0912_1135_gb300.autograd import null_project
from paper_0912_1135_gb300.batch import Batch

DEV = "cuda:0"

# What a program sets beyond the defaults at kappa = 1e12 (bench.py's options of that workload).
SCALE_OPTS = dict(sketch_slices=6, resid_slices=10, refine_passes=4, refine_tol=1e-11, rank_tol=1e-14)


def listed():
    return [
        # the smallest step: the repository's small dense configuration (launches and latency count)
        dict(name="step_64x2048", kind="step", m=64, n=2048, l=256, k=16, kappa=1e8, dtype="f64", omega="gaussian",
             mode="mixed", out="null"),
        # the smallest call: one right-hand side through a small kept preconditioner
        dict(name="apply_64x2048_k1", kind="apply", m=64, n=2048, l=256, k=1, kappa=1e8, dtype="f64",
             omega="gaussian", mode="mixed", out="null"),
        # ragged sizes, float32 data, uniform variates, all three outputs
        dict(name="step_333x12345", kind="step", m=333, n=12345, l=698, k=7, kappa=1e4, dtype="f32",
             omega="uniform", mode="mixed", out="all"),
        # the headline configuration: a new preconditioner for every block of right-hand sides
        dict(name="step_512x65536", kind="step", m=512, n=65536, l=516, k=64, kappa=1e10, dtype="f64",
             omega="gaussian", mode="mixed", out="null"),
        # the headline configuration with the preconditioner kept: projection and least squares
        dict(name="apply_512x65536_k64", kind="apply", m=512, n=65536, l=516, k=64, kappa=1e10, dtype="f64",
             omega="gaussian", mode="mixed", out="all"),
        # precision at scale: the largest dense configuration, 256 right-hand sides
        dict(name="step_2048x262144", kind="step", m=2048, n=262144, l=4128, k=256, kappa=1e12, dtype="f64",
             omega="gaussian", mode="scale", out="null"),
        # the plain float64 form, which a user picks for well-conditioned problems
        dict(name="step_fp64_256x8192", kind="step", m=256, n=8192, l=544, k=32, kappa=1e4, dtype="f64",
             omega="gaussian", mode="fp64", out="null"),
        # one interior-point iteration (the batching study's sizes)
        dict(name="ipm_1024x32768", kind="ipm", m=1024, n=32768, l=2080, k=32, kappa=1e8),
        # a projection layer's training step: float32, a batch of 4096, gradients of A and B
        dict(name="layer_256x8192_b4096", kind="layer", m=256, n=8192, l=1024, k=4096, kappa=1e6),
        # uneven small instances, replayed as one graph (an eighth of the batching study's count)
        dict(name="batch_64", kind="batch", count=64, sizes_seed=999, m_lo=16, m_hi=512, k=32),
        # the paper's own setting: Eq. 21's sparse matrix plus Eq. 22's rank-10 term, a step
        # and one vector
        dict(name="sparse_step_1000x300000", kind="sparse", keep=False, family="paper", m=1000, n=300000, l=1004,
             k=1, r=10, kappa=1e8, passes=2),
        # an irregular sparse matrix, kept preconditioner, a hundred vectors
        dict(name="sparse_apply_1000x300000", kind="sparse", keep=True, family="random", m=1000, n=300000, l=1004,
             k=100, r=0, kappa=1e3, passes=2),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "apply", "apply", "ipm", "layer", "batch", "sparse", "sparse"])
    if kind in ("step", "apply"):
        mode = rng.choice(["mixed"] * 5 + ["fp64"])
        m = int(_log(rng, 24, 700 if mode == "mixed" else 300))
        n = int(min(m * _log(rng, 4, 128), 2.0 ** (25.5 if mode == "mixed" else 22) / m))
        n = max(n, 4 * m)
        l = min(n, rng.choice([m + 4, 2 * m + 32, 4 * m]))
        dtype = rng.choice(["f64", "f64", "f32"])
        top = 4 if dtype == "f32" or mode == "fp64" else 9
        return dict(kind=kind, m=m, n=n, l=l, k=int(_log(rng, 1, 257)), kappa=float("%.2g" % 10 ** rng.uniform(1, top)),
                    dtype=dtype, omega=rng.choice(["gaussian", "gaussian", "uniform", "rademacher"]), mode=mode,
                    out=rng.choice(["null", "null", "row", "all"]))
    if kind == "ipm":
        m = int(_log(rng, 100, 1024))
        n = m * rng.randint(8, 32) + rng.randint(0, 63)
        return dict(kind=kind, m=m, n=n, l=2 * m + 32, k=int(_log(rng, 4, 65)), kappa=float("%.2g" % 10 ** rng.uniform(3, 8)))
    if kind == "layer":
        m = int(_log(rng, 32, 257))
        n = m * rng.randint(8, 32) + rng.randint(0, 31)
        return dict(kind=kind, m=m, n=n, l=4 * m, k=int(_log(rng, 64, 4097)), kappa=float("%.2g" % 10 ** rng.uniform(2, 6)))
    if kind == "batch":
        return dict(kind=kind, count=rng.randint(8, 64), sizes_seed=rng.randint(0, 9999), m_lo=16, m_hi=int(_log(rng, 64, 513)), k=int(_log(rng, 1, 33)))
    m = int(_log(rng, 40, 1100))
    n = m * max(3, int(_log(rng, 3000, 300000) / m))
    family = rng.choice(["paper", "random"])
    return dict(kind="sparse", keep=rng.random() < 0.5, family=family, m=m, n=n, l=m + 4, k=int(_log(rng, 1, 101)),
                r=rng.choice([0, 0, 10]), kappa=float("%.2g" % 10 ** rng.uniform(2, 8 if family == "paper" else 3)),
                passes=rng.randint(1, 3))


# -- inputs --------------------------------------------------------------------------------

def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _normal(g, *shape, dtype=torch.float64):
    return torch.randn(*shape, generator=g, device=DEV, dtype=dtype)


def _dense(g, m, n, kappa, dtype=torch.float64):
    """A = U diag(sigma) N / sqrt(n): U orthogonal, sigma log-spaced over [1 / kappa, 1], N standard
    normal, so that kappa(A) is kappa to a small factor when n is well above m."""
    u = torch.linalg.qr(_normal(g, m, m))[0]
    sigma = torch.logspace(0, -math.log10(kappa), m, device=DEV, dtype=torch.float64)
    return ((u * (sigma / math.sqrt(n))) @ _normal(g, m, n)).to(dtype)


def _instances(case):
    """The batching study's sizes: m log-uniform, n / m log-uniform over [4, 64]."""
    rng = np.random.default_rng(case["sizes_seed"])
    sizes = []
    for _ in range(case["count"]):
        m = int(round(np.exp(rng.uniform(np.log(case["m_lo"]), np.log(case["m_hi"])))))
        n = int(round(m * np.exp(rng.uniform(np.log(4), np.log(64)))))
        sizes.append((m, max(2 * m + 32, (n + 15) // 16 * 16)))
    return sizes


def _sparse(case, seed):
    """Compressed sparse rows (and the low-rank factors) on the device."""
    m, n, r = case["m"], case["n"], case["r"]
    if case["family"] == "paper":
        row_ptr, col, val, _, _, _ = workloads.paper_test_csr(m, n, case["kappa"], seed)
    else:
        # two to eight entries a column, more of them in the first rows, rows of different scales
        rng = np.random.default_rng(seed)
        per = rng.integers(2, 9, n)
        col = np.repeat(np.arange(n, dtype=np.int32), per)
        row = np.minimum((m * rng.random(col.size) ** 2).astype(np.int64), m - 1)
        row[np.cumsum(per) - per] = np.arange(n) % m          # no row is empty
        order = np.argsort(row, kind="stable")
        row, col = row[order], col[order]
        scale = case["kappa"] ** -rng.random(m)
        val = rng.standard_normal(col.size) * scale[row]
        row_ptr = np.concatenate([[0], np.cumsum(np.bincount(row, minlength=m))]).astype(np.int64)
    U = V = None
    if r:
        g = _generator(seed + 1)
        U, V = _normal(g, m, r) / math.sqrt(m * n), _normal(g, r, n)
    return torch.from_numpy(row_ptr).to(DEV), torch.from_numpy(col).to(DEV), torch.from_numpy(val).to(DEV), U, V


def _inputs(case, seed):
    g = _generator(seed)
    kind, dtype = case["kind"], torch.float32 if case.get("dtype") == "f32" else torch.float64
    if kind == "batch":
        sizes = _instances(case)
        return {"As": [_dense(g, m, n, 1e4, torch.float32) for m, n in sizes],
                "Bs": [_normal(g, case["k"], n, dtype=torch.float32) for _, n in sizes]}
    if kind == "sparse":
        return {"A": _sparse(case, seed), "B": _normal(g, case["k"], case["n"])}
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "layer":
        return {"A": _dense(g, m, n, case["kappa"], torch.float32), "B": _normal(g, k, n, dtype=torch.float32),
                "G": _normal(g, k, n, dtype=torch.float32)}
    x = {"A": _dense(g, m, n, case["kappa"], dtype), "B": _normal(g, k, n, dtype=dtype)}
    if kind == "ipm":
        x["d"] = 10.0 ** (12.0 * torch.rand(n, generator=g, device=DEV, dtype=torch.float64) - 6.0)
    return x


def prepare(case, seed):
    x = _inputs(case, seed)
    s = {"case": case, "seed": seed, **x}
    kind = case["kind"]
    if kind in ("step", "apply"):
        opts = dict(mode="fp64") if case["mode"] == "fp64" else SCALE_OPTS if case["mode"] == "scale" else {}
        s["P"] = Projector(x["A"], l_max=case["l"], k_max=case["k"], omega=case["omega"], **opts)
        if kind == "apply":
            s["P"].precondition(seed, case["l"])
    elif kind == "ipm":
        s["P"] = Projector(x["A"], l_max=case["l"], k_max=case["k"], scalable=1, refine_passes=3, refine_tol=1e-12)
    elif kind == "layer":
        x["A"].requires_grad_(True)
        x["B"].requires_grad_(True)
    elif kind == "batch":
        sizes = [tuple(A.shape) for A in x["As"]]
        s["Zs"] = [torch.empty_like(B) for B in x["Bs"]]
        s["batch"] = Batch(x["As"], [case["k"]] * len(sizes), [2 * m + 32 for m, _ in sizes])
        s["batch"].capture(x["Bs"], [seed + i for i in range(len(sizes))], s["Zs"])
    else:
        row_ptr, col, val, U, V = x["A"]
        s["P"] = SparseProjector(row_ptr, col, val, case["n"], U=U, V=V, l_max=case["l"], k_max=case["k"],
                                 refine_passes=case["passes"])
        if case["keep"]:
            s["P"].precondition(seed, case["l"])
    return s


def run(s):
    case, kind = s["case"], s["case"]["kind"]
    if kind == "batch":
        s["batch"].replay()
        return s["Zs"]
    if kind == "layer":
        Z = null_project(s["A"], s["B"], seed=s["seed"], l=case["l"])
        dA, dB = torch.autograd.grad(Z, (s["A"], s["B"]), s["G"])
        return [Z.detach(), dA, dB]
    P = s["P"]
    if kind == "ipm":
        P.set_scaling(s["d"])
    if kind in ("step", "ipm") or (kind == "sparse" and not case["keep"]):
        P.precondition(s["seed"], case["l"])
    out = case.get("out", "null")
    Z, row, h = P.project(s["B"], null=out != "row", row=out != "null", lstsq=out == "all")
    return [t for t in (Z, row, h) if t is not None]


# -- what the path cannot do without -------------------------------------------------------

def work(case):
    kind = case["kind"]
    if kind == "batch":
        k, total = case["k"], {"bytes": 0.0, "flops": 0.0}
        for m, n in _instances(case):
            total["bytes"] += 4.0 * (m * n + 2 * k * n)
            total["flops"] += _build_flops(m, n, 2 * m + 32, m * n) + 8.0 * m * n * k
        return total
    m, n, l, k = case["m"], case["n"], case["l"], case["k"]
    e = 4 if kind == "layer" or case.get("dtype") == "f32" else 8
    outs = {"null": n, "row": n, "all": 2 * n + m}[case.get("out", "null")]
    if kind == "sparse":
        nnz = 5 * n
        build = 0.0 if case["keep"] else _build_flops(m, n, l, nnz)
        return {"bytes": 12.0 * nnz + 8.0 * (m + n) * case["r"] + 8.0 * k * (n + outs),
                "flops": build + (2 + 2 * case["passes"]) * 2.0 * k * (nnz + case["r"] * (m + n))}
    if kind == "layer":   # forward, the upstream gradient's apply, and dA = -(H^* Y + W^* Z)
        return {"bytes": 4.0 * (2 * m * n + 4 * k * n),
                "flops": _build_flops(m, n, l, m * n) + 16.0 * m * n * k + 4.0 * m * n * k}
    # c = A b, A^* h and one refinement pass (two more products) at two flops an entry
    return {"bytes": float(e) * (m * n + k * (n + outs)),
            "flops": (0.0 if kind == "apply" else _build_flops(m, n, l, m * n)) + 8.0 * m * n * k}


def _build_flops(m, n, l, nnz):
    """The sketch, the pivoted QR, the Gram matrix (a triangle of A A^*) and the Cholesky factor."""
    return 2.0 * nnz * l + 2.0 * l * m * m - 2.0 * m ** 3 / 3 + float(nnz) * m + m ** 3 / 3.0


# -- the same outputs in float64, by plain torch -------------------------------------------

def _pieces(x, bits, count):
    """x (rows x cols) as a sum of `count` matrices whose entries are `bits`-bit multiples of a power
    of two, one power per row and piece."""
    top = 2.0 ** torch.ceil(torch.log2(x.abs().amax(1, keepdim=True).clamp_min(1e-300)))
    out = []
    for _ in range(count):
        c = 1.5 * 2.0 ** (52 - bits) * top
        p = (x + c) - c
        out.append(p)
        x, top = x - p, top * 2.0 ** -bits
    return out


def _sum_products(first, xs, ys):
    """first - xs @ ys^T from exact piece products, largest first, in two words."""
    hi, lo = first.clone(), torch.zeros_like(first)
    for level in range(len(xs)):
        for p in range(level + 1):
            t = -(xs[p] @ ys[level - p].T)
            s = hi + t
            b = s - hi
            lo += (hi - (s - b)) + (t - b)
            hi = s
    return hi + lo


def _solve(A, B):
    """Z, row and h of the rows of B for A (m x n), both float64."""
    m, n = A.shape
    Q, R = torch.linalg.qr(A.T)
    bits = (52 - max(1, math.ceil(math.log2(n)))) // 2
    count = -(-72 // bits)
    As = _pieces(A, bits, count)
    Ats = _pieces(A.T.contiguous(), bits, count)
    solve = lambda r: torch.linalg.solve_triangular(R, torch.linalg.solve_triangular(R.T, r.T, upper=False), upper=True).T
    h = torch.linalg.solve_triangular(R, (B @ Q).T, upper=True).T
    parts = [h]                                      # h as a sum of words, so that A^* h carries all of them
    z = B
    for _ in range(4):
        z = B
        for word in parts:
            z = _sum_products(z, _pieces(word, bits, count), Ats)
        dh = solve(_sum_products(torch.zeros_like(h), _pieces(z, bits, count), As).neg())
        parts.append(dh)
    z = _sum_products(z, _pieces(parts[-1], bits, count), Ats)
    h = sum(reversed(parts))
    return z, B - z, h


def exact(case, seed):
    kind = case["kind"]
    x = _inputs(case, seed)
    if kind == "batch":
        return [_solve(A.double(), B.double())[0] for A, B in zip(x["As"], x["Bs"])]
    if case["m"] * case["n"] > 3e8 + 1:
        return None
    if kind == "sparse":
        row_ptr, col, val, U, V = x["A"]
        A = torch.zeros(case["m"], case["n"], device=DEV, dtype=torch.float64)
        row = torch.repeat_interleave(torch.arange(case["m"], device=DEV), row_ptr.diff())
        A.index_put_((row, col.long()), val, accumulate=True)
        if U is not None:
            A += U @ V
    else:
        A = x["A"].double()
        if kind == "ipm":
            A *= x["d"]
    Z, row, h = _solve(A, x["B"].double())
    if kind == "layer":
        Y, _, w = _solve(A, x["G"].double())
        return [Z, -(h.T @ Y + w.T @ Z), Y]
    out = case.get("out", "null")
    return [t for t, keep in ((Z, out != "row"), (row, out != "null"), (h, out == "all")) if keep]
