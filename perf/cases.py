"""Performance cases: the calls a user of this package makes, over the sizes it is used at.

Every case goes through the public Python API (api.py, autograd.py).  Inputs are drawn on
the GPU from the seed; the distributions are those of workloads.py (N(0, 1/n) matrices,
uniform vectors, jittered and relabelled Kuhn tet meshes, random CSR matrices, log-uniform
batch mixes).
"""
from __future__ import annotations

import math
import random

import torch

from paper_2507_13204_gb300 import api
from paper_2507_13204_gb300.autograd import gradient_descent

_DT = {"f64": torch.float64, "f32": torch.float32}
_ES = {"f64": 8, "f32": 4}


def listed():
    return [
        # the smallest calls, where launches and latency count: the paper's own 1-D example at
        # its largest size, value and both gradients
        dict(name="laplace-10000", kind="laplace", dtype="f64", n=10000),
        # one small dense model, value and gradient
        dict(name="dense-f64-64", kind="dense", dtype="f64", m=64, n=64),
        # an ordinary least-squares matrix that fits L2
        dict(name="dense-f64-2000x1500", kind="dense", dtype="f64", m=2000, n=1500),
        # the largest square one, streamed from HBM
        dict(name="dense-f64-10000", kind="dense", dtype="f64", m=10000, n=10000),
        # many observations of few unknowns, odd row length (rows not 16-byte aligned)
        dict(name="dense-f64-150001x255", kind="dense", dtype="f64", m=150001, n=255),
        # the same in single precision, shorter rows
        dict(name="dense-f32-400000x100", kind="dense", dtype="f32", m=400000, n=100),
        # value and gradient on a large tet mesh
        dict(name="tet-f64-100", kind="tet", op="grad", dtype="f64", strategy="auto", jitter=False,
             a=100, b=100, c=100),
        # Newton-CG on an ordinary ragged mesh: reproducible Hessian-vector products
        dict(name="tet-hvp-f64-37x41x29", kind="tet", op="hvp", dtype="f64", strategy="csr", jitter=True,
             a=37, b=41, c=29),
        # a large random sparse matrix, value and gradient
        dict(name="sparse-f64-1048576", kind="sparse", dtype="f64", strategy="auto", m=1 << 20, n=1 << 20,
             lo=8, hi=24, gval=False),
        # a rectangular one in single precision with ragged rows: reproducible, gradients w.r.t.
        # x and the stored values
        dict(name="sparse-f32-300001x200003", kind="sparse", dtype="f32", strategy="transpose", m=300001,
             n=200003, lo=1, hi=60, gval=True),
        # whole call: a batch of small problems in one launch
        dict(name="batch-f64-128+16", kind="batch", dtype="f64", dense=128, tets=16, jitter=False, mix=3),
        # whole call: gradient descent through torch.autograd (taped forward, reverse from the tape)
        dict(name="descent-f32-64x60x67", kind="descent", dtype="f32", jitter=True, a=64, b=60, c=67,
             steps=8),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["laplace", "dense", "dense", "dense", "tet", "tet", "sparse", "sparse", "batch",
                       "descent"])
    dtype = rng.choice(["f64", "f32"])
    if kind == "laplace":
        return dict(kind=kind, dtype=dtype, n=_log(rng, 10, 10000))
    if kind == "dense":
        n = _log(rng, 32, 10240)
        m = _log(rng, 32, min(400000, 40_000_000 // n))
        return dict(kind=kind, dtype=dtype, m=m, n=n)
    if kind == "sparse":
        lo = rng.randint(1, 8)
        hi = rng.randint(lo, 60)
        rows = min(1 << 20, 2 * 16_000_000 // (lo + hi))
        return dict(kind=kind, dtype=dtype, strategy=rng.choice(["auto", "transpose"]),
                    m=_log(rng, 1000, rows), n=_log(rng, 1000, 1 << 20), lo=lo, hi=hi,
                    gval=rng.random() < 0.5)
    if kind == "batch":
        dense = rng.randint(16, 128)
        return dict(kind=kind, dtype=dtype, dense=dense, tets=max(1, dense // 8), jitter=rng.random() < 0.5,
                    mix=rng.randint(0, 10**6))
    side = _log(rng, 6, 100 if kind == "tet" else 64)
    a, b, c = (max(1, round(side * rng.uniform(0.7, 1.0))) for _ in range(3))
    box = dict(dtype=dtype, jitter=rng.random() < 0.5, a=a, b=b, c=c)
    if kind == "descent":
        return dict(kind=kind, steps=rng.randint(1, 8), **box)
    return dict(kind=kind, op=rng.choice(["grad", "hvp"]), strategy=rng.choice(["auto", "csr"]), **box)


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return g


def _uniform(n, dtype, g):
    return (torch.rand(n, generator=g, dtype=torch.float64, device="cuda") * 2 - 1).to(dtype)


def _matrix(m, n, dtype, g):
    return torch.randn((m, n), generator=g, dtype=dtype, device="cuda") * math.sqrt(1.0 / n)


def _mesh(a, b, c, dtype, jitter, g):
    """Kuhn-split a x b x c box of unit cubes, vertices relabelled at random; jitter moves the
    interior vertices, so that every element has its own shape."""
    nv = (a + 1) * (b + 1) * (c + 1)
    ar = lambda k: torch.arange(k, device="cuda")  # noqa: E731
    sy, sz = a + 1, (a + 1) * (b + 1)
    base = (ar(c)[:, None, None] * sz + ar(b)[None, :, None] * sy + ar(a)[None, None, :]).reshape(-1)
    step = (1, sy, sz)
    conn = torch.stack([torch.stack([base, base + step[p], base + step[p] + step[q], base + 1 + sy + sz], 1)
                        for p, q in ((0, 1), (0, 2), (1, 0), (1, 2), (2, 0), (2, 1))], 1).reshape(-1, 4)
    v = ar(nv)
    xyz = torch.stack([v % sy, v // sy % (b + 1), v // sz], 1).double()
    if jitter:
        top = torch.tensor([a, b, c], device="cuda", dtype=torch.float64)
        inside = ((xyz > 0) & (xyz < top)).all(1)
        xyz += inside[:, None] * (torch.rand((nv, 3), generator=g, dtype=torch.float64, device="cuda") * 0.2 - 0.1)
    p = xyz[conn]
    e1, e2, e3 = p[:, 1] - p[:, 0], p[:, 2] - p[:, 0], p[:, 3] - p[:, 0]
    r1, r2, r3 = (torch.linalg.cross(s, t) for s, t in ((e2, e3), (e3, e1), (e1, e2)))
    det = (e1 * r1).sum(1, keepdim=True)
    g1, g2, g3 = r1 / det, r2 / det, r3 / det
    G = torch.stack([-(g1 + g2 + g3), g1, g2, g3], 2).reshape(-1, 12).to(dtype).contiguous()
    perm = torch.randperm(nv, generator=g, device="cuda")
    return perm[conn].to(torch.int32).contiguous(), G, nv


def _csr(m, n, lo, hi, dtype, g):
    # the row lengths are the case's, so that every seed has the same number of stored entries
    deg = torch.randint(lo, hi + 1, (m,), generator=_gen(m), device="cuda")
    rowptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = deg.cumsum(0)
    nnz = int(rowptr[-1])
    rows = torch.repeat_interleave(torch.arange(m, device="cuda"), deg)
    col = (rows * n + torch.randint(0, n, (nnz,), generator=g, device="cuda")).sort().values % n
    val = torch.randn(nnz, generator=g, dtype=dtype, device="cuda") / deg[rows].to(dtype).sqrt()
    return rowptr.to(torch.int32), col.to(torch.int32), val


def _mix(case):
    """Sizes of a batch: dense n log-uniform in 32..2048, tet boxes of 1e3..5e4 elements."""
    r = random.Random(case["mix"])
    sizes = [_log(r, 32, 2048) for _ in range(case["dense"])]
    boxes = []
    for _ in range(case["tets"]):
        t = math.exp(r.uniform(math.log(1e3), math.log(5e4)))
        s = max(1, int((t / 6) ** (1 / 3)))
        boxes.append((s, s, max(1, round(t / (6 * s * s)))))
    return sizes, boxes


def _slots(lengths):
    """Offsets of vectors laid out one after another, each on a 256-byte boundary."""
    off, at = [], 0
    for k in lengths:
        off.append(at)
        at += (k + 63) // 64 * 64
    return off, at


def _inputs(case, seed):
    g, dt, kind = _gen(seed), _DT[case["dtype"]], case["kind"]
    if kind == "laplace":
        return dict(b=_uniform(case["n"], dt, g), x=_uniform(case["n"], dt, g))
    if kind == "dense":
        return dict(A=_matrix(case["m"], case["n"], dt, g), x=_uniform(case["n"], dt, g))
    if kind == "sparse":
        rowptr, col, val = _csr(case["m"], case["n"], case["lo"], case["hi"], dt, g)
        return dict(rowptr=rowptr, col=col, val=val, x=_uniform(case["n"], dt, g))
    if kind == "batch":
        sizes, boxes = _mix(case)
        mats = [_matrix(n, n, dt, g) for n in sizes]
        meshes = [_mesh(*box, dt, case["jitter"], g) for box in boxes]
        off, total = _slots(sizes + [nv for _, _, nv in meshes])
        x = _uniform(total, dt, g)
        return dict(mats=mats, meshes=meshes, off=off, x=x)
    conn, G, nv = _mesh(case["a"], case["b"], case["c"], dt, case["jitter"], g)
    return dict(conn=conn, G=G, nv=nv, x=_uniform(nv, dt, g), v=_uniform(nv, dt, g))


# --------------------------------------------------------------- the calls
def prepare(case, seed):
    i, kind = _inputs(case, seed), case["kind"]
    s = dict(case=case, x=i["x"])
    if kind == "laplace":
        s["problem"] = api.Laplace1D(i["b"])
        s["gb"] = torch.empty_like(i["b"])
    elif kind == "dense":
        s["problem"] = api.QuadForm(i["A"])
    elif kind == "sparse":
        s["problem"] = api.SpQuadForm(i["rowptr"], i["col"], i["val"], case["n"], strategy=case["strategy"])
        s["gval"] = torch.empty_like(i["val"]) if case["gval"] else None
    elif kind == "batch":
        probs = [api.QuadForm(A) for A in i["mats"]] + [api.TetEnergy(c, G, nv) for c, G, nv in i["meshes"]]
        s["batch"] = api.Batch(probs)
        s["f"] = torch.zeros(len(probs), dtype=i["x"].dtype, device="cuda")
        s["gx"] = torch.zeros_like(i["x"])
        cut = lambda t: [t[o:o + p.nx] for o, p in zip(i["off"], probs)]  # noqa: E731
        s["buffers"] = s["batch"].bind(cut(i["x"]), [s["f"][k] for k in range(len(probs))], cut(s["gx"]))
    else:
        s["problem"] = api.TetEnergy(i["conn"], i["G"], i["nv"], strategy=case.get("strategy", "auto"))
        s["v"] = i["v"]
    return s


def run(state):
    case, p = state["case"], state.get("problem")
    kind = case["kind"]
    if kind == "laplace":
        f, gx = p.grad(state["x"], gdata=state["gb"])
        return f, gx, state["gb"]
    if kind == "sparse":
        f, gx = p.grad(state["x"], gdata=state["gval"])
        return (f, gx, state["gval"]) if case["gval"] else (f, gx)
    if kind == "batch":
        state["batch"].grad(state["buffers"])
        return state["f"], state["gx"]
    if kind == "descent":
        history = []
        u = gradient_descent(p, state["x"], 0.01, case["steps"], history=history)
        return u, history
    if kind == "tet" and case["op"] == "hvp":
        return p.hvp(state["x"], state["v"])
    return p.grad(state["x"])


# ---------------------------------------------------------------- the work
def _tet_work(ne, nv, es):
    return ne * (16 + 12 * es) + 2 * nv * es, 80 * ne


def _counts(case):
    a, b, c = case["a"], case["b"], case["c"]
    return 6 * a * b * c, (a + 1) * (b + 1) * (c + 1)


def work(case):
    es, kind = _ES[case["dtype"]], case["kind"]
    if kind == "laplace":
        return {"bytes": 4 * es * case["n"], "flops": 16 * case["n"]}
    if kind == "dense":
        m, n = case["m"], case["n"]
        return {"bytes": es * (m * n + 2 * n), "flops": 4 * m * n}
    if kind == "sparse":
        m, n = case["m"], case["n"]
        nnz = m * (case["lo"] + case["hi"]) // 2
        more = es * nnz if case["gval"] else 0
        return {"bytes": 4 * (m + 1) + (4 + es) * nnz + 2 * es * n + more, "flops": 4 * nnz}
    if kind == "batch":
        sizes, boxes = _mix(case)
        by = sum(es * (n * n + 2 * n) for n in sizes)
        fl = sum(4 * n * n for n in sizes)
        for a, b, c in boxes:
            tb, tf = _tet_work(6 * a * b * c, (a + 1) * (b + 1) * (c + 1), es)
            by, fl = by + tb, fl + tf
        return {"bytes": by, "flops": fl}
    ne, nv = _counts(case)
    by, fl = _tet_work(ne, nv, es)
    if kind == "descent":
        return {"bytes": case["steps"] * by, "flops": case["steps"] * fl}
    if case["op"] == "hvp":
        return {"bytes": by + nv * es, "flops": 120 * ne}
    return {"bytes": by, "flops": fl}


# --------------------------------------------------------- values in 64 bits
def _dense_exact(A, x):
    A, x = A.double(), x.double()
    y = A @ x
    return (y * y).sum(), 2 * (y @ A)


def _gathered(conn, G, u):
    return torch.einsum("erk,ek->er", G, u[conn])


def _scattered(conn, G, h, nv):
    out = torch.zeros(nv, dtype=torch.float64, device=h.device)
    return out.index_add_(0, conn.reshape(-1), torch.einsum("erk,er->ek", G, h).reshape(-1))


def _tet_exact(conn, G, u, nv):
    conn, G, u = conn.long(), G.double().view(-1, 3, 4), u.double()
    g = _gathered(conn, G, u)
    s = (g * g).sum(1)
    return torch.log1p(s).sum(), _scattered(conn, G, 2 * g / (1 + s)[:, None], nv)


def exact(case, seed):
    i, kind = _inputs(case, seed), case["kind"]
    if kind == "laplace":
        x, b = i["x"].double(), i["b"].double()
        zero = torch.zeros(1, dtype=torch.float64, device="cuda")
        lap = lambda t: 2 * t - torch.cat([zero, t[:-1]]) - torch.cat([t[1:], zero])  # noqa: E731
        y = lap(3 * x) - b
        return (y * y).sum(), 6 * lap(y), -2 * y
    if kind == "dense":
        return _dense_exact(i["A"], i["x"])
    if kind == "sparse":
        rows = torch.repeat_interleave(torch.arange(case["m"], device="cuda"), i["rowptr"].diff().long())
        col, val, x = i["col"].long(), i["val"].double(), i["x"].double()
        y = torch.zeros(case["m"], dtype=torch.float64, device="cuda").index_add_(0, rows, val * x[col])
        gx = torch.zeros_like(x).index_add_(0, col, 2 * val * y[rows])
        f = (y * y).sum()
        return (f, gx, 2 * x[col] * y[rows]) if case["gval"] else (f, gx)
    if kind == "batch":
        fs, gx = [], torch.zeros_like(i["x"], dtype=torch.float64)
        nd = len(i["mats"])
        for k, o in enumerate(i["off"]):
            if k < nd:
                n = i["mats"][k].shape[1]
                f, g = _dense_exact(i["mats"][k], i["x"][o:o + n])
            else:
                conn, G, n = i["meshes"][k - nd]
                f, g = _tet_exact(conn, G, i["x"][o:o + n], n)
            fs.append(f)
            gx[o:o + n] = g
        return torch.stack(fs), gx
    if kind == "descent":
        u, history = i["x"].double(), []
        for _ in range(case["steps"]):
            f, g = _tet_exact(i["conn"], i["G"], u, i["nv"])
            history.append(f)
            u = u - 0.01 * g
        return u, history
    if case["op"] == "hvp":
        conn, G = i["conn"].long(), i["G"].double().view(-1, 3, 4)
        g, d = _gathered(conn, G, i["x"].double()), _gathered(conn, G, i["v"].double())
        w = (2 / (1 + (g * g).sum(1)))[:, None]
        return _scattered(conn, G, w * d - w * w * (g * d).sum(1, keepdim=True) * g, i["nv"])
    return _tet_exact(i["conn"], i["G"], i["x"], i["nv"])
