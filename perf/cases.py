"""Workloads by which the library's speed is judged.

Each case is one call of the public API as a user's program makes it: a plan
(or a batch context) made once, inputs and outputs in device memory, then a
factorization A = Q R, a least-squares solve, or a batch of them. Shapes are
those of the library's configurations, benchmark and tests (4096 x 64, the
128-column tall-skinny matrix, 2^21 x 512, near-square, the least-squares
request stream with m up to 262144 and n of 16 to 256, the grouped batch),
with ragged sizes beside them, since users' matrices are seldom a multiple of
a tile.
"""
from __future__ import annotations

import math
import random

import torch

import paper_1710_08471_gb300 as cq

PRECISIONS = {"fp64": cq.CQR2_FP64, "split7": cq.CQR2_OZAKI_BF16, "split6": cq.CQR2_OZAKI_BF16_S6}
GROUP_WORK_LIMIT = 1 << 24  # the request server's limit on m n^2 for the grouped kernel


def _factor(name, m, n, precision="fp64", kappa=1.0, fused=False, panel=0, sync=False):
    return {"name": name, "kind": "factor", "m": m, "n": n, "precision": precision, "kappa": kappa, "fused": fused,
            "panel": panel, "sync": sync}


def _lstsq(name, m, n, precision, kappa, capacity):
    return {"name": name, "kind": "lstsq", "m": m, "n": n, "precision": precision, "kappa": kappa,
            "capacity": capacity}


def _batch(name, count, m_lo, m_hi, widths, precision, kappa, rhs, limit):
    return {"name": name, "kind": "batch", "count": count, "m_lo": m_lo, "m_hi": m_hi, "widths": widths,
            "precision": precision, "kappa": kappa, "rhs": rhs, "limit": limit, "shapes": 1}


def listed():
    return [
        # a single tiny regression fit: the smallest call, all latency and launches
        _lstsq("tiny_fit", 1024, 16, "fp64", 10.0, 1024),
        # the small configuration, plain two-pass FP64, outcome read by the caller
        _factor("small", 4096, 64, sync=True),
        # an ordinary regression of ragged shape in FP64 (design matrix of 100 columns)
        _lstsq("ragged_fit", 50021, 100, "fp64", 1e3, 50021),
        # the tall-skinny FP64 configuration at a quarter of its rows, fused
        _factor("tall_fp64", 1 << 21, 128, kappa=1e6, fused=True),
        # an ordinary FP64 factorization wider than one panel kernel serves, ragged
        _factor("mid_fp64", 6001, 777, kappa=1e2),
        # near-square FP64 on column panels
        _factor("near_square", 8192, 2048, kappa=1e4, panel=512),
        # one request of the least-squares stream at its widest, served in split
        # precision by a plan sized for the stream's largest request
        _lstsq("request", 131601, 256, "split7", 1e3, 262144),
        # split precision: the full tall-skinny configuration
        _factor("tall_split", 1 << 23, 128, "split7", kappa=1e6),
        # split precision: the 512-column configuration
        _factor("wide_split", 1 << 21, 512, "split7", kappa=1e4),
        # split precision with six slices, ragged
        _factor("ragged_split6", 1000037, 200, "split6", kappa=1e2),
        # many equal small factorizations in one call: the grouped kernel
        _batch("batch_small", 1024, 4096, 4096, "32", "fp64", 1.0, False, 4096 * 32 * 32),
        # a burst of the request stream as one batch call: uneven least-squares problems
        _batch("batch_requests", 48, 1024, 262144, "16,32,64,128,256", "split7", 1e2, True, GROUP_WORK_LIMIT),
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, round(math.exp(rng.uniform(math.log(lo), math.log(hi))))))


def draw(rng):
    """One more case of the same ranges: factorizations and least squares in
    each precision from the smallest to the largest sizes, and batches."""
    kind = rng.choice(["factor", "factor", "factor", "lstsq", "lstsq", "batch"])
    kappa = 10.0 ** rng.uniform(0.0, 5.0)
    if kind == "batch":
        count = _log_int(rng, 16, 1024)
        if rng.random() < 0.5:  # small problems for the grouped kernel
            n = rng.randint(8, 64)
            m = _log_int(rng, max(256, n), max(512, 4096 * 32 * 32 // (n * n)))
            return _unnamed(_batch("", count, m // 2 + n, m + n, str(n), "fp64", kappa, rng.random() < 0.5, 1 << 24))
        return _unnamed(_batch("", min(count, 64), 1024, _log_int(rng, 8192, 262144), "16,32,64,128,256",
                               rng.choice(["fp64", "split7"]) if count < 24 else "split7", min(kappa, 1e4), True,
                               GROUP_WORK_LIMIT))
    precision = rng.choice(["fp64", "fp64", "split7", "split6"])
    if precision == "split6":
        kappa = min(kappa, 1e4)
    n = _log_int(rng, 8, 1024) if precision == "fp64" else _log_int(rng, 16, 768)
    if rng.random() < 0.3:  # powers of two are common as well
        n = 1 << max(3, round(math.log2(n)))
    # bounded by the largest listed case: 1.4e11 FP64 flops, 2^30 entries in split precision
    m_hi = min(1 << 22, int(1.2e11 / (4.0 * n * n)) if precision == "fp64" else (1 << 30) // n)
    m = _log_int(rng, max(2 * n, 256), max(m_hi, 2 * n + 1))
    if kind == "lstsq":
        m = min(m, 262144)
        return _unnamed(_lstsq("", m, n, precision, kappa, max(m, _log_int(rng, m, 262144))))
    fused = precision == "fp64" and rng.random() < 0.5
    panel = 128 * rng.randint(1, 4) if precision == "fp64" and n > 512 and rng.random() < 0.5 else 0
    return _unnamed(_factor("", m, n, precision, kappa, fused, panel, rng.random() < 0.3))


def _unnamed(case):
    case.pop("name")
    return case


def _shapes(case):
    """The (m, n) of each problem of a case."""
    if case["kind"] != "batch":
        return [(case["m"], case["n"])]
    rng = random.Random(case["shapes"])
    widths = [int(w) for w in case["widths"].split(",")]
    out = []
    for _ in range(case["count"]):
        m = rng.randint(case["m_lo"], case["m_hi"])
        n = rng.choice(widths)
        out.append((max(m, n), n))
    return out


def _matrix(m, n, kappa, gen):
    """Column-major A = G diag(sigma) V: G iid N(0, 1), sigma log-spaced from 1
    to 1 / kappa, V random orthogonal; iid N(0, 1) for kappa = 1."""
    gt = torch.randn(n, m, dtype=torch.float64, device="cuda", generator=gen)
    if kappa == 1.0 or n == 1:
        return gt.t()
    v, _ = torch.linalg.qr(torch.randn(n, n, dtype=torch.float64, device="cuda", generator=gen))
    sigma = torch.logspace(0.0, -math.log10(kappa), n, dtype=torch.float64, device="cuda")
    return torch.matmul((sigma[:, None] * v).t(), gt).t()


def _inputs(case, seed):
    """[(A, b or None)] of the case's problems, from the seed alone."""
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    rhs = _has_rhs(case)
    return [(_matrix(m, n, case["kappa"], gen),
             torch.randn(m, dtype=torch.float64, device="cuda", generator=gen) if rhs else None)
            for m, n in _shapes(case)]


def _pool(sizes):
    """One zeroed buffer with room for blocks of these sizes at 256-byte
    boundaries, and the blocks: a program with many problems keeps their
    outputs in one allocation."""
    starts, total = [], 0
    for k in sizes:
        starts.append(total)
        total += (k + 31) // 32 * 32
    buf = torch.zeros(total, dtype=torch.float64, device="cuda")
    return buf, [buf[s:s + k] for s, k in zip(starts, sizes)]


def _layout(case):
    """The output pools of a case's problems and each problem's (Q, R, x)."""
    shapes = _shapes(case)
    qb, qs = _pool([m * n for m, n in shapes])
    rb, rs = _pool([n * n for _, n in shapes])
    xb, xs = _pool([n for _, n in shapes])
    outs = [(q.view(n, m).t(), r.view(n, n).t(), x) for (m, n), q, r, x in zip(shapes, qs, rs, xs)]
    return {"Q": qb, "R": rb, "x": xb}, outs


def _has_rhs(case):
    return case["kind"] == "lstsq" or (case["kind"] == "batch" and case["rhs"])


def prepare(case, seed):
    data = _inputs(case, seed)
    prec = PRECISIONS[case["precision"]]
    pools, outs = _layout(case)
    if not _has_rhs(case):
        del pools["x"]
    state = {"case": case, "data": data, "outs": outs, "pools": pools}
    if case["kind"] == "batch":
        problems = [(A, Q, R) if b is None else (A, Q, R, b, x) for (A, b), (Q, R, x) in zip(data, outs)]
        state["batch"] = cq.Batch(case["count"], precision=prec, small_work_limit=case["limit"])
        state["problems"] = cq.Batch.descriptors(problems)
    elif case["kind"] == "lstsq":
        state["plan"] = cq.Plan(case["capacity"], case["n"], precision=prec)
    else:
        state["plan"] = cq.Plan(case["m"], case["n"], precision=prec, fused=case["fused"])
        if case["panel"]:
            state["plan"].set_panel_width(case["panel"])
    return state


def run(state):
    case = state["case"]
    if case["kind"] == "batch":
        state["batch"].factor(state["problems"], sync=False)
        return dict(state["pools"])
    (A, b), (Q, R, x) = state["data"][0], state["outs"][0]
    if case["kind"] == "lstsq":
        state["plan"].lstsq_rows(A, b, Q=Q, R=R, x=x, sync=False)
        return {"Q": Q, "R": R, "x": x}
    state["plan"].factor(A, Q=Q, R=R, sync=case["sync"])
    return {"Q": Q, "R": R}


def work(case):
    """Compulsory traffic (A in, Q and R out, b and x where there is a solve)
    and the method's nominal flops, 4 m n^2 + (5/3) n^3, with 2 m n + n^2 for a solve."""
    rhs = _has_rhs(case)
    nbytes = flops = 0.0
    for m, n in _shapes(case):
        nbytes += 8.0 * (2 * m * n + n * n + (m + n if rhs else 0))
        flops += 4.0 * m * n * n + 5.0 / 3.0 * n**3 + (2.0 * m * n + n * n if rhs else 0.0)
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    """Householder QR with R's diagonal made positive, and x from R x = Q^T b."""
    pools, outs = _layout(case)
    for (A, b), (Qo, Ro, xo) in zip(_inputs(case, seed), outs):
        Q, R = torch.linalg.qr(A)
        d = torch.sign(torch.diagonal(R))
        Qo.copy_(Q.mul_(d))
        Ro.copy_(R.mul_(d[:, None]))
        if b is not None:
            xo.copy_(torch.linalg.solve_triangular(Ro, (Qo.t() @ b)[:, None], upper=True)[:, 0])
    if not _has_rhs(case):
        del pools["x"]
    if case["kind"] == "batch":
        return pools
    return dict(zip(pools, outs[0]))
