"""The work a user of this library has it do, as measurable cases.

A case names one call of the public Python entry points (`radic_det`, `radic_det_exact_wide`,
`BatchPlan.radic_det_batched`, `radic_det_autograd`) with its sizes, arithmetic and element type.
The sizes are the library's five benchmark workloads (workloads.py) and the shapes between and
below them that its tests use; `draw` spreads over the same ranges.
"""
from __future__ import annotations

import math
from fractions import Fraction

import numpy as np
import torch

import paper_1508_01326_gb300 as R

_TORCH = {"i8": torch.int8, "i32": torch.int32, "f32": torch.float32, "f64": torch.float64}
_BYTES = {"i8": 1, "i32": 4, "f32": 4, "f64": 8}


def listed():
    return [
        # the smallest benchmark workload: one exact integer determinant, all latency
        dict(name="exact_i32_3x12", kind="det", mode="exact", dtype="i32", m=3, n=12),
        # a small binary64 matrix between the workloads (4368 minors): launches and fixed costs
        dict(name="fp64_5x16", kind="det", mode="fp64", dtype="f64", m=5, n=16),
        # the single-matrix workload in its two arithmetics (10.5 million minors)
        dict(name="mixed_8x32", kind="det", mode="mixed", dtype="f64", m=8, n=32),
        dict(name="fp64_8x32", kind="det", mode="fp64", dtype="f64", m=8, n=32),
        # more rows than the prefix mapping takes in binary64: a warp group per minor
        dict(name="fp64_12x20", kind="det", mode="fp64", dtype="f64", m=12, n=20),
        # exact integer determinants: the 10 x 24 block and the full 12 x 40 workload, the largest
        # single determinant (5.59e9 minors)
        dict(name="exact_i8_10x24", kind="det", mode="exact", dtype="i8", m=10, n=24),
        dict(name="exact_i8_12x40", kind="det", mode="exact", dtype="i8", m=12, n=40),
        # the exact value of real input, beyond 128 bits
        dict(name="wide_f64_8x32", kind="wide", dtype="f64", m=8, n=32),
        # the uneven batch of the headline benchmark (3.4e9 minors), through the router
        dict(name="batched_mixed_4096", kind="batched", mode="mixed", dtype="f64", batch=4096, m_lo=2, m_hi=10,
             d_hi=20, shapes=4),
        # an ordinary batch in plain binary64 from binary32 entries
        dict(name="batched_fp64_300", kind="batched", mode="fp64", dtype="f32", batch=300, m_lo=2, m_hi=9, d_hi=16,
             shapes=7),
        # training: forward and backward of the differentiation workload, and of a smaller, odd
        # one through the router
        dict(name="train_fp64_256x6x28", kind="train", mode="fp64", batch=256, m=6, n=28),
        dict(name="train_mixed_30x5x19", kind="train", mode="mixed", batch=30, m=5, n=19),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: its kind and arithmetic, then a shape whose work lies between the smallest and
    the largest listed case of that kind (evenly in the logarithm of the number of minors)."""
    kind = rng.choice(["det", "det", "det", "wide", "batched", "train"])
    if kind == "batched":
        lo = rng.randint(2, 8)
        return dict(kind=kind, mode=rng.choice(["mixed", "fp64"]), dtype=rng.choice(["f64", "f32"]),
                    batch=_log_int(rng, 9, 900), m_lo=lo, m_hi=rng.randint(lo, 9), d_hi=rng.randint(3, 16),
                    shapes=rng.randint(10, 1 << 20))
    if kind == "train":
        m, n = _shape(rng, 3, 8, 28, 20, 400_000)
        return dict(kind=kind, mode=rng.choice(["fp64", "mixed"]), m=m, n=n,
                    batch=min(256, _log_int(rng, 1, max(2, min(256, 96_000_000 // math.comb(n, m))))))
    if kind == "wide":
        m, n = _shape(rng, 3, 8, 32, 200, 10_518_300)
        return dict(kind=kind, dtype=rng.choice(["f64", "f32"]), m=m, n=n)
    mode = rng.choice(["fp64", "mixed", "pair", "exact"])
    if mode == "exact":
        m, n = _shape(rng, 3, 12, 40, 200, 100_000_000)
        return dict(kind=kind, mode=mode, dtype=rng.choice(["i8", "i32"]), m=m, n=n)
    m, n = _shape(rng, 3, 12 if mode == "fp64" else 10, 40, 200, 12_000_000)
    if m > 10 and math.comb(n, m) > 400_000:
        n = m + 7
    return dict(kind=kind, mode=mode, dtype=rng.choice(["f64", "f64", "f32"]), m=m, n=n)


def _shape(rng, m_lo, m_hi, n_hi, lo, hi):
    """m x n with m in [m_lo, m_hi], m < n <= n_hi and C(n, m) near a count drawn from [lo, hi]."""
    want = math.exp(rng.uniform(math.log(lo), math.log(hi)))
    m = rng.randint(m_lo, m_hi)
    n = m + 1
    while n < n_hi and math.comb(n + 1, m) <= want:
        n += 1
    return m, n


def _batch_shapes(case):
    rng = np.random.default_rng(case["shapes"])
    ms = rng.integers(case["m_lo"], case["m_hi"] + 1, case["batch"])
    ds = rng.integers(1, case["d_hi"] + 1, case["batch"])
    return [(int(m), int(m + d)) for m, d in zip(ms, ds)]


def _matrix(case, seed, shape):
    """Entries as the benchmark workloads draw them: integers in [-3, 3] (int8) or [-9, 9] (int32),
    reals uniform in [-1, 1); batches N(0, 1)."""
    rng = np.random.default_rng([0x5241, seed])
    dt = case.get("dtype", "f64")
    if dt in ("i8", "i32"):
        b = 3 if dt == "i8" else 9
        return torch.from_numpy(rng.integers(-b, b + 1, shape).astype(np.int8 if dt == "i8" else np.int32))
    a = rng.standard_normal(shape) if case["kind"] == "batched" else rng.uniform(-1.0, 1.0, shape)
    return torch.from_numpy(a).to(_TORCH[dt])


def _host(case, seed):
    if case["kind"] == "batched":
        return _matrix(case, seed, sum(m * n for m, n in _batch_shapes(case)))
    if case["kind"] == "train":
        return _matrix(case, seed, (case["batch"], case["m"], case["n"]))
    return _matrix(case, seed, (case["m"], case["n"]))


def _grad_out(case, seed):
    return torch.from_numpy(np.random.default_rng([0x4752, seed]).uniform(0.5, 1.5, case["batch"]))


def _fields(out):
    """The result record's fields: value, sum of |terms|, error bound, and its whole-number words."""
    f = out.view(torch.float64)
    return {"value": f[..., 0], "abs_sum": f[..., 1], "err_bound": f[..., 2], "words": out[..., 3:]}


def prepare(case, seed):
    A = _host(case, seed).cuda()
    s = {"kind": case["kind"], "mode": case.get("mode"), "A": A}
    if case["kind"] == "det":
        # a program that calls in a loop keeps its result record and workspace
        s["out"] = R.new_result()
        s["ws"] = torch.empty(max(256, R.radic_workspace_bytes(case["m"], case["n"], case["mode"])), dtype=torch.uint8,
                              device="cuda")
        s["fields"] = _fields(s["out"])
    elif case["kind"] == "wide":
        s["out"] = torch.zeros(R.api.WIDE_RESULT_BYTES, dtype=torch.uint8, device="cuda")
        s["fields"] = {"value": s["out"][:8].view(torch.float64), "words": s["out"][8:].view(torch.int64)}
    elif case["kind"] == "batched":
        s["plan"] = R.BatchPlan(_batch_shapes(case), mode=case["mode"])
        s["out"] = s["plan"].new_results()
        s["fields"] = _fields(s["out"])
    else:
        s["A"] = A.requires_grad_(True)
        s["w"] = _grad_out(case, seed).cuda()
    return s


def run(state):
    if state["kind"] == "det":
        R.radic_det(state["A"], mode=state["mode"], out=state["out"], workspace=state["ws"])
        return state["fields"]
    if state["kind"] == "wide":
        R.radic_det_exact_wide(state["A"], out=state["out"])
        return state["fields"]
    if state["kind"] == "batched":
        state["plan"].radic_det_batched(state["A"], out=state["out"])
        return state["fields"]
    d = R.radic_det_autograd(state["A"], state["mode"])
    (g,) = torch.autograd.grad(d, state["A"], state["w"])
    return {"det": d.detach(), "grad": g}


def work(case):
    """Matrix in, result out; arithmetic: each signed minor enters the sum and the sum of
    magnitudes (floating modes: a D-term product and two additions, taken as 7 operations) or, where
    only the sum is returned (exact modes per prime, gradients), one multiply-add."""
    if case["kind"] == "batched":
        shapes = _batch_shapes(case)
        return {"bytes": sum(m * n for m, n in shapes) * _BYTES[case["dtype"]] + 128 * len(shapes),
                "flops": 7 * sum(math.comb(n, m) for m, n in shapes)}
    mn, c = case["m"] * case["n"], math.comb(case["n"], case["m"])
    if case["kind"] == "train":
        return {"bytes": case["batch"] * (2 * mn * 8 + 16), "flops": case["batch"] * (7 + 2) * c}
    if case["kind"] == "wide":
        return {"bytes": mn * _BYTES[case["dtype"]] + 192, "flops": 2 * 15 * c}
    return {"bytes": mn * _BYTES[case["dtype"]] + 128, "flops": (6 if case["mode"] == "exact" else 7) * c}


# ---------------------------------------------------------------------------
# The same quantities in plain Python integers, numpy and torch.  Summed over the ascending column
# sequences, det_R satisfies a recurrence over the columns: f[S], the signed sum of the minors of
# the rows S over the columns taken so far, gains for column j and each row i of S the Laplace term
# (-1)^(|S| + position of i in S) (-1)^j a_ij f[S without i].
# ---------------------------------------------------------------------------
def _steps(m):
    """Per row i: the row sets S that hold i, S without i, and the Laplace signs."""
    steps = []
    for i in range(m):
        S = np.array([s for s in range(1 << m) if s >> i & 1])
        pos = np.array([bin(s & ((1 << i) - 1)).count("1") + 1 for s in S])
        size = np.array([bin(s).count("1") for s in S])
        steps.append((S, S ^ (1 << i), np.where((pos + size) % 2 == 0, 1, -1)))
    return steps


def _sum_exact(a):
    """det_R of a host matrix as a Fraction."""
    m, n = a.shape
    rows = [[Fraction(x) for x in r] for r in a.tolist()]
    scale = [max(x.denominator for x in r) for r in rows]
    ints = [[int(x * s) for x in r] for r, s in zip(rows, scale)]
    f = np.zeros(1 << m, dtype=object)
    f[0] = 1
    steps = _steps(m)
    for j in range(n):
        g = f.copy()
        for i, (S, rest, sign) in enumerate(steps):
            g[S] += f[rest] * sign * (ints[i][j] if j % 2 else -ints[i][j])
        f = g
    total = int(f[-1]) * (-1 if m * (m + 1) // 2 % 2 else 1)
    return Fraction(total, math.prod(scale))


def _sum_f64(a):
    """det_R of a (batch, m, n) binary64 tensor, differentiable."""
    b, m, n = a.shape
    steps = [(torch.from_numpy(rest).to(a.device), torch.from_numpy(sign).to(a)) for _, rest, sign in _steps(m)]
    at = [torch.from_numpy(S).to(a.device) for S, _, _ in _steps(m)]
    f = torch.zeros(b, 1 << m, dtype=torch.float64, device=a.device)
    f[:, 0] = 1.0
    for j in range(n):
        add = torch.zeros_like(f)
        for i in range(m):
            add = add.index_add(1, at[i], f[:, steps[i][0]] * steps[i][1] * a[:, i, j].unsqueeze(1))
        f = f + (add if j % 2 else -add)
    return f[:, -1] * (-1.0 if m * (m + 1) // 2 % 2 else 1.0)


def _sum_abs(a):
    """Sum of |minor| of a (m, n) binary64 tensor."""
    m, n = a.shape
    c = torch.arange(n - m + 1, device=a.device).unsqueeze(1)
    for k in range(1, m):
        room = n - m + k - c[:, -1]
        first = torch.repeat_interleave(room.cumsum(0) - room, room)
        step = torch.arange(int(room.sum()), device=a.device) - first
        c = torch.repeat_interleave(c, room, dim=0)
        c = torch.cat([c, (c[:, -1] + 1 + step).unsqueeze(1)], dim=1)
    total = 0.0
    for part in c.split(400_000):
        total += float(torch.linalg.det(a[:, part].permute(1, 0, 2).contiguous()).abs().sum())
    return total


def exact(case, seed):
    a = _host(case, seed)
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    if case["kind"] in ("det", "wide"):
        value = torch.tensor(float(_sum_exact(a)), dtype=torch.float64)
        if case["kind"] == "wide":
            return {"value": value.reshape(1), "words": None}
        if case["mode"] == "exact":
            zero = torch.zeros((), dtype=torch.float64)
            return {"value": value, "abs_sum": zero, "err_bound": zero, "words": None}
        tot = _sum_abs(a.double().to(dev)) if math.comb(case["n"], case["m"]) <= 12_000_000 else None
        return {"value": value, "abs_sum": None if tot is None else torch.tensor(tot, dtype=torch.float64),
                "err_bound": None, "words": None}
    if case["kind"] == "batched":
        shapes = _batch_shapes(case)
        offs = np.concatenate([[0], np.cumsum([m * n for m, n in shapes])])
        value = torch.zeros(len(shapes), dtype=torch.float64)
        for m in sorted({m for m, _ in shapes}):
            ids = [b for b, (mm, _) in enumerate(shapes) if mm == m]
            pad = torch.zeros(len(ids), m, max(shapes[b][1] for b in ids), dtype=torch.float64)  # zero columns add 0
            for k, b in enumerate(ids):
                pad[k, :, :shapes[b][1]] = a[offs[b]:offs[b + 1]].double().reshape(shapes[b])
            value[ids] = _sum_f64(pad.to(dev)).cpu()
        return {"value": value, "abs_sum": None, "err_bound": None, "words": None}
    x = a.to(dev).requires_grad_(True)
    d = _sum_f64(x)
    (g,) = torch.autograd.grad(d, x, _grad_out(case, seed).to(dev))
    return {"det": d.detach(), "grad": g}
