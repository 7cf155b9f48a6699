"""The work that users of the generalized Nystrom library have it do.

Every case is one pass through the public Python entry points.  The kinds:

approx_f64  sketch, core and factors of a double-precision matrix in one call
            (Algorithm 2 end to end; the plain FP64 path).  ``rank`` > 0 makes a
            numerically low-rank matrix, where the stabilised branch truncates.
sketch      AX and Y^T A on the tensor cores from bf16, split-bf16 or e4m3
            operands; ``src`` names the type of a matrix that is quantized first
            ("" when the operands are already in the tensor-core format).
core        C = (Y^T A) X, its QR, the detector and the truncation rule, from
            an FP32 sketch (what follows a tensor-core sketch).
factors     F = (AX) R^-1 and G = Q^T (Y^T A) from FP32 sketches and a core.
apply       A_hat W or W A_hat from the sketches and the core, A_hat not formed.
adjoint     forward and backward of the differentiable approximant, FP32.
batched     sketches and cores of many uneven small problems in one call.

Matrices are low rank plus noise, sum_i i^-p u_i v_i^T with Gaussian u, v, as
the dense experiments of the method use; sketches are Gaussian.  Inputs are
drawn on the GPU from the seed alone.
"""
import math
import random

import torch

import paper_2009_11392_gb300 as gn

DEV = "cuda"
EPS32 = 10 * 2.0 ** -24 # detector level of FP32-accumulated sketches, relative to ||C||
EPS64 = 10 * 2.0 ** -53
BF16_NOISE = 1.1e-3 # rms rounding of bf16 storage, relative to the matrix' rms entry


def listed():
    return [
        # a small dense double-precision matrix (the paper's 1000 x 500 example): latency and launches
        {"name": "approx_f64_1000x500_r20", "kind": "approx_f64", "m": 1000, "n": 500, "r": 20, "l": 10, "rank": 0},
        # a numerically low-rank matrix: the stabilised form with its second QR
        {"name": "approx_f64_trunc_4096x2048_r100", "kind": "approx_f64", "m": 4096, "n": 2048, "r": 100, "l": 50,
         "rank": 60},
        # the large double-precision example
        {"name": "approx_f64_20000x10000_r500", "kind": "approx_f64", "m": 20000, "n": 10000, "r": 500, "l": 250,
         "rank": 0},
        # a ragged FP32 matrix, stored as bf16 and sketched
        {"name": "quantize_sketch_bf16_3001x1777_r97", "kind": "sketch", "dtype": "bf16", "src": "f32", "m": 3001,
         "n": 1777, "r": 97, "l": 49},
        # the benchmark's sketch
        {"name": "sketch_bf16_32768x16384_r1000", "kind": "sketch", "dtype": "bf16", "src": "", "m": 32768,
         "n": 16384, "r": 1000, "l": 500},
        # 8-bit storage of a matrix that is sketched more than once
        {"name": "sketch_e4m3_16384x8192_r500", "kind": "sketch", "dtype": "e4m3", "src": "", "m": 16384, "n": 8192,
         "r": 500, "l": 250},
        # the core of a small and of the benchmark's approximation
        {"name": "core_n2048_r100", "kind": "core", "m": 4096, "n": 2048, "r": 100, "l": 50},
        {"name": "core_n16384_r1000", "kind": "core", "m": 32768, "n": 16384, "r": 1000, "l": 500},
        # the benchmark's factors, for users who want A_hat = F G
        {"name": "factors_32768x16384_r1000", "kind": "factors", "m": 32768, "n": 16384, "r": 1000, "l": 500},
        # A_hat as an operator on a block of vectors
        {"name": "apply_32768x16384_r1000_64", "kind": "apply", "m": 32768, "n": 16384, "r": 1000, "l": 500,
         "kw": 64, "side": 0},
        # the approximant inside a differentiated program: value and gradient
        {"name": "adjoint_f32_4096_r256", "kind": "adjoint", "m": 4096, "n": 4096, "r": 256, "l": 128},
        # many uneven problems at once (a part of the benchmark's batch)
        {"name": "batched_128", "kind": "batched", "count": 128, "m": 4096, "r": 128},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("approx_f64", "approx_f64", "sketch", "sketch", "core", "core", "factors", "apply", "adjoint",
                       "batched"))
    if kind == "batched":
        return {"kind": kind, "count": _log(rng, 8, 128), "m": _log(rng, 512, 4096), "r": _log(rng, 32, 128)}
    if kind == "approx_f64":
        m = _log(rng, 500, 16000)
        n = _log(rng, 400, min(m, 8000))
        r = _log(rng, 16, min(400, n // 4))
        return {"kind": kind, "m": m, "n": n, "r": r, "l": r // 2, "rank": r * 3 // 5 if rng.random() < 0.3 else 0}
    if kind == "adjoint":
        m, n = _log(rng, 600, 4096), 4 * _log(rng, 150, 1024) # FP32 rows are 16-byte aligned
        r = 8 * _log(rng, 4, 32)
        return {"kind": kind, "m": m, "n": n, "r": r, "l": r // 2}
    m = _log(rng, 1500, 32768)
    n = _log(rng, 1000, 16384)
    r = _log(rng, 16, min(1000, m // 3, n // 2))
    case = {"kind": kind, "m": m, "n": n, "r": r, "l": r // 2}
    if kind == "sketch":
        case["dtype"] = rng.choice(("bf16", "bf16", "split", "e4m3"))
        case["src"] = rng.choice(("", "", "f32", "f64"))
    if kind == "apply":
        case["kw"], case["side"] = _log(rng, 1, 100), rng.randrange(2)
    return case


# ---------------------------------------------------------------- inputs


class _Draw:
    """Gaussian draws of one case from its seed."""

    def __init__(self, seed):
        self.g = torch.Generator(device=DEV)
        self.g.manual_seed(seed & 0x7FFFFFFF)

    def __call__(self, rows, cols, dtype=torch.float32):
        return torch.randn(rows, cols, generator=self.g, device=DEV, dtype=dtype)


def _decay(modes, p, dtype=torch.float64):
    return torch.arange(1, modes + 1, device=DEV, dtype=dtype) ** -p


def _matrix(d, m, n, modes, p, noise, dtype):
    """sum_i i^-p u_i v_i^T + noise N(0, 1), u, v Gaussian of variance 1 / modes."""
    a = (d(m, modes, dtype) / modes * _decay(modes, p, dtype)) @ d(n, modes, dtype).T
    if noise:
        a += noise * d(m, n, dtype)
    return a


def _bf16(t):
    out = gn.padded(t.shape[0], t.shape[1], torch.bfloat16, DEV)
    out.copy_(t)
    return out


def _modes(c):
    return min(c["n"], 4 * c["r"], 2000)


def _sketches(d, c, with_ax):
    """Y^T A (FP32), X (bf16) and A X (FP32) of a bf16-stored low-rank-plus-noise
    matrix, drawn as products with its factors (the matrix itself is not formed)."""
    m, n, r, rl, k = c["m"], c["n"], c["r"], c["r"] + c["l"], _modes(c)
    s = _decay(k, 2.0)
    rms = math.sqrt(float((s * s).sum())) / k
    X = _bf16(d(n, r))
    v = d(n, k, torch.float64) / k * s
    yta = (d(rl, k, torch.float64) * math.sqrt(m)) @ v.T
    yta += BF16_NOISE * rms * math.sqrt(m) * d(rl, n, torch.float64)
    AX = None
    if with_ax:
        AX = (d(m, k) @ (v.T @ X.double()).float()).contiguous()
        AX += BF16_NOISE * rms * math.sqrt(n) * d(m, r)
    return yta.float(), X, AX


def _positive_qr(C):
    Q, R = torch.linalg.qr(C)
    s = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(C.dtype)
    return Q * s, R * s[:, None]


def _batch_shapes(c):
    rng = random.Random("%d %d %d" % (c["count"], c["m"], c["r"]))
    shapes = []
    for _ in range(c["count"]):
        m = rng.randint(256, c["m"])
        r = rng.randint(16, c["r"])
        n = rng.randint(128, m)
        shapes.append((m, n, r, r // 2))
    return shapes


def _batch(c, seed):
    """The batch's operands, one dict of A, X, Y (bf16) per problem."""
    d = _Draw(seed)
    made = []
    for m, n, r, l in _batch_shapes(c):
        k = min(n, 4 * r)
        s = 2.0 ** (-torch.arange(1, k + 1, device=DEV, dtype=torch.float32) / 10)
        a = (d(m, k) / k * s) @ d(n, k).T
        made.append({"A": _bf16(a), "X": _bf16(d(n, r)), "Y": _bf16(d(m, r + l))})
    return made


def _batch_views(shapes, what, dtype):
    """One flat zeroed buffer with a 16-byte aligned view per problem."""
    sizes = [what(*s) for s in shapes]
    flat = torch.zeros(sum((a * b + 3) // 4 * 4 for a, b in sizes), dtype=dtype, device=DEV)
    views, at = [], 0
    for a, b in sizes:
        views.append(flat[at:at + a * b].view(a, b))
        at += (a * b + 3) // 4 * 4
    return flat, views


_BATCH_OUT = (("AX", lambda m, n, r, l: (m, r), torch.float32), ("YtA", lambda m, n, r, l: (r + l, n), torch.float32),
              ("Q", lambda m, n, r, l: (r + l, r), torch.float64), ("R", lambda m, n, r, l: (r, r), torch.float64),
              ("Q2", lambda m, n, r, l: (r, r), torch.float64), ("R2", lambda m, n, r, l: (r, r), torch.float64))


def _inputs(c, seed):
    """What exact() needs too: the inputs, without the library's own objects."""
    d = _Draw(seed)
    kind, m, n, r = c["kind"], c.get("m"), c.get("n"), c.get("r")
    if kind == "batched":
        return _batch(c, seed)
    rl = r + c["l"]
    if kind == "approx_f64":
        if c["rank"]:
            A = _matrix(d, m, n, c["rank"], 0.5, 0.0, torch.float64)
        else:
            A = _matrix(d, m, n, _modes(c), 2.0, 1e-8 / _modes(c), torch.float64)
        return A, d(n, r, torch.float64), d(m, rl, torch.float64)
    if kind == "sketch":
        dt = torch.float64 if c["src"] == "f64" else torch.float32
        return _matrix(d, m, n, min(512, n), 2.0, 0.0, torch.float32).to(dt), d(n, r), d(m, rl)
    if kind == "core":
        yta, X, _ = _sketches(d, c, False)
        return yta, X
    if kind in ("factors", "apply"):
        yta, X, AX = _sketches(d, c, True)
        C = yta.double() @ X.double()
        if kind == "factors":
            return AX, yta, C
        W = d(n, c["kw"], torch.float64) if c["side"] == 0 else d(c["kw"], m, torch.float64)
        return AX, yta, C, W
    k = min(1024, m, n)
    return _matrix(d, m, n, k, 1.5, 1e-6 / k, torch.float32), d(n, r), d(m, rl), d(m, n)


def _empty(rows, cols, dtype):
    return torch.empty(rows, cols, dtype=dtype, device=DEV)


def prepare(case, seed):
    c = case
    kind = c["kind"]
    h = gn.Handle()
    s = {"case": c, "h": h}
    made = _inputs(c, seed)
    if kind == "batched":
        shapes = _batch_shapes(c)
        for name, what, dt in _BATCH_OUT:
            s[name], views = _batch_views(shapes, what, dt)
            for p, v in zip(made, views):
                p[name] = v
        s["k"] = torch.zeros(len(made), dtype=torch.int32, device=DEV)
        for i, p in enumerate(made):
            p["k"] = s["k"][i:i + 1]
        s["problems"] = made
        s["ws"] = h.batched_prepare(made)
        return s
    m, n, r, l = c["m"], c["n"], c["r"], c["l"]
    if kind == "approx_f64":
        s["A"], s["X"], s["Y"] = made
        s["AX"], s["YtA"] = _empty(m, r, torch.float64), _empty(r + l, n, torch.float64)
        s["F"], s["G"] = _empty(m, r, torch.float64), _empty(r, n, torch.float64)
        s["core"] = gn.Core.empty(r, l, DEV)
        s["ws"] = h.workspace(m, n, r, l, gn.F64)
    elif kind == "sketch":
        A, X, Y = made
        s["lo"] = None
        if c["dtype"] == "e4m3":
            s["X"], s["Y"] = h.quantize_e4m3(X, data=False), h.quantize_e4m3(Y, data=False)
        else:
            s["X"], s["Y"] = h.quantize(X), h.quantize(Y)
        s["A"] = A
        if not c["src"]:
            s["A"], s["lo"] = _quantized(h, c["dtype"], A)
        s["AX"], s["YtA"] = _empty(m, r, torch.float32), _empty(r + l, n, torch.float32)
        s["ws"] = h.workspace(m, n, r, l, {"bf16": gn.BF16, "split": gn.BF16X2, "e4m3": gn.E4M3}[c["dtype"]])
    elif kind == "core":
        s["YtA"], s["X"] = made
        s["core"] = gn.Core.empty(r, l, DEV)
        s["ws"] = h.workspace(m, n, r, l, gn.BF16)
    elif kind in ("factors", "apply"):
        s["AX"], s["YtA"], C = made[:3]
        core = gn.Core.empty(r, l, DEV)
        Q, R = _positive_qr(C)
        core.Q.copy_(Q)
        core.R.copy_(R)
        core.C.copy_(C)
        core.k = r
        s["core"] = core
        if kind == "factors":
            s["F"], s["G"] = _empty(m, r, torch.float64), _empty(r, n, torch.float64)
            s["ws"] = h.workspace(m, n, r, l, gn.BF16)
        else:
            s["W"] = made[3]
    else:
        s["A"], s["X"], s["Y"], s["grad"] = made
        s["A"].requires_grad_(True)
    return s


def _quantized(h, dtype, A):
    if dtype == "e4m3":
        return h.quantize_e4m3(A), None
    if dtype == "split":
        return h.quantize(A, split=True)
    return h.quantize(A), None


def run(state):
    s = state
    c, h = s["case"], s["h"]
    kind = c["kind"]
    if kind == "approx_f64":
        eps = 1e-11 if c["rank"] else EPS64
        core = h.approx(s["A"], s["X"], s["Y"], eps, gn.AUTO | gn.EPS_RELATIVE, s["AX"], s["YtA"], s["core"], s["F"],
                        s["G"], s["ws"])
        out = {"AX": s["AX"], "YtA": s["YtA"], "F": s["F"][:, :core.k], "G": s["G"][:core.k], "k": core.k}
        if core.k == c["r"]: # after a truncation the trailing columns of Q hold no information
            out["Q"], out["R"] = core.Q, core.R
        return out
    if kind == "sketch":
        A, lo = (s["A"], s["lo"]) if not c["src"] else _quantized(h, c["dtype"], s["A"])
        h.sketch(A, s["X"], s["Y"], s["AX"], s["YtA"], s["ws"], A_lo=lo)
        return {"AX": s["AX"], "YtA": s["YtA"]}
    if kind == "core":
        core = h.core(s["YtA"], s["X"], EPS32, gn.AUTO | gn.EPS_RELATIVE, s["core"], s["ws"])
        return {"C": core.C, "Q": core.Q, "R": core.R, "k": core.k, "rinv": core.rinv_est, "norm": core.c_norm_est}
    if kind == "factors":
        h.factors(s["AX"], s["YtA"], s["core"], s["F"], s["G"], s["ws"])
        return {"F": s["F"], "G": s["G"]}
    if kind == "apply":
        return {"out": h.apply(s["AX"], s["YtA"], s["core"], s["W"], side=c["side"])}
    if kind == "adjoint":
        value = gn.gn_approx_dense(s["A"], s["X"], s["Y"], h)
        grad, = torch.autograd.grad(value, s["A"], s["grad"])
        return {"value": value.detach(), "grad": grad}
    h.batched_run(EPS32, gn.AUTO | gn.EPS_RELATIVE, s["ws"])
    return {"AX": s["AX"], "YtA": s["YtA"], "Q": s["Q"], "R": s["R"], "k": s["k"]}


# ---------------------------------------------------------------- cost and reference


def _core_flops(r, rl, n):
    return 2.0 * rl * r * n + 4.0 * rl * r * r - 4.0 / 3.0 * r ** 3


def work(case):
    c = case
    kind = c["kind"]
    if kind == "batched":
        b = f = 0.0
        for m, n, r, l in _batch_shapes(c):
            rl = r + l
            b += 2.0 * (m * n + n * r + m * rl) + 4.0 * (m * r + rl * n) + 8.0 * (rl * r + r * r)
            f += 2.0 * m * n * (r + rl) + _core_flops(r, rl, n)
        return {"bytes": b, "flops": f}
    m, n, r = c["m"], c["n"], c["r"]
    rl = r + c["l"]
    if kind == "approx_f64":
        k = c["rank"] or r
        return {"bytes": 8.0 * (m * n + n * r + m * rl + m * r + rl * n + m * k + k * n + rl * r + r * r),
                "flops": 2.0 * m * n * (r + rl) + _core_flops(r, rl, n) + 1.0 * m * k * k + 2.0 * k * rl * n}
    if kind == "sketch":
        e = {"bf16": 2.0, "split": 4.0, "e4m3": 1.0}[c["dtype"]]
        ea = {"": e, "f32": 4.0, "f64": 8.0}[c["src"]]
        es = 1.0 if c["dtype"] == "e4m3" else 2.0
        return {"bytes": ea * m * n + es * (n * r + m * rl) + 4.0 * (m * r + rl * n),
                "flops": (2 if c["dtype"] == "split" else 1) * 2.0 * m * n * (r + rl)}
    if kind == "core":
        return {"bytes": 4.0 * rl * n + 2.0 * n * r + 8.0 * (2 * rl * r + r * r), "flops": _core_flops(r, rl, n)}
    if kind == "factors":
        return {"bytes": 12.0 * m * r + 4.0 * rl * n + 8.0 * (r * n + rl * r + r * r),
                "flops": 1.0 * m * r * r + 2.0 * r * rl * n}
    if kind == "apply":
        kw = c["kw"]
        return {"bytes": 4.0 * (m * r + rl * n) + 8.0 * (rl * r + r * r + kw * (m + n)),
                "flops": 2.0 * kw * (rl * n + r * rl + m * r) + 1.0 * kw * r * r}
    # adjoint: the value's two sketches and its product F G; the gradient's three m x n x r contractions
    return {"bytes": 4.0 * (4 * m * n + n * r + m * rl),
            "flops": 2.0 * m * n * (r + rl) + _core_flops(r, rl, n) + 2.0 * m * n * r
                     + 2.0 * m * n * (rl + r) + 2.0 * m * n * (r + rl)}


def exact(case, seed):
    c = case
    kind = c["kind"]
    made = _inputs(c, seed)
    if kind == "batched":
        out = {"AX": [], "YtA": []}
        for p in made:
            A, X, Y = (p[k].double() for k in ("A", "X", "Y"))
            for name, t in (("AX", A @ X), ("YtA", Y.T @ A)):
                t = t.reshape(-1)
                out[name].append(torch.nn.functional.pad(t, (0, -t.numel() % 4)))
        return {"AX": torch.cat(out["AX"]), "YtA": torch.cat(out["YtA"]), "Q": None, "R": None, "k": None}
    r = c["r"]
    if kind == "approx_f64":
        A, X, Y = made
        AX, YtA = A @ X, Y.T @ A
        out = {"AX": AX, "YtA": YtA, "F": None, "G": None, "k": c["rank"] or r}
        Q, R = _positive_qr(YtA @ X)
        if c["rank"]:
            k = c["rank"]
            Q2, R2 = _positive_qr(R[:k].T.contiguous())
            out["F"] = torch.linalg.solve_triangular(R2.T, AX @ Q2, upper=False, left=False)
            out["G"] = Q[:, :k].T @ YtA
        else:
            out["F"] = torch.linalg.solve_triangular(R, AX, upper=True, left=False)
            out["G"], out["Q"], out["R"] = Q.T @ YtA, Q, R
        return out
    if kind == "sketch":
        A, X, Y = (t.float() for t in made)
        if c["dtype"] == "e4m3":
            A, X, Y = (_e4m3_values(t) for t in (A, X, Y))
        else:
            hi = A.bfloat16()
            A, X, Y = (hi.double() + (A - hi.float()).bfloat16().double() if c["dtype"] == "split" else hi.double(),
                       X.bfloat16().double(), Y.bfloat16().double())
        return {"AX": A @ X, "YtA": Y.T @ A}
    if kind == "core":
        yta, X = made
        C = yta.double() @ X.double()
        Q, R = _positive_qr(C)
        return {"C": C, "Q": Q, "R": R, "k": r, "rinv": None, "norm": None}
    if kind == "factors":
        AX, yta, C = made
        Q, R = _positive_qr(C)
        return {"F": torch.linalg.solve_triangular(R, AX.double(), upper=True, left=False), "G": Q.T @ yta.double()}
    if kind == "apply":
        AX, yta, C, W = made
        Q, R = _positive_qr(C)
        AX, yta = AX.double(), yta.double()
        if c["side"] == 0:
            return {"out": AX @ torch.linalg.solve_triangular(R, Q.T @ (yta @ W), upper=True)}
        return {"out": torch.linalg.solve_triangular(R, W @ AX, upper=True, left=False) @ Q.T @ yta}
    A, X, Y, G = (t.double() for t in made)
    A.requires_grad_(True)
    AX, YtA = A @ X, Y.T @ A
    Q, R = torch.linalg.qr(YtA @ X)
    value = torch.linalg.solve_triangular(R, AX, upper=True, left=False) @ (Q.T @ YtA)
    grad, = torch.autograd.grad(value, A, G)
    return {"value": value.detach(), "grad": grad}


def _e4m3_values(t):
    """``t`` rounded to e4m3 under one power-of-two scale per 128 x 128 tile, the
    smallest with max |t| <= 448 * scale, as FP64."""
    rows, cols = t.shape
    p = torch.nn.functional.pad(t, (0, -cols % 128, 0, -rows % 128))
    tiles = p.view(p.shape[0] // 128, 128, p.shape[1] // 128, 128)
    top = tiles.abs().amax(dim=(1, 3), keepdim=True).double()
    mant, e = torch.frexp(top / 448.0)
    e = torch.where(mant == 0.5, e - 1, e).clamp(-127, 127)
    e = torch.where(top == 0, torch.zeros_like(e), e)
    scale = torch.ldexp(torch.ones_like(top), e)
    q = (tiles.double() / scale).float().clamp(-448, 448).to(torch.float8_e4m3fn).double()
    return (q * scale).reshape(p.shape)[:rows, :cols].contiguous()
