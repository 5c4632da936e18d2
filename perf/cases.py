"""Performance cases of the library: what its users have it do, sized as they do.

Every case runs through the public entry points of
``paper_1502_02389_gb300.lift`` (and ``costmodel.Trainer``, which drives the
cost model's training through them) with the default policy, the default
stream and no explicit variant.  Kinds:

  reduce    one fp32 reduction (asum, dot, nrm2 or sum) of a vector
  dot_scal  the dot + scal step of the vector benchmark
  views     a solver's vector step on slices of larger arrays: odd lengths,
            starts that are not 16-byte aligned; compensated dot, axpy, nrm2
            and asum
  gemv      y <- a A x + b y and z <- a A^T w + b z with one matrix: square,
            tall and narrow, few long rows (a Krylov basis), odd rows
  mixed     asum and dot of bf16 and of block-scaled fp8 vectors
  bs        BlackScholes prices of a list of options
  batch     many small and large calls of uneven sizes in one batched launch
  mlp       one training step of the variant cost model (forward, loss,
            gradients, Adam)
"""
import math

import numpy as np
import torch

from paper_1502_02389_gb300 import costmodel, lift

ALPHA, BETA = 1.0, 0.5                  # of every gemv
STRIKE, RATE, VOL, YEARS = 20.0, 0.02, 0.30, 1.0
BLOCK = 4096                            # elements per fp8 scale


def listed():
    return [
        # one norm of a million floats: a call where launches count
        {"name": "asum_1m", "kind": "reduce", "op": "asum", "n": 1 << 20},
        # the library's headline step: dot and scal of 64M floats
        {"name": "dot_scal_64m", "kind": "dot_scal", "n": 1 << 26},
        # vector updates of an iterative solver on unaligned slices of odd length
        {"name": "views_16m", "kind": "views", "n": (1 << 24) + 43, "ox": 1, "oy": 3},
        # the square matrix of the gemv benchmark, both directions
        {"name": "gemv_8192", "kind": "gemv", "M": 8192, "N": 8192, "pad": 0},
        # the tall matrix of the gemv benchmark (a least-squares system)
        {"name": "gemv_65536x1024", "kind": "gemv", "M": 65536, "N": 1024, "pad": 0},
        # a basis of 32 long vectors: projections h = V w and updates V^T h
        {"name": "gemv_32x1000003", "kind": "gemv", "M": 32, "N": 1000003, "pad": 0},
        # an ordinary matrix whose rows are not whole 16-byte granules
        {"name": "gemv_4097x3001", "kind": "gemv", "M": 4097, "N": 3001, "pad": 0},
        # low-precision vectors of the mixed benchmark
        {"name": "mixed_256m", "kind": "mixed", "n": 1 << 28},
        # the paper's problem size of its finance application
        {"name": "bs_4m", "kind": "bs", "n": 1 << 22},
        # the batched benchmark's distribution of calls, a tenth of its count
        {"name": "batch_2000", "kind": "batch", "count": 2000, "lo": 8, "hi": 22, "mlo": 6,
         "mhi": 12, "ops": 3},
        # thousands of small calls, where per-call work counts
        {"name": "batch_small_4000", "kind": "batch", "count": 4000, "lo": 8, "hi": 14, "mlo": 6,
         "mhi": 8, "ops": 3},
        # one step of training the cost model on the timing sweep (2308 shapes,
        # 265 outputs)
        {"name": "mlp_step", "kind": "mlp", "B": 2308, "V": 265},
    ]


def _log(rng, lo, hi):
    """An integer log-uniform in [lo, hi]."""
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["reduce", "dot_scal", "views", "gemv", "gemv", "mixed", "bs", "batch", "mlp"])
    if kind == "reduce":
        return {"kind": kind, "op": rng.choice(["asum", "dot", "nrm2", "sum"]),
                "n": _log(rng, 1 << 8, 1 << 26)}
    if kind == "dot_scal":
        return {"kind": kind, "n": _log(rng, 1 << 16, 1 << 26)}
    if kind == "views":
        return {"kind": kind, "n": _log(rng, 1 << 16, 1 << 24), "ox": rng.randrange(4),
                "oy": rng.randrange(4)}
    if kind == "gemv":
        M = _log(rng, 16, 65536)
        N = _log(rng, 64, min(1 << 20, (1 << 26) // M))
        if rng.random() < 0.4:              # whole 16-byte granules, as often met
            N = (N + 3) // 4 * 4
        return {"kind": kind, "M": M, "N": N, "pad": rng.choice([0, 0, 0, 1, 8])}
    if kind == "mixed":
        return {"kind": kind, "n": _log(rng, 1 << 16, 1 << 28)}
    if kind == "bs":
        return {"kind": kind, "n": _log(rng, 1 << 12, 1 << 24)}
    if kind == "batch":
        hi = rng.randint(14, 22)
        return {"kind": kind, "count": _log(rng, 50, 2000), "lo": 8, "hi": hi, "mlo": 6,
                "mhi": 8 + (hi - 14) // 2, "ops": rng.randrange(1 << 20)}
    return {"kind": kind, "B": _log(rng, 256, 4096), "V": _log(rng, 64, 512)}


# ---------------------------------------------------------------------------
# inputs (plain torch and numpy, from the seed alone)
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(seed)


def _pair(n, g):
    """Two correlated vectors, as a solver's p and A p or a residual and its
    image are: their dot is about n / 2."""
    x = torch.randn(n, device="cuda", generator=g)
    y = torch.randn(n, device="cuda", generator=g).add_(x, alpha=0.5)
    return x, y


def _outliers(n, g):
    """N(0, 1) with one entry in a hundred 1000 times larger."""
    v = torch.randn(n, device="cuda", generator=g)
    return torch.where(torch.rand(n, device="cuda", generator=g) < 0.01, v * 1e3, v)


def _fp8(v):
    """e4m3 values and one scale per 4096 of them (amax / 448)."""
    nb = (v.numel() + BLOCK - 1) // BLOCK
    p = torch.zeros(nb * BLOCK, device="cuda")
    p[:v.numel()] = v
    p = p.view(nb, BLOCK)
    s = p.abs().amax(1) / 448.0
    s = torch.where(s == 0, torch.ones_like(s), s)
    q = (p / s[:, None]).clamp_(-448.0, 448.0).to(torch.float8_e4m3fn)
    return q.view(-1)[:v.numel()].clone(), s


def _batch_ops(case):
    """Kinds and sizes of a batch, as arrays: asum, dot and gemv (and scal in
    batches of short vectors), drawn from the case's own seed."""
    g = np.random.Generator(np.random.PCG64(case["ops"]))
    c = case["count"]
    kinds = [lift.OP_ASUM, lift.OP_DOT, lift.OP_GEMV] + ([lift.OP_SCAL] if case["hi"] <= 16 else [])
    op = np.array(kinds)[g.integers(0, len(kinds), c)]
    n = np.rint(2.0 ** g.uniform(case["lo"], case["hi"], c)).astype(np.int64)
    M = np.rint(2.0 ** g.uniform(case["mlo"], case["mhi"], c)).astype(np.int64)
    N = np.rint(2.0 ** g.uniform(case["mlo"], case["mhi"], c)).astype(np.int64)
    return op, n, M, N


def _batch_layout(case):
    """Where each op's arrays start: x / y / A in a pool of 256-byte aligned
    slices, scalar results, gemv outputs and scal outputs in arrays of their
    own."""
    op, n, M, N = _batch_ops(case)
    up = lambda v: (v + 63) // 64 * 64  # noqa: E731
    gemv, dot, scal = op == lift.OP_GEMV, op == lift.OP_DOT, op == lift.OP_SCAL
    nx = up(np.where(gemv, N, n))
    ny = up(np.where(dot, n, 0))
    nA = up(np.where(gemv, M * N, 0))
    end = np.cumsum(nx + ny + nA)
    x = end - (nx + ny + nA)
    nout = up(np.where(gemv, M, 0))
    zout = up(np.where(scal, n, 0))
    return {"op": op, "n": n, "M": M, "N": N, "x": x, "y": x + nx, "A": x + nx + ny,
            "pool": int(end[-1]), "out": np.cumsum(nout) - nout, "outs": int(nout.sum()),
            "z": np.cumsum(zout) - zout, "zs": int(zout.sum())}


def _batch_values(L, seed):
    g = _gen(seed)
    pool = torch.randn(L["pool"], device="cuda", generator=g)
    y = torch.randn(max(1, L["outs"]), device="cuda", generator=g)
    for i in np.flatnonzero(L["op"] == lift.OP_DOT):
        x0, y0, n = int(L["x"][i]), int(L["y"][i]), int(L["n"][i])
        pool[y0:y0 + n].add_(pool[x0:x0 + n], alpha=0.5)
    return pool, y


class _Batch:
    """A batch handle, given back with its state."""

    def __init__(self, descs):
        self.handle = lift.lift_batch_create(descs)

    def __del__(self):
        lift.lift_batch_destroy(self.handle)


def _mlp_data(case, seed):
    """Features, targets (log-time ratios), the measured entries and the
    parameters and Adam state of a training under way."""
    g = np.random.Generator(np.random.PCG64(seed))
    B, V = case["B"], case["V"]
    X = g.random((B, costmodel.D_IN)).astype(np.float32)
    T = np.abs(g.standard_normal((B, V)) * 0.5).astype(np.float32)
    M = (g.random((B, V)) < 0.06).astype(np.float32)
    p = costmodel.init_params(V, seed % (1 << 31))
    m = (g.standard_normal(p.size) * 1e-3).astype(np.float32)
    v = (m.astype(np.float64) ** 2 + 1e-6 * (1 + g.random(p.size))).astype(np.float32)
    return X, T, M, p, m, v


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
MLP_T, MLP_LR = 100, 3e-3


def prepare(case, seed):
    lift.lift_init()
    k, g, dev = case["kind"], _gen(seed), "cuda"
    r = lambda c=1: torch.zeros(c, device=dev)  # noqa: E731
    st = {"case": case}
    if k == "reduce":
        st["x"], st["y"] = _pair(case["n"], g)
        if case["op"] != "dot":
            st["x"].add_(0.25)
        st["r"] = r()
    elif k == "dot_scal":
        st["x"], st["y"] = _pair(case["n"], g)
        st["r"], st["z"] = r(), torch.empty_like(st["x"])
    elif k == "views":
        n, ox, oy = case["n"], case["ox"], case["oy"]
        x, y = _pair(n + 3, g)
        st["x"], st["y"] = x[ox:ox + n], y[oy:oy + n]
        st["dot"], st["nrm2"], st["asum"] = r(), r(), r()
    elif k == "gemv":
        M, N = case["M"], case["N"]
        st["A"] = torch.rand((M, N + case["pad"]), device=dev, generator=g).mul_(2).sub_(1)
        u = lambda c: torch.rand(c, device=dev, generator=g).mul_(2).sub_(1)  # noqa: E731
        st["x"], st["y"], st["w"], st["z"] = u(N), u(M), u(M), u(N)
    elif k == "mixed":
        x, y = _outliers(case["n"], g), _outliers(case["n"], g)
        y.add_(x, alpha=0.5)
        st["xb"], st["yb"] = x.bfloat16(), y.bfloat16()
        (st["xq"], st["xs"]), (st["yq"], st["ys"]) = _fp8(x), _fp8(y)
        st["r"] = [r() for _ in range(4)]
    elif k == "bs":
        st["s"] = torch.rand(case["n"], device=dev, generator=g).mul_(25).add_(5)
        st["call"], st["put"] = torch.empty_like(st["s"]), torch.empty_like(st["s"])
    elif k == "batch":
        L = _batch_layout(case)
        st["pool"], st["y"] = _batch_values(L, seed)
        st["r"], st["z"] = r(case["count"]), r(max(1, L["zs"]))
        base, yb, rb, zb = (st[t].data_ptr() for t in ("pool", "y", "r", "z"))
        d = (lift.OpDesc * case["count"])()
        for i in range(case["count"]):
            op, n, M, N = (int(L[t][i]) for t in ("op", "n", "M", "N"))
            e = d[i]
            e.op, e.variant, e.x = op, -1, base + 4 * int(L["x"][i])
            if op == lift.OP_GEMV:
                e.n, e.M, e.N, e.lda, e.alpha, e.beta = M * N, M, N, N, ALPHA, BETA
                e.A = base + 4 * int(L["A"][i])
                e.out = e.y = yb + 4 * int(L["out"][i])
            else:
                e.n, e.alpha = n, 1.5
                e.out = zb + 4 * int(L["z"][i]) if op == lift.OP_SCAL else rb + 4 * i
                if op == lift.OP_DOT:
                    e.y = base + 4 * int(L["y"][i])
        st["batch"] = _Batch(d)
    else:
        X, T, M, p, m, v = _mlp_data(case, seed)
        t = costmodel.Trainer(X, T, M, params=p)
        t.m.copy_(torch.from_numpy(m))
        t.v.copy_(torch.from_numpy(v))
        t.t = MLP_T
        st["trainer"] = t
    return st


def run(st):
    c = st["case"]
    k = c["kind"]
    if k == "reduce":
        if c["op"] == "dot":
            lift.lift_dot(st["x"], st["y"], c["n"], st["r"])
        else:
            getattr(lift, "lift_" + c["op"])(st["x"], c["n"], st["r"])
        return st["r"]
    if k == "dot_scal":
        lift.lift_dot(st["x"], st["y"], c["n"], st["r"])
        lift.lift_scal(c["n"], 1.5, st["x"], st["z"])
        return {"dot": st["r"], "scal": st["z"]}
    if k == "views":
        x, y, n = st["x"], st["y"], c["n"]
        lift.lift_dot_comp(x, y, n, st["dot"])
        lift.lift_axpy(n, -1e-4, x, y)
        lift.lift_nrm2(y, n, st["nrm2"])
        lift.lift_asum(x, n, st["asum"])
        return {"dot": st["dot"], "nrm2": st["nrm2"], "asum": st["asum"], "y": y}
    if k == "gemv":
        M, N, lda = c["M"], c["N"], c["N"] + c["pad"]
        lift.lift_gemv(M, N, ALPHA, st["A"], lda, st["x"], BETA, st["y"])
        lift.lift_gemv_t(M, N, ALPHA, st["A"], lda, st["w"], BETA, st["z"])
        return {"y": st["y"], "z": st["z"]}
    if k == "mixed":
        n, r = c["n"], st["r"]
        lift.lift_asum_ex(lift.BF16, st["xb"], None, n, r[0])
        lift.lift_dot_ex(lift.BF16, st["xb"], None, st["yb"], None, n, r[1])
        lift.lift_asum_ex(lift.FP8_E4M3, st["xq"], st["xs"], n, r[2])
        lift.lift_dot_ex(lift.FP8_E4M3, st["xq"], st["xs"], st["yq"], st["ys"], n, r[3])
        return r
    if k == "bs":
        lift.lift_blackscholes(c["n"], st["s"], STRIKE, RATE, VOL, YEARS, st["call"], st["put"])
        return {"call": st["call"], "put": st["put"]}
    if k == "batch":
        lift.lift_batch_run(st["batch"].handle)
        return {"r": st["r"], "y": st["y"], "z": st["z"]}
    t = st["trainer"]
    t.step(MLP_LR)
    return {"P": t.P, "loss": t.loss, "grads": t.g, "params": t.p, "m": t.m, "v": t.v}


def work(case):
    k = case["kind"]
    if k == "reduce":
        n, ins = case["n"], 2 if case["op"] == "dot" else 1
        return {"bytes": 4 * ins * n, "flops": 2 * n}
    if k == "dot_scal":           # x of both calls, y, and the scaled vector
        return {"bytes": 16 * case["n"], "flops": 3 * case["n"]}
    if k == "views":              # 2 + 3 + 1 + 1 vectors
        return {"bytes": 28 * case["n"], "flops": 14 * case["n"]}
    if k == "gemv":               # A once for each call
        M, N = case["M"], case["N"]
        return {"bytes": 8 * M * N + 12 * (M + N), "flops": 4 * M * N}
    if k == "mixed":
        n = case["n"]
        return {"bytes": 9 * n + 12 * ((n + BLOCK - 1) // BLOCK), "flops": 6 * n}
    if k == "bs":
        return {"bytes": 12 * case["n"], "flops": 40 * case["n"]}
    if k == "batch":
        op, n, M, N = (v.astype(np.float64) for v in _batch_ops(case))
        gemv = op == lift.OP_GEMV
        words = np.where(gemv, M * N + N + 2 * M, np.where(op == lift.OP_ASUM, n, 2 * n))
        return {"bytes": float(4 * words.sum()), "flops": float(2 * np.where(gemv, M * N, n).sum())}
    B, V = case["B"], case["V"]
    d, h1, h2 = costmodel.D_IN, costmodel.H1, costmodel.H2
    weights = d * h1 + h1 * h2 + h2 * V
    params = weights + h1 + h2 + V
    # X, targets and mask read, predictions and their gradient written; the
    # parameters, gradients and Adam moments updated
    return {"bytes": 4 * (B * d + 4 * B * V + 7 * params),
            "flops": B * (6 * weights - 2 * d * h1) + 12 * params}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------
def exact(case, seed):
    k, g = case["kind"], _gen(seed)
    if k == "reduce":
        x, y = _pair(case["n"], g)
        if case["op"] != "dot":
            x.add_(0.25)
        x, y = x.double(), y.double()
        v = {"dot": lambda: x @ y, "asum": lambda: x.abs().sum(), "sum": lambda: x.sum(),
             "nrm2": lambda: (x @ x).sqrt()}[case["op"]]()
        return v.view(1)
    if k == "dot_scal":
        x, y = (v.double() for v in _pair(case["n"], g))
        return {"dot": (x @ y).view(1), "scal": x * 1.5}
    if k == "views":
        n, ox, oy = case["n"], case["ox"], case["oy"]
        x, y = _pair(n + 3, g)
        x, y = x[ox:ox + n].double(), y[oy:oy + n].double()
        y1 = y + float(np.float32(-1e-4)) * x
        return {"dot": (x @ y).view(1), "nrm2": (y1 @ y1).sqrt().view(1),
                "asum": x.abs().sum().view(1), "y": y1}
    if k == "gemv":
        M, N = case["M"], case["N"]
        A = torch.rand((M, N + case["pad"]), device="cuda", generator=g).mul_(2).sub_(1)
        u = lambda c: torch.rand(c, device="cuda", generator=g).mul_(2).sub_(1).double()  # noqa: E731
        x, y, w, z = u(N), u(M), u(M), u(N)
        A = A[:, :N].double()
        return {"y": ALPHA * (A @ x) + BETA * y, "z": ALPHA * (A.T @ w) + BETA * z}
    if k == "mixed":
        x, y = _outliers(case["n"], g), _outliers(case["n"], g)
        y.add_(x, alpha=0.5)
        out = []
        xb, yb = x.bfloat16().double(), y.bfloat16().double()
        out += [xb.abs().sum(), xb @ yb]
        del xb, yb

        def wide(v):
            q, s = _fp8(v)
            return q.double() * s.double().repeat_interleave(BLOCK)[:v.numel()]
        xq, yq = wide(x), wide(y)
        return [v.view(1) for v in out + [xq.abs().sum(), xq @ yq]]
    if k == "bs":
        s = torch.rand(case["n"], device="cuda", generator=g).mul_(25).add_(5).double()
        K, R, S, T = (float(np.float32(v)) for v in (STRIKE, RATE, VOL, YEARS))
        sq = S * math.sqrt(T)
        d1 = (torch.log(s / K) + (R + 0.5 * S * S) * T) / sq
        n = lambda v: 0.5 * torch.erfc(-v / math.sqrt(2.0))  # noqa: E731
        ke = K * math.exp(-R * T)
        call = s * n(d1) - ke * n(d1 - sq)
        return {"call": call, "put": call - s + ke}
    if k == "batch":
        L = _batch_layout(case)
        pool, y = _batch_values(L, seed)
        y = y.double()
        res = torch.zeros(case["count"], device="cuda", dtype=torch.float64)
        z = torch.zeros(max(1, L["zs"]), device="cuda", dtype=torch.float64)
        for i in range(case["count"]):
            op, n, M, N, x0, y0, A0, o, q = (int(L[t][i]) for t in ("op", "n", "M", "N", "x", "y",
                                                                   "A", "out", "z"))
            if op == lift.OP_GEMV:
                A = pool[A0:A0 + M * N].view(M, N).double()
                y[o:o + M] = ALPHA * (A @ pool[x0:x0 + N].double()) + BETA * y[o:o + M]
            elif op == lift.OP_DOT:
                res[i] = pool[x0:x0 + n].double() @ pool[y0:y0 + n].double()
            elif op == lift.OP_ASUM:
                res[i] = pool[x0:x0 + n].double().abs().sum()
            else:
                z[q:q + n] = pool[x0:x0 + n].double() * 1.5
        return {"r": res, "y": y, "z": z}
    X, T, M, p, m, v = (torch.from_numpy(a).cuda().double() for a in _mlp_data(case, seed))
    B, V = case["B"], case["V"]
    d, h1, h2 = costmodel.D_IN, costmodel.H1, costmodel.H2
    W1, b1, W2, b2, W3, b3 = torch.split(p, [d * h1, h1, h1 * h2, h2, h2 * V, V])
    W1, W2, W3 = W1.view(d, h1), W2.view(h1, h2), W3.view(h2, V)
    Z1 = X @ W1 + b1
    H1 = Z1.clamp(min=0)
    Z2 = H1 @ W2 + b2
    H2 = Z2.clamp(min=0)
    P = H2 @ W3 + b3
    inv = float(np.float32(1.0 / max(1.0, float(M.sum()))))
    E = M * (P - T)
    dP = 2 * E * inv
    dZ2 = (dP @ W3.T) * (Z2 > 0)
    dZ1 = (dZ2 @ W2.T) * (Z1 > 0)
    gr = torch.cat([t.reshape(-1) for t in (X.T @ dZ1, dZ1.sum(0), H1.T @ dZ2, dZ2.sum(0),
                                            H2.T @ dP, dP.sum(0))])
    f = lambda s: float(np.float32(s))  # noqa: E731
    c1, c2, t = f(0.9), f(0.999), MLP_T + 1
    m1, v1 = c1 * m + (1 - c1) * gr, c2 * v + (1 - c2) * gr * gr
    step = f(MLP_LR) * (m1 / (1 - c1 ** t)) / ((v1 / (1 - c2 ** t)).sqrt() + f(1e-8))
    return {"P": P, "loss": ((E * E).sum() * inv).view(1), "grads": gr, "params": p - step, "m": m1,
            "v": v1}
