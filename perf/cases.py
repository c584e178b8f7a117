"""The workloads by which this library's speed is judged: one pass of each
through the public Python entry points, and the same numbers in 64 bits from
plain torch (no code of the library), to say how exact a pass is.

Sizes: the benchmark's own configurations (the planted 1000 x 800 problem, the
dense 65,536 x 16,384 matrix in its precisions and sketches, the 2e6 x 5e5
text matrix, the 1024 uneven instances, the k = 32 network's mini-batches) and
the shapes of the dense datasets of the paper's Table 1, whose odd sizes take
the unaligned paths.  draw() spreads the same kinds over their ranges.
"""
import math
import random

import numpy as np
import torch

import paper_2009_02845_gb300 as pkg

DEV = "cuda"
SKETCH = {"gaussian": pkg.GAUSSIAN, "rademacher": pkg.RADEMACHER, "subsample": pkg.SUBSAMPLE,
          "identity": pkg.IDENTITY}
PREC = {"fp32": pkg.FP32, "bf16": pkg.BF16, "fp8": pkg.FP8}
MASK = 0xFFFFFFFF


def _dense(name, m, n, k, d, dv, **kw):
    c = dict(kind="dense", m=m, n=n, k=k, d=d, dv=dv, sketch="gaussian", prec="fp32", reassoc=False, rcd=False,
             inner=1, graph=True, steps=1)
    c.update(kw)
    return dict(c, name=name) if name else c


def _text(name, m, n, k, d, dv, prec, steps, mean=100):
    c = dict(kind="text", m=m, n=n, k=k, d=d, dv=dv, prec=prec, mean=mean, steps=steps)
    return dict(c, name=name) if name else c


def listed():
    big = (65536, 16384, 64, 2048, 2048)
    return [
        # the smallest problem of the benchmark, run to its full 50 iterations: launches and latency
        _dense("small planted fp32", 1000, 800, 10, 100, 100, steps=50),
        # a small face-image matrix (Table 1's FACE: odd sizes) with the paper's k and its coordinate descent
        # on sampled columns (d = d' = 2k), all options otherwise at their defaults (no graph)
        _dense("faces subsample rcd fp32", 2429, 361, 100, 200, 200, sketch="subsample", rcd=True, graph=False,
               steps=4),
        # a mid-size dense matrix whose rows are no multiple of 8 (Table 1's GISETTE), the plain FP32 form
        _dense("gisette gaussian fp32", 13500, 5000, 100, 500, 1350),
        # the headline: the dense image-like matrix in bf16, the paper's order
        _dense("dense gaussian bf16", *big, prec="bf16"),
        # the same in the cheaper order R = M (S B^T)
        _dense("dense gaussian bf16 reassoc", *big, prec="bf16", reassoc=True, steps=4),
        # the same in FP8
        _dense("dense gaussian fp8", *big, prec="fp8"),
        # the same matrix with sampled columns, FP32
        _dense("dense subsample fp32", *big, sketch="subsample", steps=4),
        # the large text matrix (1.4e8 entries), both stored precisions of the factors
        _text("text fp32", 2_000_000, 500_000, 100, 5000, 5000, "fp32", 5),
        _text("text bf16", 2_000_000, 500_000, 100, 5000, 5000, "bf16", 5),
        # 1024 uneven instances advanced together for their 100 iterations, then every factor read back
        dict(name="batch of 1024 bf16", kind="batch", count=1024, shapes=0, prec="bf16", rcd=False, steps=100),
        # ten training steps of the warm start's network (16 groups of 512 rows each)
        dict(name="network training", kind="train", k=32, hidden=256, groups=16, rows=512, steps=10),
        # the relative error that a run logs, on the dense matrix
        dict(name="dense error", kind="error", m=65536, n=16384, k=64),
    ]


def _span(rng, lo, hi, mult=1):
    """A size between lo and hi, spread over its logarithm, a multiple of `mult`."""
    v = int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))
    return max(mult, v // mult * mult)


def draw(rng):
    kind = rng.choice(["dense", "dense", "dense", "sampled", "sampled", "text", "text", "batch", "train", "predict",
                       "error"])
    if kind == "dense":
        prec = rng.choice(["fp32", "fp32", "bf16", "bf16", "fp8"])
        mult = 1 if prec == "fp32" else 16
        m, n = _span(rng, 1000, 65536, mult), _span(rng, 361, 16384, mult)
        if prec == "fp32":
            m, n = min(m, 20000), min(n, 8000)
        k = rng.choice([10, 16, 31, 32, 48, 64, 100])
        f = rng.uniform(0.05, 0.15)
        d, dv = max(8, int(n * f) // 8 * 8), min(2048, max(8, int(m * f) // 8 * 8))
        sketch = rng.choice(["gaussian", "gaussian", "rademacher"] + (["identity"] if prec == "bf16" else []))
        rcd = rng.random() < 0.2
        if rcd:  # coordinate descent wants more equations than unknowns
            d, dv = max(d, 8 * ((2 * k + 7) // 8)), max(dv, 8 * ((2 * k + 7) // 8))
        if sketch == "identity":
            d, dv = n, m
        return _dense(None, m, n, k, d, dv, prec=prec, sketch=sketch, rcd=rcd,
                      inner=1 if rcd else rng.choice([1, 1, 4]), reassoc=sketch != "identity" and rng.random() < 0.4,
                      graph=rng.random() < 0.5, steps=rng.choice([1, 2, 4]))
    if kind == "sampled":
        m, n, k = _span(rng, 1000, 65536), _span(rng, 361, 16384), rng.choice([10, 31, 32, 48, 64, 100])
        f, rcd = rng.uniform(0.02, 0.15), rng.random() < 0.3
        lo = 2 * k if rcd else 8
        return _dense(None, m, n, k, max(lo, int(n * f)), max(lo, int(m * f / 2)), sketch="subsample", rcd=rcd,
                      graph=rng.random() < 0.5, steps=rng.choice([1, 2, 4]))
    if kind == "text":
        m, n = _span(rng, 20_000, 1_500_000), _span(rng, 10_000, 400_000)
        prec = rng.choice(["fp32", "bf16"])
        k = rng.choice([20, 48, 66, 100, 128] if prec == "fp32" else [48, 66, 100, 128])
        return _text(None, m, n, k, max(50, n // 100), max(50, m // rng.choice([400, 100])), prec,
                     rng.choice([2, 5]), rng.choice([20, 100]))
    if kind == "batch":
        return dict(kind="batch", count=_span(rng, 8, 128), shapes=rng.randrange(1 << 20),
                    prec=rng.choice(["fp32", "bf16"]), rcd=rng.random() < 0.3, steps=rng.choice([5, 10]))
    if kind in ("train", "predict"):
        c = dict(kind=kind, k=rng.choice([8, 20, 32]), hidden=rng.choice([64, 100, 256]))
        if kind == "train":
            return dict(c, groups=_span(rng, 1, 16), rows=_span(rng, 100, 512), steps=5)
        return dict(c, groups=rng.choice([1, 1, 3]), rows=_span(rng, 1000, 65536))
    return dict(kind="error", m=_span(rng, 1000, 65536), n=_span(rng, 361, 16384),
                k=rng.choice([10, 31, 32, 48, 64, 100]))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed, salt=0):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + salt)
    return g


def _planted(m, n, k, g, zero=0.7):
    """U0 V0^T + |N(0, 0.01^2)|, U0 and V0 uniform with a share of zeros."""
    U = torch.rand((m, k), generator=g, device=DEV)
    V = torch.rand((n, k), generator=g, device=DEV)
    if zero:
        U[torch.rand((m, k), generator=g, device=DEV) < zero] = 0.0
        V[torch.rand((n, k), generator=g, device=DEV) < zero] = 0.0
    M = torch.randn((m, n), generator=g, device=DEV).abs_().mul_(0.01)
    return M.addmm_(U, V.T)


def _text_csr(case, seed):
    """Document lengths lognormal, term ids Zipf(1.07), repeated terms merged,
    values log(1 + count), count ~ Poisson(1) >= 1; with the transposed CSR."""
    m, n, g = case["m"], case["n"], _gen(seed)
    L = torch.empty(m, device=DEV).log_normal_(math.log(case["mean"]) - 0.5, 1.0, generator=g)
    L = L.round_().clamp_(1, n).long()
    cdf = torch.arange(1, n + 1, device=DEV, dtype=torch.float64).pow_(-1.07).cumsum_(0)
    total = int(L.sum())
    row = torch.repeat_interleave(torch.arange(m, device=DEV), L)
    key = torch.searchsorted(cdf, torch.rand(total, generator=g, device=DEV, dtype=torch.float64) * cdf[-1])
    key = key.clamp_(max=n - 1).add_(row.mul_(n))
    key = torch.unique_consecutive(key.sort()[0])
    row, col = key // n, key % n
    del key
    nnz = row.numel()
    cnt = torch.poisson(torch.ones(nnz, device=DEV), generator=g).clamp_(min=1)
    val = torch.log1p(cnt)
    del cnt
    rp, trp = torch.zeros(m + 1, dtype=torch.int64, device=DEV), torch.zeros(n + 1, dtype=torch.int64, device=DEV)
    torch.cumsum(torch.bincount(row, minlength=m), 0, out=rp[1:])
    torch.cumsum(torch.bincount(col, minlength=n), 0, out=trp[1:])
    order = (col * m).add_(row).argsort()
    return rp, col.int(), val, trp, row[order].int(), val[order]


def _shapes(case):
    """Uneven instances: m in [128, 4096], n in [64, 2048], k in {8, 16, 32}, d = max(4k, n/8), d' = max(4k, m/8)."""
    r = random.Random(case["shapes"])
    out = []
    for i in range(case["count"]):
        m, n, k = r.randint(128, 4096), r.randint(64, 2048), r.choice([8, 16, 32])
        out.append(dict(m=m, n=n, k=k, d=max(4 * k, n // 8), d_v=max(4 * k, m // 8), seed=i))
    return out


def _batch_inputs(case, seed):
    for i, s in enumerate(_shapes(case)):
        yield i, s, _planted(s["m"], s["n"], s["k"], _gen(seed, i + 1), zero=0.0)


def _triples(case, seed):
    """Row problems min 1/2 x^T (G + mu I) x - b^T x, x >= 0 with their exact minimisers: x* is sparse and b meets
    the optimality conditions with it."""
    k, groups, rows, g = case["k"], case["groups"], case["rows"], _gen(seed)
    Y = torch.rand((groups, 1024, k), generator=g, device=DEV)
    Y[torch.rand((groups, 1024, k), generator=g, device=DEV) < 0.7] = 0.0
    G = torch.bmm(Y.transpose(1, 2), Y)
    mu = 1.0 + torch.randint(0, 300, (groups,), generator=g, device=DEV).float()
    x = torch.rand((groups, rows, k), generator=g, device=DEV)
    off = torch.rand((groups, rows, k), generator=g, device=DEV) < 0.6
    x[off] = 0.0
    slack = torch.rand((groups, rows, k), generator=g, device=DEV) * 5.0
    b = torch.bmm(x, G) + mu[:, None, None] * x - torch.where(off, slack, torch.zeros_like(slack))
    o = torch.arange(0, groups + 1, dtype=torch.int64, device=DEV) * rows
    return G.contiguous(), mu, o, b.reshape(-1, k).contiguous(), x.reshape(-1, k).contiguous()


def _params(case, seed):
    """Starting weights of the network: W1g, W1b, b1, W2, b2, W3, b3, uniform by fan-in."""
    k, h = case["k"], case["hidden"]
    r = np.random.default_rng(int(seed) + 77)
    fan = [(h * k * k, k * k + k), (h * k, k * k + k), (h, 0), (h * h, h), (h, 0), (k * h, h), (k, 0)]
    return np.concatenate([r.uniform(-1, 1, c).astype(np.float32) * np.float32(math.sqrt(3.0 / f) if f else 0.0)
                           for c, f in fan])


def _set_dense(h, M):
    torch.cuda.synchronize()  # the handle copies M on a stream of its own
    h.set_dense(M)


def prepare(case, seed):
    kind = case["kind"]
    if kind in ("dense", "text", "error"):
        m, n, k = case["m"], case["n"], case["k"]
        st = dict(U=torch.empty((m, k), device=DEV), V=torch.empty((n, k), device=DEV))
    if kind == "dense":
        h = pkg.DSANLS(m, n, k, case["d"], SKETCH[case["sketch"]], seed=seed, d_v=case["dv"],
                       solver=pkg.RCD if case["rcd"] else pkg.PGD, precision=PREC[case["prec"]],
                       order=pkg.ORDER_REASSOCIATED if case["reassoc"] else pkg.ORDER_PAPER,
                       inner_iters=case["inner"], use_graph=int(case["graph"]))
        _set_dense(h, _planted(m, n, k, _gen(seed), zero=0.0 if m * n < 1 << 20 else 0.7))
        return dict(st, case=case, h=h)
    if kind == "text":
        h = pkg.DSANLS(m, n, k, case["d"], pkg.SUBSAMPLE, seed=seed, d_v=case["dv"], use_graph=1,
                       precision=PREC[case["prec"]])
        csr = _text_csr(case, seed)
        torch.cuda.synchronize()
        h.set_csr(*csr)
        return dict(st, case=case, h=h)
    if kind == "error":
        h = pkg.DSANLS(m, n, k, max(1, n // 8), pkg.GAUSSIAN, seed=seed)
        _set_dense(h, _planted(m, n, k, _gen(seed)))
        return dict(case=case, h=h)
    if kind == "batch":
        b = pkg.Batch(_shapes(case), precision=PREC[case["prec"]], use_graph=1,
                      solver=pkg.RCD if case["rcd"] else pkg.PGD)
        if case["prec"] == "bf16":  # pinned, so that a run does not depend on what a timing chose
            b.set_tile(192, 3, 2, 1)
        for i, s, M in _batch_inputs(case, seed):
            torch.cuda.synchronize()
            b.set_dense(i, M)
        return dict(case=case, b=b)
    net = pkg.MLP(case["k"], case["hidden"], max_rows=case["groups"] * case["rows"], max_groups=case["groups"])
    net.set_params(_params(case, seed))
    n = case["steps"] if kind == "train" else 1
    return dict(case=case, net=net,
                data=[_triples(case, seed * 101 + i) for i in range(n)])


def run(state):
    case = state["case"]
    kind = case["kind"]
    if kind in ("dense", "text"):
        state["h"].step(case["steps"])
        U, V = state["h"].factors(state["U"], state["V"])
        return {"U": U, "V": V}
    if kind == "error":
        return {"error": state["h"].rel_error()}
    if kind == "batch":
        state["b"].step(case["steps"])
        got = [state["b"].factors(i) for i in range(case["count"])]
        return {"U": np.concatenate([u.reshape(-1) for u, _ in got]),
                "V": np.concatenate([v.reshape(-1) for _, v in got])}
    if kind == "train":
        loss = [state["net"].train_step(*d, 1e-3) for d in state["data"]]
        return {"loss": loss, "params": state["net"].params()}
    G, mu, off, b, _ = state["data"][0]
    return {"x": state["net"].predict(G, mu, off, b)}


def work(case):
    """Bytes and operations of a pass that no implementation of the chosen form avoids."""
    kind, steps = case["kind"], case.get("steps", 1)
    if kind == "train" or kind == "predict":
        k, h, R = case["k"], case["hidden"], case["groups"] * case["rows"]
        P = h * k * k + h * k + h + h * h + h + k * h + k
        fwd = 2.0 * R * (h * k + h * h + k * h) + 2.0 * case["groups"] * h * k * k
        if kind == "predict":
            return {"bytes": 4.0 * (2 * R * k + P), "flops": fwd}
        return {"bytes": steps * 4.0 * (2 * R * k + 6 * P), "flops": steps * 3 * fwd}
    if kind == "batch":
        e = 2 if case["prec"] == "bf16" else 4
        by = fl = 0.0
        for s in _shapes(case):
            m, n, k, d, dv = s["m"], s["n"], s["k"], s["d"], s["d_v"]
            by += 2.0 * e * m * n + 8.0 * (m + n) * k
            fl += 2.0 * m * n * (d + dv) + 2.0 * k * (m * d + n * dv) + 2.0 * k * (n * d + m * dv)
        return {"bytes": steps * by, "flops": steps * fl}
    m, n, k = case["m"], case["n"], case["k"]
    if kind == "error":
        return {"bytes": 4.0 * (m * n + (m + n) * k), "flops": 2.0 * m * n * k}
    fac = 8.0 * (m + n) * k
    upd = 2.0 * (m + n) * k * k
    if kind == "text":
        nnz = 0.7 * m * case["mean"]
        sub = nnz * case["d"] / n + nnz * case["dv"] / m
        e = 1 if case["prec"] == "fp32" else 0.5
        return {"bytes": steps * (e * fac + 8 * sub), "flops": steps * (upd + 2 * sub * k)}
    d, dv = case["d"], case["dv"]
    e = {"fp32": 4.0, "bf16": 2.0, "fp8": 1.0}[case["prec"]]
    upd *= case["inner"]
    if case["sketch"] == "subsample":
        return {"bytes": steps * (4.0 * (m * d + n * dv) + fac), "flops": steps * (upd + 2.0 * k * (m * d + n * dv))}
    if case["sketch"] == "identity":
        return {"bytes": steps * (2 * e * m * n + fac), "flops": steps * (upd + 4.0 * m * n * k)}
    small = 2.0 * k * (n * d + m * dv)
    if case["reassoc"]:
        return {"bytes": steps * (2 * e * m * n + fac), "flops": steps * (upd + 2 * small + 4.0 * m * n * k)}
    return {"bytes": steps * (2 * e * m * n + fac),
            "flops": steps * (upd + small + 2.0 * m * n * (d + dv) + 2.0 * k * (m * d + n * dv))}


# ---------------------------------------------------------------------------
# the same in 64 bits
# ---------------------------------------------------------------------------

def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 (Salmon et al. 2011) on int64 tensors that hold 32-bit words."""
    for _ in range(10):
        p0, p1 = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = ((p1 >> 32) & MASK) ^ c1 ^ k0, p1 & MASK, ((p0 >> 32) & MASK) ^ c3 ^ k1, p0 & MASK
        k0, k1 = (k0 + 0x9E3779B9) & MASK, (k1 + 0xBB67AE85) & MASK
    return c0, c1, c2, c3


def _words(seed, stream, t, rows, cols):
    """The field's words: (rows / 4 rounded up, 4, cols), word r of block q belongs to row 4 q + r."""
    q = torch.arange((rows + 3) // 4, device=DEV)[:, None]
    j = torch.arange(cols, device=DEV)[None, :]
    z = torch.zeros_like(q)
    w = _philox(q + 0 * j, j + 0 * q, z + (t & MASK), z + ((stream & 0xFF) | ((t >> 32) << 8)), seed & MASK, seed >> 32)
    return w


def _uniform(seed, stream, rows, cols):
    w = torch.stack(_words(seed, stream, 0, rows, cols), 1).reshape(-1, cols)[:rows]
    return (w >> 8).double() * 2.0 ** -24


def _field(sketch, seed, side, t, K, d):
    S = torch.empty(((K + 3) // 4, 4, d), dtype=torch.float64, device=DEV)
    a, b, c, e = _words(seed, side, t, K, d)
    if sketch == "rademacher":
        for r, w in enumerate((a, b, c, e)):
            S[:, r] = 1.0 - 2.0 * (w >> 31).double()
    else:
        for r, (u, v) in ((0, (a, b)), (2, (c, e))):
            rad = (((u >> 9) * 2 + 1).double() * 2.0 ** -24).log_().mul_(-2.0).sqrt_()
            ang = ((v >> 9) * 2 + 1).double() * (2.0 ** -24 * 2.0 * math.pi)
            S[:, r], S[:, r + 1] = rad * ang.cos(), rad * ang.sin()
    return S.reshape(-1, d)[:K].mul_(1.0 / math.sqrt(d))


def _sampled(seed, side, t, n, d):
    """The d columns of a 4-round Feistel permutation of {0..n-1} with cycle walking, ascending."""
    h = 1
    while h < 16 and (1 << (2 * h)) < n:
        h += 1
    mask = (1 << h) - 1
    x = torch.arange(d, device=DEV)
    todo = torch.ones(d, dtype=torch.bool, device=DEV)
    while bool(todo.any()):
        L, R = x >> h, x & mask
        for rnd in range(4):
            w = _philox(R, 0 * R + rnd, 0 * R + (t & MASK), 0 * R + ((0x10 | side) | ((t >> 32) << 8)), seed & MASK,
                        seed >> 32)[0]
            L, R = R, L ^ (w & mask)
        x = torch.where(todo, (L << h) | R, x)
        todo &= x >= n
    return x.sort()[0]


def _update(Z, G, R, t, rcd, inner):
    x = torch.full((G.shape[0],), 1.0 / math.sqrt(G.shape[0]), dtype=torch.float64, device=DEV)
    for _ in range(32):
        y = G @ x
        x = y / y.norm()
    mu = 1.0 + t
    eta = 1.0 / (x @ (G @ x) + mu)
    if rcd:
        Z = Z.clone()
        for j in range(G.shape[0]):
            num = mu * Z[:, j] + R[:, j] - Z @ G[:, j] + Z[:, j] * G[j, j]
            Z[:, j] = (num / (G[j, j] + mu)).clamp_(min=0)
        return Z
    X, b = Z, R + mu * Z
    for _ in range(inner):
        X = (X - eta * (X @ G + mu * X - b)).clamp_(min=0)
    return X


def _half(case, seed, side, t, X, Y, Z):
    """One half-step: X (rows x K) the data or what multiplies like it, Y (K x k) the fixed factor."""
    K, d = Y.shape[0], case["d"] if side == 0 else case["dv"]
    if case["sketch"] == "identity":
        return _update(Z, Y.T @ Y, X @ Y, t, case["rcd"], case["inner"])
    if case["sketch"] == "subsample":
        J = _sampled(seed, side, t, K, d)
        B, R = Y[J].T * math.sqrt(K / d), (X[:, J] @ Y[J]) * (K / d)
    else:
        S = _field(case["sketch"], seed, side, t, K, d)
        B = Y.T @ S
        R = X @ (S @ B.T)
    return _update(Z, B @ B.T, R, t, case["rcd"], case["inner"])


class _SampledText:
    """Columns J of a CSR matrix times rows J of Y, from the transposed CSR."""

    def __init__(self, tp, ti, tv, rows):
        self.tp, self.ti, self.tv, self.rows = tp, ti, tv, rows

    def __call__(self, J, Y):
        n = self.tp[J + 1] - self.tp[J]
        seg = torch.repeat_interleave(torch.arange(J.numel(), device=DEV), n)
        e = torch.arange(seg.numel(), device=DEV) - torch.repeat_interleave(n.cumsum(0) - n, n) + self.tp[J][seg]
        out = torch.zeros((self.rows, Y.shape[1]), dtype=torch.float64, device=DEV)
        for a in range(0, seg.numel(), 1 << 22):
            s, q = seg[a:a + (1 << 22)], e[a:a + (1 << 22)]
            out.index_add_(0, self.ti[q].long(), Y[J[s]] * self.tv[q].double()[:, None])
        return out


def _exact_text(case, seed):
    rp, col, val, trp, trow, tval = _text_csr(case, seed)
    m, n, k = case["m"], case["n"], case["k"]
    U, V = _uniform(seed, 2, m, k), _uniform(seed, 3, n, k)
    if case["prec"] == "bf16":
        U, V = U.bfloat16().double(), V.bfloat16().double()
    prod = (_SampledText(trp, trow, tval, m), _SampledText(rp, col, val, n))
    for t in range(case["steps"]):
        for side in (0, 1):
            Y, Z, d = (V, U, case["d"]) if side == 0 else (U, V, case["dv"])
            K = Y.shape[0]
            J = _sampled(seed, side, t, K, d)
            B = Y[J].T * math.sqrt(K / d)
            Z = _update(Z, B @ B.T, prod[side](J, Y) * (K / d), t, False, 1)
            U, V = (Z, V) if side == 0 else (U, Z)
    return {"U": U, "V": V}


def _iterate(case, M, steps, phil):
    m, n = M.shape
    U, V = _uniform(phil, 2, m, case["k"]), _uniform(phil, 3, n, case["k"])
    M = M.double()
    for t in range(steps):
        U = _half(case, phil, 0, t, M, V, U)
        V = _half(case, phil, 1, t, M.T, U, V)
    return U, V


def _forward(case, theta, G, mu, off, b):
    """The network with bf16-rounded weights: (o, s per row, beta)."""
    k, h = case["k"], case["hidden"]
    parts, at = [], 0
    for c in (h * k * k, h * k, h, h * h, h, k * h, k):
        parts.append(theta[at:at + c])
        at += c
    W1g, W1b, b1, W2, b2, W3, b3 = parts
    gelu = torch.nn.functional.gelu
    A = G.double() + mu.double()[:, None, None] * torch.eye(k, dtype=torch.float64, device=DEV)
    s = A.diagonal(dim1=1, dim2=2).sum(1) / k
    grp = torch.repeat_interleave(torch.arange(G.shape[0], device=DEV), off[1:] - off[:-1])
    b = b.double()
    beta = b.norm(dim=1) / math.sqrt(k)
    beta = torch.where(beta > 0, beta, torch.ones_like(beta))
    zg = (A / s[:, None, None]).reshape(-1, k * k) @ W1g.reshape(h, k * k).T
    h1 = gelu((b / beta[:, None]) @ W1b.reshape(h, k).T + zg[grp] + b1)
    h2 = gelu(h1 @ W2.reshape(h, h).T + b2)
    return h2 @ W3.reshape(k, h).T + b3, s[grp], beta


def _exact_train(case, seed):
    theta = torch.from_numpy(_params(case, seed)).to(DEV).double()
    m, v, losses = torch.zeros_like(theta), torch.zeros_like(theta), []
    for i in range(case["steps"]):
        G, mu, off, b, x = _triples(case, seed * 101 + i)
        w = theta.float().bfloat16().double().requires_grad_(True)
        o, s, beta = _forward(case, w, G, mu, off, b)
        y = x.double() * (s / beta)[:, None]
        e = torch.where(y > 0, o - y, o.clamp(min=0))
        loss = 0.5 * e.square().sum(1).mean()
        g, = torch.autograd.grad(loss, w)
        losses.append(float(loss))
        m, v = 0.9 * m + 0.1 * g, 0.999 * v + 0.001 * g * g
        theta = theta - 1e-3 * (m / (1 - 0.9 ** (i + 1))) / ((v / (1 - 0.999 ** (i + 1))).sqrt() + 1e-8)
    return {"loss": losses, "params": theta}


def exact(case, seed):
    kind = case["kind"]
    if kind == "text":
        return _exact_text(case, seed)
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "predict":
        G, mu, off, b, _ = _triples(case, seed * 101)
        theta = torch.from_numpy(_params(case, seed)).to(DEV).bfloat16().double()
        o, s, beta = _forward(case, theta, G, mu, off, b)
        return {"x": o.clamp(min=0) * (beta / s)[:, None]}
    if kind == "dense":
        M = _planted(case["m"], case["n"], case["k"], _gen(seed), zero=0.0 if case["m"] * case["n"] < 1 << 20 else 0.7)
        U, V = _iterate(case, M, case["steps"], seed)
        return {"U": U, "V": V}
    if kind == "error":
        M = _planted(case["m"], case["n"], case["k"], _gen(seed)).double()
        U, V = _uniform(seed, 2, case["m"], case["k"]), _uniform(seed, 3, case["n"], case["k"])
        return {"error": float((M - U @ V.T).norm() / M.norm())}
    if case["count"] * case["steps"] > 1300:
        return None  # hundreds of small problems for many iterations: minutes
    got = []
    for i, s, M in _batch_inputs(case, seed):
        c = dict(case, k=s["k"], d=s["d"], dv=s["d_v"], sketch="gaussian", inner=1)
        got.append(_iterate(c, M, case["steps"], s["seed"]))
    return {"U": torch.cat([u.reshape(-1) for u, _ in got]).cpu().numpy(),
            "V": torch.cat([v.reshape(-1) for _, v in got]).cpu().numpy()}
