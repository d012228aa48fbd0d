"""What the performance of this library is measured on: its adjoint rules as a
program calls them, over the sizes its configurations, tests and benchmark use.

A case is a dict of plain values.  ``prepare`` makes its inputs on the GPU
(from the seed alone) and the workspace or plan a program keeps, ``run`` is one
pass through the public entry points, ``exact`` the same outputs in 64-bit
torch arithmetic, and ``work`` the bytes and operations of one pass that no
implementation can do without.
"""
import math

import torch

from paper_2202_10297_gb300 import adpar as A
from paper_2202_10297_gb300 import autograd as AG
from paper_2202_10297_gb300.batch import Batch

DEV = "cuda"
DT = {"f32": torch.float32, "f64": torch.float64}
IT = {"i32": torch.int32, "i64": torch.int64}
ESZ = {"f32": 4, "f64": 8}
ISZ = {"i32": 4, "i64": 8}


def listed():
    return [
        # forward mode of a short linear recurrence: the smallest call of a
        # request loop, where launches and host time are the cost
        {"name": "scan_jvp_small", "kind": "scan_jvp", "op": "linrec", "dtype": "f32", "n": 4099},
        # adjoint of a product of 65536 factors, one of them zero (a likelihood
        # with a vanishing term): a single short call
        {"name": "reduce_mul_small", "kind": "reduce_mul", "dtype": "f64", "n": 65536, "zeros": 1},
        # adjoint of a long product in FP64: memory against integer arithmetic
        {"name": "reduce_mul_large", "kind": "reduce_mul", "dtype": "f64", "n": 1 << 26, "zeros": 0},
        # adjoint of a long first-order linear recurrence in FP32
        {"name": "scan_linrec_f32", "kind": "scan_vjp", "op": "linrec", "dtype": "f32", "n": 1 << 26},
        # the same in FP64 through autograd, forward and backward, odd length
        {"name": "scan_linrec_f64_autograd", "kind": "scan_autograd", "dtype": "f64", "n": 10000019},
        # a linear recurrence per channel over time steps (a recurrent layer)
        {"name": "scan_vec_linrec", "kind": "scan_vec", "dtype": "f32", "n": 8192, "d": 2048},
        # per-key products over skewed keys (reduce_by_index *), adjoint
        {"name": "hist_mul_zipf", "kind": "hist", "op": "mul", "n": 1 << 25, "m": 1 << 16, "dist": "zipf",
         "itype": "i32"},
        # per-key maxima over many keys (reduce_by_index max), adjoint and argmax
        {"name": "hist_max_uniform", "kind": "hist", "op": "max", "n": 1 << 26, "m": 1 << 22, "dist": "uniform",
         "itype": "i32"},
        # per-key linear recurrences (reduce_by_index by the general rule)
        # through autograd, forward and backward
        {"name": "hist_linrec_autograd", "kind": "hist_linrec", "n": 1 << 24, "m": 1 << 16, "dist": "zipf",
         "itype": "i32"},
        # scatter of updates into a large table through autograd
        {"name": "scatter_autograd", "kind": "scatter", "n": 1 << 26, "m": 1 << 24, "sorted": False, "itype": "i32"},
        # many instances of uneven length and mixed precision in one launch
        {"name": "batch_256", "kind": "batch", "nseg": 256, "lo": 8.0, "hi": 20.0, "plan": 3},
        # the k-means cost and its gradient in the centroids, through autograd
        {"name": "kmeans_256", "kind": "kmeans", "N": 1 << 20, "k": 256},
    ]


def _logsize(rng, lo, hi):
    """An integer spread over the logarithm of [2^lo, 2^hi]; two in three are odd."""
    n = int(round(2.0 ** rng.uniform(lo, hi)))
    return n | 1 if rng.random() < 2 / 3 else n


def draw(rng):
    kind = rng.choice(["scan_jvp", "reduce_mul", "scan_vjp", "scan_autograd", "scan_vec", "hist", "hist", "hist_linrec",
                       "scatter", "batch", "kmeans"])
    itype = rng.choice(["i32", "i32", "i32", "i64"])
    dist = rng.choice(["zipf", "uniform"])
    if kind == "scan_jvp":
        return {"kind": kind, "op": rng.choice(["linrec", "linrec", "max", "add"]), "dtype": rng.choice(["f32", "f64"]),
                "n": _logsize(rng, 10, 25)}
    if kind == "reduce_mul":
        return {"kind": kind, "dtype": rng.choice(["f32", "f64"]), "n": _logsize(rng, 10, 25.9),
                "zeros": rng.choice([0, 0, 1, 2])}
    if kind == "scan_vjp":
        return {"kind": kind, "op": rng.choice(["linrec", "add", "max"]), "dtype": "f32", "n": _logsize(rng, 10, 25.9)}
    if kind == "scan_autograd":
        return {"kind": kind, "dtype": rng.choice(["f32", "f64"]), "n": _logsize(rng, 10, 23)}
    if kind == "scan_vec":
        n = _logsize(rng, 7, 13)
        return {"kind": kind, "dtype": rng.choice(["f32", "f32", "f64"]), "n": n,
                "d": _logsize(rng, 5, 22.9 - math.log2(n))}
    if kind == "hist":
        return {"kind": kind, "op": rng.choice(["mul", "mul", "max", "max", "add"]), "n": _logsize(rng, 14, 24.9),
                "m": _logsize(rng, 8, 22), "dist": dist, "itype": itype}
    if kind == "hist_linrec":
        return {"kind": kind, "n": _logsize(rng, 12, 23.9), "m": _logsize(rng, 8, 22), "dist": dist, "itype": itype}
    if kind == "scatter":
        m = _logsize(rng, 10, 23.9)
        return {"kind": kind, "n": int(m * 2 ** rng.uniform(0.5, 2)), "m": m, "sorted": rng.random() < 0.3,
                "itype": itype}
    if kind == "batch":
        return {"kind": kind, "nseg": rng.randrange(8, 256), "lo": 8.0, "hi": rng.uniform(12, 19),
                "plan": rng.randrange(1 << 30)}
    return {"kind": "kmeans", "N": _logsize(rng, 10, 20), "k": 32 * rng.randrange(1, 9)}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _normal(g, *shape, dtype=torch.float32):
    return torch.randn(*shape, generator=g, dtype=dtype, device=DEV)


def _uniform(g, lo, hi, *shape, dtype=torch.float32):
    return torch.rand(*shape, generator=g, dtype=dtype, device=DEV) * (hi - lo) + lo


def _linrec(g, *shape, dtype):
    """Decaying recurrence: a in [0.9, 1], b and the two cotangents (or tangents) normal."""
    return [_uniform(g, 0.9, 1.0, *shape, dtype=dtype)] + [_normal(g, *shape, dtype=dtype) for _ in range(3)]


def _factors(g, n, dtype, spread):
    """Positive factors near 1 whose product over n of them stays representable:
    ln|product| has a standard deviation of at most `spread`."""
    s = min(0.3, spread / math.sqrt(max(n, 1)))
    return torch.exp(s * _normal(g, n, dtype=dtype))


def _bins(g, n, m, dist, itype):
    """Keys uniform or bounded Zipf(1.1) over m bins, 1 % of them out of range."""
    if dist == "uniform":
        inds = torch.randint(0, m, (n,), generator=g, device=DEV)
    else:
        cdf = torch.cumsum(torch.arange(1, m + 1, dtype=torch.float64, device=DEV) ** -1.1, 0)
        u = torch.rand(n, generator=g, dtype=torch.float64, device=DEV) * cdf[-1]
        inds = torch.clamp(torch.searchsorted(cdf, u, right=True), max=m - 1)
    r = torch.rand(n, generator=g, device=DEV)
    inds = torch.where(r < 0.005, torch.full_like(inds, -1), inds)
    inds = torch.where(r > 0.995, torch.full_like(inds, m), inds)
    return inds.to(IT[itype])


def _batch_plan(c):
    """Lengths, precisions and offsets (multiples of 4 elements) of the segments."""
    g = torch.Generator().manual_seed(c["plan"])
    lens = torch.round(2.0 ** (c["lo"] + (c["hi"] - c["lo"]) * torch.rand(c["nseg"], generator=g, dtype=torch.float64)))
    lens = [int(v) for v in lens]
    wide = [bool(v) for v in torch.rand(c["nseg"], generator=g) < 0.5]
    tot = {False: 0, True: 0}
    offs = []
    for n, w in zip(lens, wide):
        offs.append(tot[w])
        tot[w] += (n + 3) // 4 * 4
    return lens, wide, offs, {w: max(t, 4) for w, t in tot.items()}


def _inputs(c, seed):
    g = _gen(seed)
    kind = c["kind"]
    if kind in ("scan_vjp", "scan_jvp", "scan_autograd"):
        dt = DT[c["dtype"]]
        if c.get("op", "linrec") == "linrec":
            return _linrec(g, c["n"], dtype=dt)
        return [_normal(g, c["n"], dtype=dt), _normal(g, c["n"], dtype=dt)]
    if kind == "scan_vec":
        return _linrec(g, c["n"], c["d"], dtype=DT[c["dtype"]])
    if kind == "reduce_mul":
        a = _factors(g, c["n"], DT[c["dtype"]], 4.0)
        if c["zeros"]:
            a[torch.randperm(c["n"], generator=g, device=DEV)[:c["zeros"]]] = 0
        return [a, _normal(g, 1, dtype=DT[c["dtype"]])]
    if kind == "hist":
        n, m = c["n"], c["m"]
        inds = _bins(g, n, m, c["dist"], c["itype"])
        hsbar = _normal(g, m)
        if c["op"] != "mul":
            return [inds, hsbar, _normal(g, n)]
        # signed factors near 1 (ratios), a few of them zero
        vals = torch.exp(0.01 * _normal(g, n)) * (1 - 2 * torch.randint(0, 2, (n,), generator=g, device=DEV))
        vals[torch.randint(0, n, (8,), generator=g, device=DEV)] = 0
        return [inds, hsbar, vals]
    if kind == "hist_linrec":
        n, m = c["n"], c["m"]
        inds = _bins(g, n, m, c["dist"], c["itype"])
        return [inds, _uniform(g, 0.9, 1.0, n), _normal(g, n), _normal(g, m), _normal(g, m)]
    if kind == "scatter":
        is_ = torch.randperm(c["n"], generator=g, device=DEV)[:c["m"]]
        if c["sorted"]:
            is_ = torch.sort(is_).values
        return [_normal(g, c["n"]), is_.to(IT[c["itype"]]), _normal(g, c["m"]), _normal(g, c["n"])]
    if kind == "batch":
        lens, wide, offs, tot = _batch_plan(c)
        slabs = {}
        for w in (False, True):
            dt = torch.float64 if w else torch.float32
            n = tot[w]
            # the factors' spread follows each segment's length
            scale = torch.zeros(n, dtype=torch.float32, device=DEV)
            for ln, ww, o in zip(lens, wide, offs):
                if ww == w:
                    scale[o:o + ln] = min(0.3, 4.0 / math.sqrt(ln))
            slabs[w] = [torch.exp(scale * _normal(g, n)).to(dt)] + _linrec(g, n, dtype=dt)
        return [lens, wide, offs, slabs]
    if kind == "kmeans":
        return [_normal(g, c["N"], 32), _normal(g, c["k"], 32)]
    raise ValueError(kind)


# ----------------------------------------------------------- prepare and run
def prepare(case, seed):
    c = dict(case)
    x = _inputs(c, seed)
    kind = c["kind"]
    st = {"case": c, "x": x}
    if kind in ("scan_vjp", "scan_jvp"):
        op = A.OPS[c["op"]]
        rule = A.RULE_SCAN if kind == "scan_vjp" else A.RULE_SCAN | A.WS_MINIMAL
        st["work"] = A.workspace(A.adpar_workspace_size(rule, op, A.F64 if c["dtype"] == "f64" else A.F32, c["n"]))
        st["out"] = [torch.empty_like(x[0]) for _ in range(2 if c["op"] == "linrec" else 1)] + [None]
    elif kind == "scan_vec":
        dt = A.F64 if c["dtype"] == "f64" else A.F32
        st["work"] = A.workspace(A.adpar_workspace_size(A.RULE_SCAN_VEC, A.OP_LINREC, dt, c["n"], c["d"]))
        st["out"] = [torch.empty_like(x[0]) for _ in range(2)]
    elif kind == "reduce_mul":
        dt = A.F64 if c["dtype"] == "f64" else A.F32
        st["work"] = A.workspace(A.adpar_workspace_size(A.RULE_REDUCE, A.OP_MUL, dt, c["n"]))
        st["out"] = torch.empty_like(x[0])
    elif kind == "hist":
        st["work"] = A.workspace(A.adpar_workspace_size(A.RULE_HIST, A.OPS[c["op"]], A.F32, c["n"], c["m"]))
        st["out"] = torch.empty(c["n"], dtype=torch.float32, device=DEV)
    elif kind == "scan_autograd":
        x[0].requires_grad_()
        x[1].requires_grad_()
    elif kind == "hist_linrec":
        x[1].requires_grad_()
        x[2].requires_grad_()
    elif kind == "scatter":
        x[0].requires_grad_()
        x[2].requires_grad_()
    elif kind == "kmeans":
        x[1].requires_grad_()
    elif kind == "batch":
        lens, wide, offs, slabs = x
        outs = {w: [torch.zeros_like(slabs[w][0]) for _ in range(3)] for w in slabs}
        segs = []
        for n, w, o in zip(lens, wide, offs):
            cut = [t[o:o + n] for t in slabs[w] + outs[w]]
            segs.append(dict(zip(("x", "a", "b", "ybar_a", "ybar_b", "xbar", "abar", "bbar"), cut), ybar_prod=1.5))
        st["batch"] = Batch(segs, config=(1, 4, 1, 0))
        st["out"] = outs[False] + outs[True]
    return st


def run(state):
    c, x = state["case"], state["x"]
    kind = c["kind"]
    if kind == "scan_vjp":
        o = state["out"]
        if c["op"] == "linrec":
            return A.adpar_vjp_scan("linrec", x[0], x[2], b=x[1], ybar_b=x[3], abar=o[0], bbar=o[1],
                                    work=state["work"])[:2]
        return A.adpar_vjp_scan(c["op"], x[0], x[1], abar=o[0], work=state["work"])[0]
    if kind == "scan_jvp":
        o = state["out"]
        if c["op"] == "linrec":
            return A.adpar_jvp_scan("linrec", x[0], x[2], b=x[1], bdot=x[3], ysdot_a=o[0], ysdot_b=o[1],
                                    work=state["work"])[:2]
        return A.adpar_jvp_scan(c["op"], x[0], x[1], ysdot_a=o[0], work=state["work"])[0]
    if kind == "scan_autograd":
        ya, yb = AG.scan("linrec", x[0], x[1])
        ga, gb = torch.autograd.grad((ya, yb), (x[0], x[1]), (x[2], x[3]))
        return ya.detach(), yb.detach(), ga, gb
    if kind == "scan_vec":
        o = state["out"]
        return A.adpar_vjp_scan_vec("linrec", x[0], x[2], b=x[1], ybar_b=x[3], abar=o[0], bbar=o[1],
                                    work=state["work"])[:2]
    if kind == "reduce_mul":
        r = A.adpar_vjp_reduce("mul", x[0], x[1], abar=state["out"], want_y=True, work=state["work"])
        return r["abar"], r["y"]
    if kind == "hist":
        op = c["op"]
        r = A.adpar_vjp_hist(op, x[0], c["m"], x[1], vals=x[2], valsbar=state["out"], want_hs=op == "mul",
                             want_argidx=op == "max", work=state["work"])
        return {k: r[k] for k in ("valsbar", "hs", "argidx") if k in r}
    if kind == "hist_linrec":
        ha, hb = AG.reduce_by_index("linrec", x[1], x[0], c["m"], b=x[2])
        ga, gb = torch.autograd.grad((ha, hb), (x[1], x[2]), (x[3], x[4]))
        return ha.detach(), hb.detach(), ga, gb
    if kind == "scatter":
        ys = AG.scatter(x[0], x[1], x[2])
        gx, gv = torch.autograd.grad(ys, (x[0], x[2]), x[3])
        return ys.detach(), gx, gv
    if kind == "batch":
        state["batch"].run()
        return state["out"]
    loss = AG.kmeans_loss(x[0], x[1])
    (gc,) = torch.autograd.grad(loss, x[1])
    return loss.detach(), gc


# ------------------------------------------------------------------ work
def work(case):
    c = case
    kind = c["kind"]
    e = ESZ[c["dtype"]] if "dtype" in c else 4
    i = ISZ[c["itype"]] if "itype" in c else 4
    if kind in ("scan_vjp", "scan_jvp"):
        lin = c["op"] == "linrec"
        arrays = 6 if lin else (2 if c["op"] == "add" else 3)
        return {"bytes": arrays * e * c["n"], "flops": (10 if lin else 1) * c["n"]}
    if kind == "scan_autograd":  # a, b and two cotangents in; two outputs and two adjoints out
        return {"bytes": 8 * e * c["n"], "flops": 10 * c["n"]}
    if kind == "scan_vec":
        return {"bytes": 6 * e * c["n"] * c["d"], "flops": 10 * c["n"] * c["d"]}
    if kind == "reduce_mul":
        return {"bytes": 2 * e * c["n"], "flops": 2 * c["n"]}
    if kind == "hist":
        return {"bytes": ((i + 4) if c["op"] == "add" else (i + 8)) * c["n"] + 8 * c["m"],
                "flops": 2 * c["n"] if c["op"] == "mul" else 0}
    if kind == "hist_linrec":
        return {"bytes": (i + 16) * c["n"] + 16 * c["m"], "flops": 10 * c["n"]}
    if kind == "scatter":  # xs and the cotangent in, ys and xs's adjoint out; indices, vs in, its adjoint out
        return {"bytes": 16 * c["n"] + (i + 8) * c["m"], "flops": 0}
    if kind == "batch":  # 5 inputs and 3 outputs an element, half of the elements in FP64
        mean = (2.0 ** c["hi"] - 2.0 ** c["lo"]) / ((c["hi"] - c["lo"]) * math.log(2))
        return {"bytes": int(8 * 6 * mean * c["nseg"]), "flops": int(12 * mean * c["nseg"])}
    return {"bytes": 4 * 32 * (c["N"] + 2 * c["k"]), "flops": 2 * 32 * c["k"] * c["N"]}


# ------------------------------------------------------------------ exact
def _recur(co, d):
    """x_i = co_i x_{i-1} + d_i (x_{-1} = 0) over a 1-D FP64 array: rows of L
    consecutive elements side by side, then the rows' carries the same way."""
    n = d.numel()
    if n <= 64:
        x = torch.zeros_like(d)
        prev = torch.zeros((), dtype=d.dtype, device=d.device)
        for j in range(n):
            prev = co[j] * prev + d[j]
            x[j] = prev
        return x
    L = max(8, int(2 ** round(math.log2(n) / 2 - 1)))
    R = -(-n // L)
    pad = R * L - n
    ct = torch.nn.functional.pad(co, (0, pad)).view(R, L).t().contiguous()
    dt = torch.nn.functional.pad(d, (0, pad)).view(R, L).t().contiguous()
    for j in range(1, L):  # in place: dt becomes the local solution, ct the carry's factor
        dt[j].addcmul_(ct[j], dt[j - 1])
        ct[j].mul_(ct[j - 1])
    carry = _recur(ct[L - 1].clone(), dt[L - 1].clone())
    dt[:, 1:].addcmul_(ct[:, 1:], carry[:-1])
    return dt.t().reshape(-1)[:n]


def _linrec_exact(a, b, ya, yb, start):
    """(A, B, abar, bbar) of linear recurrences laid end to end; start marks the
    first element of each."""
    one = torch.ones_like(a)
    zero = torch.zeros_like(a)
    cf = torch.where(start, zero, a)
    Ai = _recur(cf, torch.where(start, a, zero))
    Bi = _recur(cf, b)
    nxt = torch.cat([cf[1:], cf.new_zeros(1)]).flip(0)  # a_{i+1}, 0 at a last element
    ra = _recur(nxt, ya.flip(0)).flip(0)
    rb = _recur(nxt, yb.flip(0)).flip(0)
    ap = torch.where(start, one, torch.cat([one[:1], Ai[:-1]]))
    bp = torch.where(start, zero, torch.cat([zero[:1], Bi[:-1]]))
    return Ai, Bi, ap * ra + bp * rb, rb


def _prod_exact(logs, neg, zero, seg, m, ybar):
    """Per segment the product, and per element ybar times the product of the
    segment's other elements, from sums of logarithms."""
    S = torch.zeros(m, dtype=torch.float64, device=DEV).index_add_(0, seg, logs)
    Z = torch.bincount(seg[zero], minlength=m)
    N = torch.bincount(seg[neg], minlength=m)
    sign = 1.0 - 2.0 * (N[seg] % 2).double()
    sign = torch.where(neg, -sign, sign)
    others = torch.where(zero, Z[seg] - 1, Z[seg])
    c = torch.exp(S[seg] - logs) * sign * ybar[seg]
    prod = torch.where(Z > 0, torch.zeros_like(S), torch.exp(S) * (1.0 - 2.0 * (N % 2).double()))
    return prod, torch.where(others > 0, torch.zeros_like(c), c)


def _log_abs(v):
    zero = v == 0
    return torch.log(torch.where(zero, torch.ones_like(v), v).abs()), v < 0, zero


def exact(case, seed):
    c = case
    kind = c["kind"]
    x = _inputs(c, seed)
    if kind in ("scan_vjp", "scan_jvp", "scan_autograd"):
        op = c.get("op", "linrec")
        x = [t.double() for t in x]
        n = c["n"]
        start = torch.zeros(n, dtype=torch.bool, device=DEV)
        start[0] = True
        if op == "linrec" and kind == "scan_jvp":
            a, b, ad, bd = x
            cf = torch.where(start, torch.zeros_like(a), a)
            Ai = _recur(cf, torch.where(start, a, torch.zeros_like(a)))
            Bi = _recur(cf, b)
            ap = torch.cat([Ai.new_ones(1), Ai[:-1]])
            bp = torch.cat([Bi.new_zeros(1), Bi[:-1]])
            return _recur(cf, ad * ap), _recur(cf, ad * bp + bd)
        if op == "linrec":
            Ai, Bi, ab, bb = _linrec_exact(*x, start)
            return (ab, bb) if kind == "scan_vjp" else (Ai, Bi, ab, bb)
        a, y = x
        if op == "add":
            return torch.cumsum(y, 0) if kind == "scan_jvp" else torch.cumsum(y.flip(0), 0).flip(0)
        run_max = torch.cummax(a, 0).values
        rec = start.clone()
        rec[1:] = a[1:] > run_max[:-1]
        pos = torch.cummax(torch.where(rec, torch.arange(n, device=DEV), torch.zeros(n, dtype=torch.int64, device=DEV)),
                           0).values
        if kind == "scan_jvp":
            return y[pos]
        return torch.zeros_like(a).index_add_(0, pos, y)
    if kind == "scan_vec":
        a, b, ya, yb = [t.double() for t in x]
        n = c["n"]
        Ap, Bp = torch.ones_like(a), torch.zeros_like(a)
        for j in range(1, n):
            torch.mul(a[j - 1], Ap[j - 1], out=Ap[j])
            torch.addcmul(b[j - 1], a[j - 1], Bp[j - 1], out=Bp[j])
        for j in range(n - 2, -1, -1):  # ya, yb become the return sweep's state
            ya[j].addcmul_(a[j + 1], ya[j + 1])
            yb[j].addcmul_(a[j + 1], yb[j + 1])
        return Ap * ya + Bp * yb, yb
    if kind == "reduce_mul":
        logs, neg, zero = _log_abs(x[0].double())
        S, nz = logs.sum(), int(zero.sum())
        sign = 1.0 - 2.0 * (neg.sum() % 2).double()
        ab = torch.exp(S - logs) * sign * torch.where(neg, -1.0, 1.0).double() * x[1].double()
        ab = torch.where((zero.long() == nz) if nz <= 1 else torch.zeros_like(zero), ab, torch.zeros_like(ab))
        return ab, (torch.exp(S) * sign if nz == 0 else torch.zeros_like(S)).reshape(1)
    if kind == "hist":
        inds, hsbar, vals = x[0].long(), x[1].double(), x[2].double()
        n, m = c["n"], c["m"]
        sel = ((inds >= 0) & (inds < m)).nonzero().view(-1)
        seg = inds[sel]
        vb = torch.zeros(n, dtype=torch.float64, device=DEV)
        if c["op"] == "add":
            vb[sel] = hsbar[seg]
            return {"valsbar": vb}
        if c["op"] == "mul":
            prod, cb = _prod_exact(*_log_abs(vals[sel]), seg, m, hsbar)
            vb[sel] = cb
            return {"valsbar": vb, "hs": prod}
        v = vals[sel]
        top = torch.full((m,), -math.inf, dtype=torch.float64, device=DEV).scatter_reduce_(0, seg, v, "amax")
        hit = v == top[seg]
        arg = torch.full((m,), n, dtype=torch.int64, device=DEV).scatter_reduce_(0, seg[hit], sel[hit], "amin")
        has = arg < n
        vb[arg[has]] = hsbar[has]
        return {"valsbar": vb, "argidx": None}
    if kind == "hist_linrec":
        inds = x[0].long()
        a, b, ha, hb = [t.double() for t in x[1:]]
        n, m = c["n"], c["m"]
        sel = ((inds >= 0) & (inds < m)).nonzero().view(-1)
        seg, order = torch.sort(inds[sel], stable=True)
        sel = sel[order]
        start = torch.ones_like(seg, dtype=torch.bool)
        start[1:] = seg[1:] != seg[:-1]
        last = torch.cat([start[1:], start[:1]])
        z = torch.zeros(seg.numel(), dtype=torch.float64, device=DEV)
        Ai, Bi, ab, bb = _linrec_exact(a[sel], b[sel], torch.where(last, ha[seg], z), torch.where(last, hb[seg], z),
                                       start)
        hs_a = torch.ones(m, dtype=torch.float64, device=DEV)
        hs_b = torch.zeros(m, dtype=torch.float64, device=DEV)
        hs_a[seg[last]] = Ai[last]
        hs_b[seg[last]] = Bi[last]
        ga, gb = torch.zeros_like(a), torch.zeros_like(a)
        ga[sel] = ab
        gb[sel] = bb
        return hs_a, hs_b, ga, gb
    if kind == "scatter":
        xs, is_, vs, g = x
        is_ = is_.long()
        ys = xs.double()
        ys[is_] = vs.double()
        gx = g.double()
        gv = gx[is_].clone()
        gx[is_] = 0
        return ys, gx, gv
    if kind == "batch":
        lens, wide, offs, slabs = x
        out = []
        for w in (False, True):
            xx, a, b, ya, yb = [t.double() for t in slabs[w]]
            n = xx.numel()
            start = torch.zeros(n, dtype=torch.bool, device=DEV)
            live = torch.zeros(n, dtype=torch.bool, device=DEV)
            for ln, ww, o in zip(lens, wide, offs):
                if ww == w:
                    start[o] = True
                    start[o + ln:o + (ln + 3) // 4 * 4] = True  # the gap to the next segment
                    live[o:o + ln] = True
            start[0] = True
            _, _, ab, bb = _linrec_exact(a, b, ya, yb, start)
            seg = torch.cumsum(start.long(), 0) - 1
            ns = int(seg[-1]) + 1
            _, xb = _prod_exact(*_log_abs(xx), seg, ns, torch.full((ns,), 1.5, dtype=torch.float64, device=DEV))
            out += [torch.where(live, t, torch.zeros_like(t)) for t in (xb, ab, bb)]
        return out
    X, C = x[0].double(), x[1].double()
    c2 = (C * C).sum(1)
    loss = torch.zeros((), dtype=torch.float64, device=DEV)
    grad = torch.zeros_like(C)
    for s in range(0, c["N"], 1 << 18):
        xc = X[s:s + (1 << 18)]
        best = torch.argmin(c2 - 2.0 * (xc @ C.t()), 1)
        diff = C[best] - xc
        loss += (diff * diff).sum()
        grad.index_add_(0, best, 2.0 * diff)
    return loss, grad
