"""The calls whose speed and accuracy are followed on the GPU.

One data pass of an iteration (CCA in BF16, FP32 and FP64 storage, Fisher
LDA, a batch of plans), the preconditioner with its warm start, and whole
solves, each through the package's public calls.  A case is a dict of plain
values; `prepare` makes the inputs from a seed and the plan a program keeps,
`run` makes the call, `exact` gives the same results from plain FP64 torch.

Plans over BF16 and FP32 data accumulate in FP32, so their results, which the
calls hand back in FP64 containers, are taken on in single precision, the
type such a program holds its weights in; FP64 plans' results stay FP64.
"""
import math

import torch

import paper_2106_12060_gb300 as gb

_TORCH = {"bf16": torch.bfloat16, "f32": torch.float32, "f64": torch.float64}
_BYTES = {"bf16": 2, "f32": 4, "f64": 8}


def listed():
    return [
        # The smallest calls: one pass over a small problem, where launches
        # and latency are the cost (the narrowest shape of the batched mix,
        # and the small FP64 workload).
        dict(name="pass_bf16_small", call="pass", dtype="bf16", n=10000, dx=64, dy=64, k=1),
        dict(name="pass_f64_small", call="pass", dtype="f64", n=2000, dx=50, dy=40, k=5),
        # The pass of the tall workload: what every iteration repeats.
        dict(name="pass_bf16_tall", call="pass", dtype="bf16", n=262144, dx=512, dy=512, k=10),
        # FP32 features of uneven, odd widths and a ragged number of rows.
        dict(name="pass_f32_ragged", call="pass", dtype="f32", n=100003, dx=301, dy=77, k=3),
        # A wide view beside a narrow one with the most columns an iterate has.
        dict(name="pass_bf16_wide_k20", call="pass", dtype="bf16", n=200000, dx=1024, dy=256, k=20),
        # The FDA pass of the LDA workload.
        dict(name="pass_fda_f32", call="pass_fda", dtype="f32", n=100000, dx=784, l=10, k=9),
        # One pass of eight uneven plans solved together.
        dict(name="batch_pass_bf16", call="batch_pass", dtype="bf16", count=8, n=10000, n_top=100000, mix=1),
        # Binding new data: sketch, factor and warm start, for both sketches.
        dict(name="precondition_srht_bf16", call="precondition", dtype="bf16", n=262144, dx=512, dy=512, k=10,
             sketch="srht", scaled=True),
        dict(name="precondition_countsketch_f32", call="precondition", dtype="f32", n=300000, dx=384, dy=200, k=5,
             sketch="countsketch", scaled=False),
        # Whole problems from data to weights under a fixed budget of
        # iterations (a refresh of a model whose latency is bounded): the tall
        # ill-conditioned CCA, a small FP64 CCA, and Fisher LDA.
        dict(name="solve_bf16_tall", call="solve", dtype="bf16", n=262144, dx=512, dy=512, k=10, sketch="srht",
             scaled=True, budget=16),
        dict(name="solve_f64_small", call="solve", dtype="f64", n=2000, dx=50, dy=40, k=5, sketch="countsketch",
             scaled=False, budget=40),
        dict(name="solve_lda_f32", call="solve_lda", dtype="f32", n=100000, dx=784, l=10, k=9, budget=24),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    call = rng.choice(["pass", "pass", "pass", "pass", "pass_fda", "batch_pass", "precondition", "precondition", "solve"])
    if call == "batch_pass":
        return dict(call=call, dtype=rng.choice(["bf16", "f32"]), count=rng.randint(2, 8),
                    n=_log_int(rng, 2048, 10000), n_top=_log_int(rng, 20000, 100000), mix=rng.randint(2, 10 ** 6))
    if call == "pass_fda":
        d = _log_int(rng, 24, 1000)
        l = rng.randint(2, 21)
        return dict(call=call, dtype="f32", n=_log_int(rng, 3000, 120000), dx=d, l=l,
                    k=rng.randint(1, min(20, l - 1)))
    if call == "solve":
        return dict(call=call, dtype=rng.choice(["bf16", "f32"]), n=_log_int(rng, 30000, 200000),
                    dx=8 * rng.randint(6, 40), dy=8 * rng.randint(6, 40), k=rng.randint(2, 10),
                    sketch=rng.choice(["srht", "countsketch"]), scaled=rng.random() < 0.5, budget=16)
    dtype = rng.choice(["bf16", "bf16", "f32", "f32", "f64"])
    top, wide = (20000, 128) if dtype == "f64" else (200000, 1024)
    dx, dy = _log_int(rng, 24, wide), _log_int(rng, 24, wide)
    if rng.random() < 0.5:
        dx, dy = (dx + 7) // 8 * 8, (dy + 7) // 8 * 8
    case = dict(call=call, dtype=dtype, n=_log_int(rng, 2048, top), dx=dx, dy=dy, k=rng.randint(1, 20))
    if call == "precondition":
        case.update(sketch=rng.choice(["srht", "countsketch"]), scaled=rng.random() < 0.5)
    return case


# ------------------------------------------------------------------- inputs
def _generator(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) & 0x7FFFFFFF)
    return g


def _rows(n, d, dtype):
    """An n x d matrix whose rows start on 16-byte boundaries."""
    per = 16 // _BYTES[dtype]
    return torch.zeros(n, (d + per - 1) // per * per, dtype=_TORCH[dtype], device="cuda")[:, :d]


def _views(n, dx, dy, k, dtype, seed, scaled=False):
    """Two views of k shared factors plus noise, with canonical correlations
    spread from about 0.95 to 0.4; with `scaled` the columns fall from 1 to
    1e-4 (an ill-conditioned problem)."""
    g = _generator(seed)
    m = k
    work = torch.float64 if dtype == "f64" else torch.float32
    rho = 0.95 - 0.55 * torch.arange(m, dtype=work, device="cuda") / max(1, m - 1)
    strength = 0.5 * (rho / (1.0 - rho)).sqrt()
    A = [torch.linalg.qr(torch.randn(d, m, generator=g, device="cuda", dtype=work))[0].T * strength[:, None]
         for d in (dx, dy)]
    out = [_rows(n, d, dtype) for d in (dx, dy)]
    for r0 in range(0, n, 1 << 17):
        r1 = min(n, r0 + (1 << 17))
        z = torch.randn(r1 - r0, m, generator=g, device="cuda", dtype=work)
        for v, d in enumerate((dx, dy)):
            x = z @ A[v] + 0.5 * torch.randn(r1 - r0, d, generator=g, device="cuda", dtype=work)
            if scaled:
                x = x * 10.0 ** (-4.0 * torch.arange(d, dtype=work, device="cuda") / max(1, d - 1))
            out[v][r0:r1] = x.to(_TORCH[dtype])
    return out[0], out[1]


def _classes(n, d, l, seed):
    """FP32 rows of l classes (orthogonal means of decreasing length,
    within-class variances between 0.1 and 1) with shuffled balanced labels,
    and the ridge 1e-6 tr(S_w) / d."""
    g = _generator(seed)
    length = 4.0 - 3.0 * torch.arange(l, device="cuda") / l
    means = torch.linalg.qr(torch.randn(d, l, generator=g, device="cuda"))[0].T * length[:, None]
    var = 10.0 ** (-torch.rand(d, generator=g, device="cuda"))
    y = (torch.arange(n, device="cuda") % l)[torch.randperm(n, generator=g, device="cuda")].to(torch.int32)
    X = means[y.long()] + torch.randn(n, d, generator=g, device="cuda") * var.sqrt()
    return X.contiguous(), y.contiguous(), 1e-6 * n * float(var.double().mean())


def _phi(d, k, g):
    return torch.randn(d, 2 * k, generator=g, device="cuda", dtype=torch.float64) / math.sqrt(d)


def _draws(case, seed):
    """Sketch randomness a program fixes to repeat a run."""
    g = _generator(seed + 7919)
    n, s = case["n"], _sketch_rows(case)
    if case["sketch"] == "srht":
        h = torch.randperm(_pad(n), generator=g, device="cuda")[:s].to(torch.int32)
        m = _pad(n)
    else:
        h = torch.randint(0, s, (n,), generator=g, device="cuda", dtype=torch.int32)
        m = n
    sign = (2 * torch.randint(0, 2, (m,), generator=g, device="cuda") - 1).to(torch.int8)
    return h.contiguous(), sign.contiguous()


def _pad(n):
    return 1 << (n - 1).bit_length()


def _sketch_rows(case):
    s = 4 * (case["dx"] + case["dy"])
    return min(s, _pad(case["n"]) if case["sketch"] == "srht" else case["n"])


def _ridge(case):
    return 1e-4 if case.get("scaled") else 1e-3


def _mix(case):
    """The uneven shapes (n, dx, dy, k) of a batch."""
    g = torch.Generator().manual_seed(case["mix"])
    dims, ks, out = (64, 128, 256, 512, 1024), (1, 5, 10, 20), []
    for _ in range(case["count"]):
        u = torch.rand(4, generator=g, dtype=torch.float64).tolist()
        n = int(round(math.exp(math.log(case["n"]) + u[0] * math.log(case["n_top"] / case["n"]))))
        n = max(n, 1024)
        out.append((n, dims[int(5 * u[1])], dims[int(5 * u[2])], ks[int(4 * u[3])]))
    return out


def _sketch_kind(case):
    return gb.SRHT if case["sketch"] == "srht" else gb.COUNTSKETCH


def prepare(case, seed):
    call, dtype = case["call"], case["dtype"]
    s = dict(case=case)
    if call == "pass":
        n, dx, dy, k = (case[f] for f in ("n", "dx", "dy", "k"))
        s["X"], s["Y"] = _views(n, dx, dy, k, dtype, seed)
        g = _generator(seed + 104729)
        s["Px"], s["Py"] = _phi(dx, k, g), _phi(dy, k, g)
        s["plan"] = gb.cca_plan(n, dx, dy, k, dtype, gb.default_options(warm_start=0))
        gb.cca_precondition(s["plan"], s["X"], s["Y"], 1e-3, 1e-3)
    elif call == "pass_fda":
        n, d, l, k = (case[f] for f in ("n", "dx", "l", "k"))
        s["X"], s["y"], s["lam"] = _classes(n, d, l, seed)
        s["Px"] = _phi(d, k, _generator(seed + 104729))
        s["plan"] = gb.lda_plan(n, d, l, k, dtype, gb.default_options(max_iter=1))
        gb.lda_solve(s["plan"], s["X"], s["y"], s["lam"])  # binds the data
    elif call == "batch_pass":
        g = _generator(seed + 104729)
        s["plans"], s["data"], s["Px"], s["Py"] = [], [], [], []
        for i, (n, dx, dy, k) in enumerate(_mix(case)):
            X, Y = _views(n, dx, dy, k, dtype, seed + 1000 * i)
            plan = gb.cca_plan(n, dx, dy, k, dtype, gb.default_options())
            gb.cca_precondition(plan, X, Y, 1e-3, 1e-3)
            s["plans"].append(plan)
            s["data"].append((X, Y))
            s["Px"].append(_phi(dx, k, g))
            s["Py"].append(_phi(dy, k, g))
        s["batch"] = gb.batch_create(s["plans"])
    elif call == "precondition":
        n, dx, dy, k = (case[f] for f in ("n", "dx", "dy", "k"))
        s["X"], s["Y"] = _views(n, dx, dy, k, dtype, seed, case["scaled"])
        s["h"], s["g"] = _draws(case, seed)
        s["plan"] = gb.cca_plan(n, dx, dy, k, dtype, gb.default_options(sketch=_sketch_kind(case)))
    elif call == "solve":
        n, dx, dy, k = (case[f] for f in ("n", "dx", "dy", "k"))
        s["X"], s["Y"] = _views(n, dx, dy, k, dtype, seed, case["scaled"])
        opt = dict(sketch=_sketch_kind(case), max_iter=case["budget"])
        if dtype != "f64":
            opt.update(gtol=0.0, rtol=1e-7, check_every=4, refine=2)
        s["plan"] = gb.cca_plan(n, dx, dy, k, dtype, gb.default_options(**opt))
    else:
        n, d, l, k = (case[f] for f in ("n", "dx", "l", "k"))
        s["X"], s["y"], s["lam"] = _classes(n, d, l, seed)
        s["plan"] = gb.lda_plan(n, d, l, k, dtype, gb.default_options(gtol=0.0, rtol=1e-7, max_iter=case["budget"]))
    return s


def run(s):
    case = s["case"]
    call = case["call"]
    if call == "pass":
        out = gb.fused_pass(s["plan"], s["Px"], s["Py"])
    elif call == "pass_fda":
        Gx, _, Gram = gb.fused_pass(s["plan"], s["Px"])
        out = (Gx, Gram)
    elif call == "batch_pass":
        G, Gram = gb.batch_fused_pass(s["batch"], s["Px"], s["Py"])
        out = (*G, *Gram)
    elif call == "precondition":
        p, ridge = s["plan"], _ridge(case)
        gb.cca_precondition(p, s["X"], s["Y"], ridge, ridge, s["h"], s["g"])
        out = tuple(gb.query(p, q) for q in (gb.Q_R_X, gb.Q_R_Y, gb.Q_WARM_U, gb.Q_WARM_V))
    elif call == "solve":
        p, ridge = s["plan"], _ridge(case)
        gb.cca_precondition(p, s["X"], s["Y"], ridge, ridge)
        out = gb.cca_solve(p)[:3]
    else:
        out = gb.lda_solve(s["plan"], s["X"], s["y"], s["lam"])[:2]
    return tuple(t.float() for t in out) if case["dtype"] != "f64" else tuple(out)


def work(case):
    """Bytes and operations a call cannot do without: the data once, the
    small inputs and outputs once, and the products of one pass (a solve: of
    its sketch, factors and one pass)."""
    b = _BYTES[case["dtype"]]
    call = case["call"]
    if call == "batch_pass":
        parts = [work(dict(call="pass", dtype=case["dtype"], n=n, dx=dx, dy=dy, k=k)) for n, dx, dy, k in _mix(case)]
        return {f: sum(p[f] for p in parts) for f in ("bytes", "flops")}
    n, dx, dy, k = case["n"], case["dx"], case.get("dy", 0), case["k"]
    D, views = dx + dy, 2 if dy else 1
    cols = 2 * k * views
    data = n * D * b
    sweep = 2.0 * n * D * 2 * k + 2.0 * n * D * cols
    if call in ("pass", "pass_fda"):
        return {"bytes": data + 8 * (D * 2 * k + D * cols + cols * cols), "flops": sweep + 2.0 * D * 2 * k * cols}
    s = _sketch_rows(case) if dy else min(n, 3 * dx)
    sketch = n * D * (math.log2(_pad(n)) if case.get("sketch") == "srht" else 2.0)
    factor = sum(s * d * d + d ** 3 / 3.0 for d in (dx, dy))
    if call == "precondition":
        return {"bytes": data + 8 * (dx * dx + dy * dy + D * k) + 5 * n, "flops": sketch + factor}
    return {"bytes": data + 8 * (D * k + k), "flops": sketch + factor + sweep}


# ------------------------------------------------------------- FP64 results
def _pass64(Z, P):
    """(Z_v^T W for every view, W^T W), W = [Z_v P_v], in row chunks."""
    n, cols = Z[0].shape[0], sum(p.shape[1] for p in P)
    G = [torch.zeros(z.shape[1], cols, dtype=torch.float64, device="cuda") for z in Z]
    Gram = torch.zeros(cols, cols, dtype=torch.float64, device="cuda")
    for r0 in range(0, n, 1 << 16):
        z = [t[r0:r0 + (1 << 16)].double() for t in Z]
        W = torch.cat([a @ p for a, p in zip(z, P)], 1)
        for g, a in zip(G, z):
            g += a.T @ W
        Gram += W.T @ W
    return G, Gram


def _gram64(A, B):
    out = torch.zeros(A.shape[1], B.shape[1], dtype=torch.float64, device="cuda")
    for r0 in range(0, A.shape[0], 1 << 16):
        out += A[r0:r0 + (1 << 16)].double().T @ B[r0:r0 + (1 << 16)].double()
    return out


def _upper(M, ridge):
    return torch.linalg.cholesky(M + ridge * torch.eye(M.shape[0], dtype=M.dtype, device=M.device)).T.contiguous()


def _centred(X, y, l):
    X = X.double()
    at = y.long()
    count = torch.bincount(at, minlength=l).double()
    means = torch.zeros(l, X.shape[1], dtype=torch.float64, device="cuda").index_add_(0, at, X) / count[:, None]
    return X - means[at], count.sqrt()[:, None] * (means - X.mean(0))


def _signs(U):
    top = U.gather(0, U.abs().argmax(0, keepdim=True))
    return torch.where(top < 0, -1.0, 1.0).to(U.dtype)


def _sketch64(Z, case, h, sign):
    s = _sketch_rows(case)
    if case["sketch"] == "countsketch":
        out = torch.zeros(s, Z.shape[1], dtype=torch.float64, device="cuda")
        return out.index_add_(0, h.long(), Z.double() * sign[:, None].double())
    m = _pad(case["n"])
    a = torch.zeros(m, Z.shape[1], dtype=torch.float64, device="cuda")
    a[:case["n"]] = Z.double()
    a *= sign[:, None].double()
    span = 1
    while span < m:  # Walsh-Hadamard butterflies
        a = a.view(m // (2 * span), 2, span, -1)
        a = torch.stack((a[:, 0] + a[:, 1], a[:, 0] - a[:, 1]), 1)
        span *= 2
    return a.reshape(m, -1)[h.long()] / math.sqrt(s)


def exact(case, seed):
    call, dtype = case["call"], case["dtype"]
    if call == "pass":
        X, Y = _views(case["n"], case["dx"], case["dy"], case["k"], dtype, seed)
        g = _generator(seed + 104729)
        P = (_phi(case["dx"], case["k"], g), _phi(case["dy"], case["k"], g))
        G, Gram = _pass64((X, Y), P)
        return G[0], G[1], Gram
    if call == "pass_fda":
        X, y, _ = _classes(case["n"], case["dx"], case["l"], seed)
        G, Gram = _pass64((_centred(X, y, case["l"])[0],), (_phi(case["dx"], case["k"], _generator(seed + 104729)),))
        return G[0], Gram
    if call == "batch_pass":
        g = _generator(seed + 104729)
        Gs, Grams = [], []
        for i, (n, dx, dy, k) in enumerate(_mix(case)):
            X, Y = _views(n, dx, dy, k, dtype, seed + 1000 * i)
            P = (_phi(dx, k, g), _phi(dy, k, g))
            G, Gram = _pass64((X, Y), P)
            Gs.append(torch.cat(G))
            Grams.append(Gram)
        return (*Gs, *Grams)
    if call == "precondition":
        views = _views(case["n"], case["dx"], case["dy"], case["k"], dtype, seed, case["scaled"])
        h, sign = _draws(case, seed)
        R = []
        for Z in views:
            SZ = _sketch64(Z, case, h, sign)
            R.append(_upper(SZ.T @ SZ, _ridge(case)).reshape(-1))
        return R[0], R[1], None, None  # the warm start has its own iteration
    if call == "solve":
        X, Y = _views(case["n"], case["dx"], case["dy"], case["k"], dtype, seed, case["scaled"])
        Rx, Ry = _upper(_gram64(X, X), _ridge(case)), _upper(_gram64(Y, Y), _ridge(case))
        C = torch.linalg.solve_triangular(Rx.T, _gram64(X, Y), upper=False)
        C = torch.linalg.solve_triangular(Ry.T, C.T, upper=False).T
        A, sigma, Bt = torch.linalg.svd(C)
        U = torch.linalg.solve_triangular(Rx, A[:, :case["k"]], upper=True)
        V = torch.linalg.solve_triangular(Ry, Bt[:case["k"]].T, upper=True)
        sg = _signs(U)
        return sigma[:case["k"]], U * sg, V * sg
    X, y, lam = _classes(case["n"], case["dx"], case["l"], seed)
    Xc, Yhat = _centred(X, y, case["l"])
    R = _upper(_gram64(Xc, Xc), lam)
    H = torch.linalg.solve_triangular(R.T, Yhat.T, upper=False)
    w, Q = torch.linalg.eigh(H.T @ H)
    w, Q = w.flip(0)[:case["k"]], Q.flip(1)[:, :case["k"]]
    W = torch.linalg.solve_triangular(R, (H @ Q) / w.sqrt(), upper=True)
    return w, W * _signs(W)
