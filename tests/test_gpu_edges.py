"""Sizes at the edges of tiles and remainders, against plain FP64 NumPy with
rounding bounds on every entry."""
import numpy as np
import pytest

from gpu_util import bound_ratio, np64, to_dev
from synth import lda_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gb():
    import torch
    import __graft_entry__ as g
    g.build()
    import paper_2106_12060_gb300 as m
    torch.cuda.set_device(0)
    return m


@pytest.mark.parametrize("n,d,l,k", [(40, 1, 2, 1), (130, 31, 3, 2), (777, 97, 5, 4), (1031, 129, 21, 20),
                                     (1100, 1024, 64, 20)])
def test_class_tables_and_fda_pass_f64(gb, n, d, l, k):
    """Class means (sums over the row chunks, their remainders) and the FP64
    FDA pass, whose class-mean correction is the means times Phi over every
    remainder of d.  Means: a sum of n_c terms in FP64.  Pass: chains of d
    and n terms and the l-term correction in FP64."""
    import torch
    P = lda_problem(n, d, l, dtype="f64", seed=d)
    y = P["y"]
    plan = gb.lda_plan(n, d, l, k, "f64", gb.default_options(max_iter=1))
    gb.lda_solve(plan, to_dev(P["X"], "f64"), torch.from_numpy(y).cuda(), 1e-1)
    X = P["X64"]
    M = np.stack([X[y == c].mean(0) for c in range(l)])
    aM = np.stack([np.abs(X[y == c]).mean(0) for c in range(l)])
    eps = 2.0 ** -53
    got = np64(gb.query(plan, gb.Q_CLASS_MEANS)).reshape(l, d)
    assert bound_ratio(got, M, aM, 2 * (n + 2) * eps) <= 1.0
    Phi = np.random.default_rng(d + 1).standard_normal((d, 2 * k))
    G, _, Gram = gb.fused_pass(plan, torch.from_numpy(Phi).cuda())
    W = (X - M[y]) @ Phi
    aW = (np.abs(X) + aM[y]) @ np.abs(Phi)
    gamma = 4 * (n + 2 * d + l + 4) * eps
    assert bound_ratio(np64(G), (X - M[y]).T @ W, (np.abs(X) + aM[y]).T @ aW, gamma) <= 1.0
    assert bound_ratio(np64(Gram), W.T @ W, aW.T @ aW, gamma) <= 1.0


def _layouts(a, tdt):
    """The same matrix contiguous, with rows padded to 16 bytes, with an odd
    row stride, and starting one element past an aligned address."""
    import torch
    t = torch.from_numpy(a).to(tdt).cuda()
    n, d = t.shape
    out = [t]
    for ld, off in (((d + 7) // 8 * 8, 0), (d + 1 + d % 2, 0), ((d + 7) // 8 * 8, 1)):
        buf = torch.full((n * ld + off,), float("nan"), dtype=tdt, device="cuda")
        v = buf[off:].view(n, ld)[:, :d]
        v.copy_(t)
        out.append(v)
    return out


@pytest.mark.parametrize("n,d", [(5, 1), (33, 3), (700, 31), (1500, 301), (2100, 516)])
def test_f32_copy_layouts_cca(gb, n, d):
    """The BF16 hi/lo copy of FP32 views (16-byte and element-wise loads, a
    ragged last chunk): the pass over it is bitwise the same for every layout
    of the same values, and within 2^-16 (the representation of data and Phi)
    plus FP32 accumulation of the exact products."""
    import torch
    rng = np.random.default_rng(d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    k = 1
    P = rng.standard_normal((d, 2 * k))
    got = []
    for x in _layouts(X, torch.float32):
        plan = gb.cca_plan(n, d, d, k, "f32", gb.default_options(warm_start=0))
        gb.cca_precondition(plan, x, x, 1e-1, 1e-1)
        Phi = torch.from_numpy(P).cuda()
        Gx, Gy, _ = gb.fused_pass(plan, Phi, Phi)
        got.append((np64(Gx), np64(Gy)))
    for g in got[1:]:
        assert np.array_equal(g[0], got[0][0]) and np.array_equal(g[1], got[0][1])
    X64 = X.astype(np.float64)
    W = np.hstack([X64 @ P, X64 @ P])
    aW = np.hstack([np.abs(X64) @ np.abs(P)] * 2)
    gamma = 4 * 2.0 ** -16 + 2 * (n + d + 8) * 2.0 ** -23
    assert bound_ratio(got[0][0], X64.T @ W, np.abs(X64).T @ aW, gamma) <= 1.0


@pytest.mark.parametrize("n,d,l", [(60, 3, 2), (900, 33, 5), (1400, 301, 10)])
def test_f32_copy_layouts_fda(gb, n, d, l):
    """The copy of the class-centred rows: bitwise the same pass for every
    layout, and within the same bound of the exact centred products."""
    import torch
    P = lda_problem(n, d, l, dtype="f32", seed=d)
    y = P["y"]
    k = 1
    Phi = np.random.default_rng(d + 1).standard_normal((d, 2 * k))
    got = []
    for x in _layouts(P["X"], torch.float32):
        plan = gb.lda_plan(n, d, l, k, "f32", gb.default_options(max_iter=1))
        gb.lda_solve(plan, x, torch.from_numpy(y).cuda(), 1e-1)
        got.append(np64(gb.fused_pass(plan, torch.from_numpy(Phi).cuda())[0]))
    for g in got[1:]:
        assert np.array_equal(g, got[0])
    X = P["X64"]
    M = np.stack([X[y == c].mean(0) for c in range(l)])
    Xc = X - M[y]
    W, aW = Xc @ Phi, np.abs(Xc) @ np.abs(Phi)
    gamma = 4 * 2.0 ** -16 + 2 * (n + d + 8) * 2.0 ** -23
    assert bound_ratio(got[0], Xc.T @ W, np.abs(Xc).T @ aW, gamma) <= 1.0


@pytest.mark.parametrize("dt", ["bf16", "f32", "f64"])
@pytest.mark.parametrize("n,d,s", [(3, 1, 2), (257, 33, 40), (2003, 131, 131), (40000, 260, 13000)])
def test_countsketch_sum_layouts(gb, dt, n, d, s):
    """Sums of buckets of every size (empty ones; more than 32 rows), columns
    that do not fill a lane's vector, more buckets than the shared-memory
    counters hold, and every row alignment, against exact row-order FP64
    sums: bitwise equal, since the order of a bucket's rows is fixed."""
    import torch
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32, "f64": torch.float64}[dt]
    rng = np.random.default_rng(n + d)
    X = rng.standard_normal((n, d)) * 10.0 ** rng.integers(-3, 4, (n, 1))
    X[rng.random((n, d)) < 0.05] = 0.0
    X = torch.from_numpy(X).to(tdt).double().numpy()
    h = rng.integers(0, s, n).astype(np.int32)
    if n > 1000:
        h[:100] = 1
        h[h == 0] = 2  # an empty bucket
    g = np.where(rng.random(n) < 0.5, -1, 1).astype(np.int8)
    ref = np.zeros((s, d))
    for i in range(n):
        ref[h[i]] += g[i] * X[i]
    for x in _layouts(X, tdt):
        plan = gb.cca_plan(n, d, d, 1, dt, gb.default_options(s=s, warm_start=0))
        gb.cca_precondition(plan, x, x, 1e3, 1e3, torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda())
        assert np.array_equal(np64(gb.query(plan, gb.Q_SKETCH_X)).reshape(s, d), ref)


@pytest.mark.parametrize("dt", ["bf16", "f32"])
@pytest.mark.parametrize("n,dx,dy,k", [(9, 1, 2, 1), (64, 8, 7, 3), (513, 9, 130, 9), (1300, 121, 17, 12),
                                       (1290, 129, 520, 13), (2050, 1024, 41, 20)])
def test_tc_pass_sums(gb, dt, n, dx, dy, k):
    """Views whose rows do not fill a block of the slab sums, every split of
    the slabs over the threads, one and two column groups: G and the Gram
    against the exact products at the rounded Phi, within 2^-16 of W (its
    hi + lo operand) and FP32 accumulation."""
    import torch
    rng = np.random.default_rng(n + k)
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32}[dt]
    data = []
    for d in (dx, dy):
        t = torch.zeros(n, (d + 7) // 8 * 8, dtype=tdt, device="cuda")[:, :d]
        t.copy_(torch.from_numpy(rng.standard_normal((n, d))))
        data.append(t)
    P = [rng.standard_normal((d, 2 * k)) for d in (dx, dy)]
    plan = gb.cca_plan(n, dx, dy, k, dt, gb.default_options(warm_start=0))
    gb.cca_precondition(plan, *data, 1.0, 1.0)
    Gx, Gy, Gram = (np64(t) for t in gb.fused_pass(plan, *(torch.from_numpy(p).cuda() for p in P)))
    Z = [np64(t) for t in data]
    W = np.hstack([z @ p for z, p in zip(Z, P)])
    aW = np.hstack([np.abs(z) @ np.abs(p) for z, p in zip(Z, P)])
    gamma = 6 * 2.0 ** -16 + 2 * (n + dx + dy + 8) * 2.0 ** -23
    for G, z in ((Gx, Z[0]), (Gy, Z[1])):
        assert bound_ratio(G, z.T @ W, np.abs(z).T @ aW, gamma) <= 1.0
    ref = np.vstack([np.abs(p).T @ (np.abs(z).T @ aW) for p, z in zip(P, Z)])
    assert bound_ratio(Gram, W.T @ W, ref, gamma) <= 1.0


@pytest.mark.parametrize("n,dx,dy,k", [(2, 1, 1, 1), (15, 9, 3, 2), (70, 65, 33, 9), (1000, 128, 31, 11),
                                       (5000, 260, 64, 20)])
def test_pass_f64_edges(gb, n, dx, dy, k):
    """The FP64 pass at row counts around its tiles and chunks, inner
    dimensions around its steps and every column count class: chains of dx +
    dy + n terms in FP64, entrywise."""
    import torch
    rng = np.random.default_rng(n + k)
    X, Y = rng.standard_normal((n, dx)), rng.standard_normal((n, dy))
    P = [rng.standard_normal((d, 2 * k)) for d in (dx, dy)]
    plan = gb.cca_plan(n, dx, dy, k, "f64", gb.default_options(warm_start=0))
    gb.cca_precondition(plan, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), 1.0, 1.0)
    Gx, Gy, Gram = (np64(t) for t in gb.fused_pass(plan, *(torch.from_numpy(p).cuda() for p in P)))
    W = np.hstack([X @ P[0], Y @ P[1]])
    aW = np.hstack([np.abs(X) @ np.abs(P[0]), np.abs(Y) @ np.abs(P[1])])
    gamma = 4 * (n + dx + dy + 8) * 2.0 ** -53
    assert bound_ratio(Gx, X.T @ W, np.abs(X).T @ aW, gamma) <= 1.0
    assert bound_ratio(Gy, Y.T @ W, np.abs(Y).T @ aW, gamma) <= 1.0
    assert bound_ratio(Gram, W.T @ W, aW.T @ aW, gamma) <= 1.0
    assert np.array_equal(Gram, Gram.T)


@pytest.mark.parametrize("d,k", [(1, 1), (7, 3), (33, 10), (130, 20)])
def test_thin_products_f64(gb, d, k):
    """The FP64 products with R^{-1} (inner ranges cut at the diagonal): the
    warm start maps an orthonormal block back through R^{-1}, so R times it
    has orthonormal columns, to FP64 rounding times the condition of R."""
    import torch
    from synth import countsketch_draws
    n, s, lam = 8 * d + 40, 3 * d + 10, 1e-1
    rng = np.random.default_rng(d)
    X = rng.standard_normal((n, d))
    Y = 0.5 * X + rng.standard_normal((n, d))
    h, g = countsketch_draws(n, s, seed=3)
    plan = gb.cca_plan(n, d, d, k, "f64", gb.default_options(s=s, max_iter=1, gtol=0.0))
    gb.cca_precondition(plan, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), lam, lam,
                        torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda())
    for q, w in ((gb.Q_R_X, gb.Q_WARM_U), (gb.Q_R_Y, gb.Q_WARM_V)):
        R = np64(gb.query(plan, q)).reshape(d, d)
        A = R @ np64(gb.query(plan, w)).reshape(d, k)
        assert np.max(np.abs(A.T @ A - np.eye(k))) < 1e-10


@pytest.mark.parametrize("retraction", [0, 1])
@pytest.mark.parametrize("kind,d,k", [("cca", 1, 1), ("cca", 9, 2), ("cca", 40, 11), ("cca", 60, 17), ("cca", 64, 20),
                                      ("lda", 6, 1), ("lda", 30, 5), ("lda", 80, 20)])
def test_small_geometry_trajectory_f64(gb, kind, d, k, retraction):
    """Line search and direction (factors, Jacobi sweeps and Sylvester
    solves for odd and even k up to the largest): ten iterations of an FP64
    solve from a random start follow the oracle's Riemannian CG with the
    library's own R.  Both compute in FP64, so f agrees to rounding grown by
    the iterations (1e-9 relative), the accepted steps and the gradient norm
    to 1e-6."""
    import torch
    from oracle import lda as OL
    from oracle.cca import sigmas
    from oracle.problems import CCAProblem, FDAProblem
    from oracle.rcg import rcg
    n, iters, lam = 20 * d + 60, 10, 1e-1
    rng = np.random.default_rng(10 * d + k)
    mu = np.linspace(2.0, 1.0, k) if k > 1 else np.ones(1)
    opt = gb.default_options(warm_start=0, max_iter=iters, gtol=0.0, retraction=retraction)
    if kind == "cca":
        X, Y = rng.standard_normal((n, d)), rng.standard_normal((n, d + 1))
        Y[:, :d] += X * np.linspace(1.5, 0.2, d)
        starts = [rng.standard_normal((d, k)), rng.standard_normal((d + 1, k))]
        plan = gb.cca_plan(n, d, d + 1, k, "f64", opt)
        gb.cca_precondition(plan, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), lam, lam)
        gb.cca_solve(plan, mu=list(mu), U=torch.from_numpy(starts[0].copy()).cuda(),
                     V=torch.from_numpy(starts[1].copy()).cuda())
        prob = CCAProblem(*sigmas(X, Y, lam, lam), mu)
        dims = (d, d + 1)
    else:
        P = lda_problem(n, d, k + 1, dtype="f64", seed=d, var_range=(0.1, 1.0))
        starts = [rng.standard_normal((d, k))]
        plan = gb.lda_plan(n, d, k + 1, k, "f64", opt)
        gb.lda_solve(plan, to_dev(P["X"], "f64"), torch.from_numpy(P["y"]).cuda(), lam, mu=list(mu),
                     W=torch.from_numpy(starts[0].copy()).cuda())
        _, _, _, Yhat, Xhat = OL.class_stats(P["X64"], P["y"], k + 1)
        prob = FDAProblem(Yhat.T @ Yhat, Xhat.T @ Xhat + lam * np.eye(d), mu)
        dims = (d,)
    hist = np64(gb.query(plan, gb.Q_HISTORY)).reshape(-1, 3)
    Ms = []
    for q, m in zip((gb.Q_R_X, gb.Q_R_Y), dims):
        R = np64(gb.query(plan, q)).reshape(m, m)
        Ms.append(R.T @ R)
    ho = np.array(rcg(prob, Ms, starts, max_iter=iters, gtol=0.0,
                      retraction="polar" if retraction else "qr")["history"])
    m = len(ho)
    if k == d:  # U spans everything: f is constant and the steps are rounding
        m = 1
    assert m > 1 or k == d
    assert np.max(np.abs(hist[:m, 0] - ho[:, 0][:m]) / np.abs(ho[:m, 0])) < 1e-9
    if m > 1:
        assert np.max(np.abs(hist[1:m, 2] - ho[1:m, 2]) / np.abs(ho[1:m, 2])) < 1e-6
        assert np.max(np.abs(hist[:m, 1] - ho[:m, 1]) / np.abs(ho[:m, 1])) < 1e-6


@pytest.mark.parametrize("retraction", [0, 1])
@pytest.mark.parametrize("d,k", [(9, 1), (12, 2), (40, 11), (60, 17), (64, 20)])
def test_small_geometry_f32(gb, d, k, retraction):
    """Line search and direction of FP32 plans for odd and even k: the first
    iterations follow the oracle's Riemannian CG.  The pass is good to some
    2^-16 of the sums of |terms|, so f is held to 1e-3; a wrong factor,
    direction or coefficient changes it by far more."""
    import torch
    from oracle.cca import sigmas
    from oracle.problems import CCAProblem
    from oracle.rcg import rcg
    n, iters, lam = 20 * d + 60, 4, 1e-1
    rng = np.random.default_rng(10 * d + k)
    mu = np.linspace(2.0, 1.0, k) if k > 1 else np.ones(1)
    X, Y = rng.standard_normal((n, d)), rng.standard_normal((n, d + 1))
    Y[:, :d] += X * np.linspace(1.5, 0.2, d)
    X, Y = X.astype(np.float32), Y.astype(np.float32)
    starts = [rng.standard_normal((d, k)), rng.standard_normal((d + 1, k))]
    plan = gb.cca_plan(n, d, d + 1, k, "f32", gb.default_options(warm_start=0, max_iter=iters, gtol=0.0, refine=0,
                                                                 retraction=retraction))
    gb.cca_precondition(plan, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), lam, lam)
    gb.cca_solve(plan, mu=list(mu), U=torch.from_numpy(starts[0].copy()).cuda(),
                 V=torch.from_numpy(starts[1].copy()).cuda())
    hist = np64(gb.query(plan, gb.Q_HISTORY)).reshape(-1, 3)
    Ms = []
    for q, m in zip((gb.Q_R_X, gb.Q_R_Y), (d, d + 1)):
        R = np64(gb.query(plan, q)).reshape(m, m)
        Ms.append(R.T @ R)
    prob = CCAProblem(*sigmas(X.astype(np.float64), Y.astype(np.float64), lam, lam), mu)
    ho = np.array(rcg(prob, Ms, starts, max_iter=iters, gtol=0.0, retraction="polar" if retraction else "qr")["history"])
    m = min(len(ho), len(hist))
    assert m > 1
    assert np.max(np.abs(hist[:m, 0] - ho[:m, 0]) / np.abs(ho[:m, 0])) < 1e-3


@pytest.mark.parametrize("d,k", [(1, 1), (5, 2), (31, 3), (33, 9), (49, 11), (130, 20)])
def test_warm_start_blocks_f32(gb, d, k):
    """The warm start of FP32 plans (products in double-float form over odd
    and even column counts, orthonormalization, small singular value
    decomposition): U and V orthonormal in the sketched metric, and U^T S_xy V
    diagonal with descending entries, since it ends with a Rayleigh-Ritz step.
    The products carry 2^-44 per term, so 1e-10 leaves the condition of R."""
    import torch
    from synth import countsketch_draws
    n, s, lam = 8 * d + 40, 3 * d + 10, 1e-1
    rng = np.random.default_rng(d)
    X = rng.standard_normal((n, d)).astype(np.float32)
    Y = (0.5 * X + rng.standard_normal((n, d))).astype(np.float32)
    h, g = countsketch_draws(n, s, seed=3)
    plan = gb.cca_plan(n, d, d, k, "f32", gb.default_options(s=s))
    gb.cca_precondition(plan, torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), lam, lam,
                        torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda())
    S = [np64(gb.query(plan, q)).reshape(s, d) for q in (gb.Q_SKETCH_X, gb.Q_SKETCH_Y)]
    B = [np64(gb.query(plan, q)).reshape(d, k) for q in (gb.Q_WARM_U, gb.Q_WARM_V)]
    for Z, b in zip(S, B):
        assert np.max(np.abs(b.T @ (Z.T @ (Z @ b)) + lam * b.T @ b - np.eye(k))) < 1e-10
    C = (S[0] @ B[0]).T @ (S[1] @ B[1])
    sig = np.diag(C)
    assert np.max(np.abs(C - np.diag(sig))) < 1e-10
    assert np.all(sig > 0) and np.all(np.diff(sig) <= 0)


@pytest.mark.parametrize("dt", ["bf16", "f32", "f64"])
@pytest.mark.parametrize("n,d,s", [(3, 1, 2), (40, 33, 40), (100, 31, 60), (700, 5, 300), (5000, 65, 500),
                                   (40000, 33, 999), (270000, 3, 2000)])
def test_srht_sizes(gb, dt, n, d, s):
    """The SRHT at every class of its two stages' lengths (up to 2^9 and 2^10),
    ragged columns and padding rows.  A sample is a sum of +-x over the column
    by log2(n') levels of additions, in FP32 (BF16/FP32 data) or FP64."""
    import torch
    from oracle.sketch import srht_apply
    from synth import srht_draws
    n_pad = 1 << max(int(n - 1).bit_length(), 0)
    if dt == "f64" and n_pad > 1 << 18:
        pytest.skip("more than the FP64 transform takes")
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32, "f64": torch.float64}[dt]
    s = min(s, n_pad)
    X = torch.from_numpy(np.random.default_rng(n).standard_normal((n, d))).to(tdt).double().numpy()
    D, rows = srht_draws(n_pad, s, seed=3)
    gamma = (np.log2(n_pad) + 4) * (2.0 ** -53 if dt == "f64" else 2.0 ** -24)
    ref = np.broadcast_to(np.abs(X).sum(0) / np.sqrt(s), (s, d))
    for x in _layouts(X, tdt)[:3]:
        plan = gb.cca_plan(n, d, d, 1, dt, gb.default_options(sketch=gb.SRHT, s=s, warm_start=0))
        gb.cca_precondition(plan, x, x, 1e3, 1e3, torch.from_numpy(rows).cuda(), torch.from_numpy(D).cuda())
        got = np64(gb.query(plan, gb.Q_SKETCH_X)).reshape(s, d)
        assert bound_ratio(got, srht_apply(X, D, rows), ref, gamma) <= 1.0


@pytest.mark.parametrize("d", [1, 15, 16, 17, 31, 32, 33, 48, 64, 65, 81, 260])
def test_factor_blocks_f32(gb, d):
    """R of FP32 plans at sizes around the 32-column panels and the 16-row
    tiles of the trailing update: upper, positive diagonal, R^T R equal to the
    sketch's Gram.  Gram: s terms of 2^-44 each; factor: chains of d terms in
    FP64 and one inverse of a 32 x 32 block."""
    import torch
    from synth import countsketch_draws
    n, s, lam = 4 * d + 20, 2 * d + 10, 1e-1
    X = np.random.default_rng(d).standard_normal((n, d)).astype(np.float32)
    h, g = countsketch_draws(n, s, seed=5)
    plan = gb.cca_plan(n, d, d, 1, "f32", gb.default_options(s=s, warm_start=0))
    x = torch.from_numpy(X).cuda()
    gb.cca_precondition(plan, x, x, lam, lam, torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda())
    S = np64(gb.query(plan, gb.Q_SKETCH_X)).reshape(s, d)
    ref = np.abs(S).T @ np.abs(S) + lam * np.eye(d)
    for q in (gb.Q_R_X, gb.Q_R_Y):  # the two views are factored side by side
        R = np64(gb.query(plan, q)).reshape(d, d)
        assert np.all(np.tril(R, -1) == 0) and np.all(np.diag(R) > 0)
        assert bound_ratio(R.T @ R, S.T @ S + lam * np.eye(d), ref, (s + 4 * d) * 2.0 ** -44) <= 1.0


@pytest.mark.parametrize("dt", ["bf16", "f32"])
@pytest.mark.parametrize("n,dx,dy,k", [(14, 13, 13, 13), (66, 64, 65, 14), (520, 513, 1, 1), (650, 385, 640, 16),
                                       (1025, 1024, 1024, 2), (30011, 128, 24, 20)])
def test_two_sweep_pass(gb, dt, n, dx, dy, k):
    """The two-sweep pass where the one-sweep kernel cannot hold the columns
    or the views: tiles and boxes of one row or column, every number of blocks
    per view, alone and in a batch with a second plan (other slab counts),
    within the bound of test_tc_pass_sums."""
    import torch
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32}[dt]
    plans, Phis, refs = [], [], []
    for i, (m, a, b, kk) in enumerate(((n, dx, dy, k), (n + 70, dy, dx, k))):
        rng = np.random.default_rng(n + k + i)
        data = []
        for d in (a, b):
            t = torch.zeros(m, (d + 7) // 8 * 8, dtype=tdt, device="cuda")[:, :d]
            t.copy_(torch.from_numpy(rng.standard_normal((m, d))))
            data.append(t)
        P = [rng.standard_normal((d, 2 * kk)) for d in (a, b)]
        plan = gb.cca_plan(m, a, b, kk, dt, gb.default_options())
        gb.cca_precondition(plan, *data, 1.0, 1.0)
        Z = [np64(t) for t in data]
        W = np.hstack([z @ p for z, p in zip(Z, P)])
        aW = np.hstack([np.abs(z) @ np.abs(p) for z, p in zip(Z, P)])
        plans.append((plan, data))
        Phis.append([torch.from_numpy(p).cuda() for p in P])
        refs.append((np.vstack([z.T @ W for z in Z]), np.vstack([np.abs(z).T @ aW for z in Z]), W.T @ W,
                     np.vstack([np.abs(p).T @ (np.abs(z).T @ aW) for p, z in zip(P, Z)]),
                     6 * 2.0 ** -16 + 2 * (m + a + b + 8) * 2.0 ** -23))
    batch = gb.Batch([p for p, _ in plans])
    Gb, Mb = gb.batch_fused_pass(batch, [f[0] for f in Phis], [f[1] for f in Phis])
    for i, (plan, _) in enumerate(plans):
        Gx, Gy, Gram = gb.fused_pass(plan, *Phis[i])
        G, aG, M, aM, gamma = refs[i]
        for got, gram in ((np.vstack([np64(Gx), np64(Gy)]), Gram), (np64(Gb[i]), Mb[i])):
            assert bound_ratio(got, G, aG, gamma) <= 1.0
            assert bound_ratio(np64(gram), M, aM, gamma) <= 1.0
    batch.close()


@pytest.mark.parametrize("n,d,k", [(80, 40, 13), (777, 385, 14), (5000, 1024, 20)])
def test_two_sweep_pass_fda(gb, n, d, k):
    """One view and more columns than one sweep holds; with a wait bound of
    one cycle (where a wait is long enough to run out) the pass gives up,
    drains what it has in flight and the solve reports it, and the next plan
    solves as before."""
    import torch
    l = k + 2
    P = lda_problem(n, d, l, dtype="f32", seed=d)
    x, y = to_dev(P["X"], "f32"), torch.from_numpy(P["y"]).cuda()
    if n == 5000:
        plan = gb.lda_plan(n, d, l, k, "f32", gb.default_options(wait_cycles=1, max_iter=3))
        with pytest.raises(gb.GbccaError) as e:
            gb.lda_solve(plan, x, y, 1e-1)
        assert e.value.code == gb.ERR_TIMEOUT
        plan.close()
    plan = gb.lda_plan(n, d, l, k, "f32", gb.default_options(max_iter=1))
    gb.lda_solve(plan, x, y, 1e-1)
    Phi = np.random.default_rng(d + 1).standard_normal((d, 2 * k))
    G, _, Gram = gb.fused_pass(plan, torch.from_numpy(Phi).cuda())
    X = P["X64"]
    M = np.stack([X[P["y"] == c].mean(0) for c in range(l)])
    Xc = X - M[P["y"]]
    W, aW = Xc @ Phi, np.abs(Xc) @ np.abs(Phi)
    gamma = 6 * 2.0 ** -16 + 2 * (n + d + 8) * 2.0 ** -23
    assert bound_ratio(np64(G), Xc.T @ W, np.abs(Xc).T @ aW, gamma) <= 1.0
    assert bound_ratio(np64(Gram), W.T @ W, np.abs(Phi).T @ (np.abs(Xc).T @ aW), gamma) <= 1.0


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("n,dx,dy,s", [(20, 1, 2, 7), (600, 63, 9, 66), (400, 129, 64, 300), (900, 200, 321, 897),
                                       (12000, 40, 33, 9000)])
def test_sketch_grams(gb, dt, n, dx, dy, s):
    """Grams of the sketches: tiles and row windows with remainders, one and
    several ranges of rows, columns over many orders of magnitude with a zero
    and an outlier row.  R^T R against the sketch's own Gram: entries are
    scaled to their columns, so the bound is 2^-46 of the columns' norms plus
    the factorization's chain of d terms."""
    import torch
    from synth import countsketch_draws
    rng = np.random.default_rng(dx)
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16}[dt]
    lam = 1e-30
    data = []
    for d in (dx, dy):
        Z = rng.standard_normal((n, d)) * 10.0 ** rng.integers(-9, 9, d)
        Z[3] *= 1e4
        Z[5] = 0.0
        data.append(torch.from_numpy(Z).to(tdt).cuda())
    h, g = countsketch_draws(n, s, seed=5)
    plan = gb.cca_plan(n, dx, dy, 1, dt, gb.default_options(s=s, warm_start=0))
    gb.cca_precondition(plan, *data, lam, lam, torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda())
    for qs, qr, d in ((gb.Q_SKETCH_X, gb.Q_R_X, dx), (gb.Q_SKETCH_Y, gb.Q_R_Y, dy)):
        S = np64(gb.query(plan, qs)).reshape(s, d)
        R = np64(gb.query(plan, qr)).reshape(d, d)
        nrm = np.linalg.norm(S, axis=0)
        # NumPy's own sum of s terms is in FP64
        assert bound_ratio(R.T @ R, S.T @ S, np.outer(nrm, nrm), 2.0 ** -46 + (s + 4 * d) * 2.0 ** -53) <= 1.0


def test_sketch_gram_rejects_overflow(gb):
    """A sketch beyond the FP32 range, or not finite, is reported as before."""
    import torch
    n, d = 64, 5
    for bad in (float("inf"), float("nan")):
        X = np.random.default_rng(0).standard_normal((n, d)).astype(np.float32)
        X[7, 2] = bad
        x = torch.from_numpy(X).cuda()
        plan = gb.cca_plan(n, d, d, 1, "f32", gb.default_options(warm_start=0))
        with pytest.raises(gb.GbccaError):
            gb.cca_precondition(plan, x, x, 1e-1, 1e-1)


@pytest.mark.parametrize("d", [400, 640])
def test_wide_f64_dispatch(gb, d):
    """FP64 plans beyond the lines of their dispatch rules: thin products
    whose operands do not fit shared memory, and a pass with so many blocks of
    columns that a CTA takes 32 of them."""
    test_thin_products_f64(gb, d, 20)
    test_pass_f64_edges(gb, 3000, d + 60, 300, 3)


def _refused(call):
    """Status of a call: True if it reported a factor that is not SPD, False
    if it went through; anything else is an error."""
    import paper_2106_12060_gb300 as gb
    try:
        call()
    except gb.GbccaError as e:
        assert e.code == gb.ERR_NOT_SPD
        return True
    return False


@pytest.mark.parametrize("dt", ["f32", "bf16"])
@pytest.mark.parametrize("n,d,s", [(64, 5, 40), (900, 65, 700)])
def test_sketch_gram_range(gb, dt, n, d, s):
    """Sketches whose products leave the FP32 range, which the rest of a plan
    shares: one column of 1e21 beside columns of order one, everything of that
    size, and squares that vanish without a ridge are refused by both forms of
    the Gram; and over columns of 2^58 to 2^68 both refuse the same ones."""
    import torch
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16}[dt]
    X = np.random.default_rng(d).standard_normal((n, d))

    def cca(Z, lam, tc):
        x = torch.from_numpy(Z).to(tdt).cuda()
        plan = gb.cca_plan(n, d, d, 1, dt, gb.default_options(s=s, tensor_cores=tc, warm_start=0))
        return _refused(lambda: gb.cca_precondition(plan, x, x, lam, lam))

    for tc in (1, 0):
        assert not cca(X, 1e-1, tc)
        assert not cca(X * 1e15, 1e-1, tc)
        big = X.copy()
        big[:, 2] *= 1e21
        assert cca(big, 1e-1, tc)
        assert cca(X * 1e22, 1e-1, tc)
        assert cca(X * 1e-26, 0.0, tc)
        assert not cca(X * 1e-26, 1e-1, tc)
    verdicts = []
    for e in np.arange(58, 68, 0.25):
        col = X.copy()
        col[:, 3] *= 2.0 ** e
        verdicts.append(cca(col, 1e-1, 1))
        assert verdicts[-1] == cca(col, 1e-1, 0)
    assert not verdicts[0] and verdicts[-1]


def test_fda_sketch_range(gb):
    """The same for FDA: data of 1e22 are refused, data of 1e15 are not, by
    both forms of the Gram."""
    import torch
    n, d, l = 300, 9, 3
    P = lda_problem(n, d, l, dtype="f32", seed=1)
    y = torch.from_numpy(P["y"]).cuda()
    for tc in (1, 0):
        for scale, refused in ((1.0, False), (1e15, False), (1e22, True)):
            x = torch.from_numpy((P["X64"] * scale).astype(np.float32)).cuda()
            plan = gb.lda_plan(n, d, l, 2, "f32", gb.default_options(max_iter=1, tensor_cores=tc))
            assert _refused(lambda: gb.lda_solve(plan, x, y, 1e-1)) == refused


@pytest.mark.parametrize("dt", ["bf16", "f32", "f64"])
@pytest.mark.parametrize("k", [2, 14])
def test_rebind_row_stride(gb, dt, k):
    """One plan bound to the same addresses with another row stride: the pass
    (one and two sweeps) and a solve replayed from a captured graph read the
    data as bound, so they give what a new plan gives, bitwise."""
    import torch
    n, dx, dy = 900, 40, 32
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32, "f64": torch.float64}[dt]
    rng = np.random.default_rng(k)
    buf = [torch.from_numpy(rng.standard_normal(n * 64)).to(tdt).cuda() for _ in range(2)]
    Phi = [torch.from_numpy(rng.standard_normal((d, 2 * k))).cuda() for d in (dx, dy)]

    def make():
        return gb.cca_plan(n, dx, dy, k, dt, gb.default_options(max_iter=8, gtol=0.0, check_every=4))

    def results(plan, lds):
        X, Y = (b.as_strided((n, d), (ld, 1)) for b, d, ld in zip(buf, (dx, dy), lds))
        gb.cca_precondition(plan, X, Y, 1e-1, 1e-1)
        return [np64(t) for t in (*gb.fused_pass(plan, *Phi), *gb.cca_solve(plan)[:3])]

    kept = make()
    for lds in ((64, 64), (48, 64), (48, 40), (45, 40)):
        for got, exp in zip(results(kept, lds), results(make(), lds)):
            assert np.array_equal(got, exp)


def test_srht_f64_longest(gb):
    """FP64 data of more than 2^18 rows, whose second stage takes 16 columns a
    CTA (a ragged last tile, tiles with one and with two halves): within the
    bound of test_srht_sizes."""
    import torch
    from oracle.sketch import srht_apply
    from synth import srht_draws
    n, s = 262145, 700
    n_pad = 1 << 19
    D, rows = srht_draws(n_pad, s, seed=3)
    for d in (3, 16, 50):
        X = np.random.default_rng(d).standard_normal((n, d))
        x = torch.from_numpy(X).cuda()
        plan = gb.cca_plan(n, d, d, 1, "f64", gb.default_options(sketch=gb.SRHT, s=s, warm_start=0))
        gb.cca_precondition(plan, x, x, 1e3, 1e3, torch.from_numpy(rows).cuda(), torch.from_numpy(D).cuda())
        ref = np.broadcast_to(np.abs(X).sum(0) / np.sqrt(s), (s, d))
        got = np64(gb.query(plan, gb.Q_SKETCH_X)).reshape(s, d)
        assert bound_ratio(got, srht_apply(X, D, rows), ref, (19 + 4) * 2.0 ** -53) <= 1.0


@pytest.mark.parametrize("dt", ["bf16", "f32", "f64"])
def test_first_error_is_reported(gb, dt):
    """Buckets outside the sketch leave it empty, so that without a ridge the
    factorization fails too: the call reports the buckets."""
    import torch
    n, d, s = 200, 4, 60
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32, "f64": torch.float64}[dt]
    x = torch.from_numpy(np.random.default_rng(0).standard_normal((n, d))).to(tdt).cuda()
    h = torch.full((n,), s, dtype=torch.int32, device="cuda")
    g = torch.ones(n, dtype=torch.int8, device="cuda")
    plan = gb.cca_plan(n, d, d, 1, dt, gb.default_options(s=s))
    for lam in (1.0, 0.0):
        with pytest.raises(gb.GbccaError) as e:
            gb.cca_precondition(plan, x, x, lam, lam, h, g)
        assert e.value.code == gb.ERR_INVALID_ARG
    gb.cca_precondition(plan, x, x, 1.0, 1.0)  # the flag does not outlive the call


@pytest.mark.parametrize("shapes", [((500, 40, 9), (600, 40, 12)), ((500, 200, 3), (600, 129, 11)),
                                    ((700, 600, 4), (800, 530, 17))])
def test_phi_image_after_nan(gb, shapes):
    """A batch of plans with different k lays their Phi images out alike; NaN
    in one call leaves nothing in the next, alone or in the batch: both give
    what they gave before, bitwise."""
    import torch
    rng = np.random.default_rng(0)
    plans, data, Phi = [], [], []
    for n, d, k in shapes:
        data.append([torch.zeros(n, (d + 7) // 8 * 8, dtype=torch.bfloat16, device="cuda")[:, :d] for _ in range(2)])
        for t in data[-1]:
            t.copy_(torch.from_numpy(rng.standard_normal((n, d))))
        plans.append(gb.cca_plan(n, d, d, k, "bf16", gb.default_options()))
        gb.cca_precondition(plans[-1], *data[-1], 1.0, 1.0)
        Phi.append([torch.from_numpy(rng.standard_normal((d, 2 * k))).cuda() for _ in range(2)])
    alone = [[np64(t) for t in gb.fused_pass(p, *f)] for p, f in zip(plans, Phi)]
    batch = gb.Batch(plans)

    def together(f):
        G, Gram = gb.batch_fused_pass(batch, [a for a, _ in f], [b for _, b in f])
        return [np64(t) for t in (*G, *Gram)]

    first = together(Phi)
    nan = [[torch.full_like(a, float("nan")) for a in f] for f in Phi]
    for _ in range(2):
        together(nan)
        for p, f, exp in zip(plans, Phi, alone):
            assert all(np.array_equal(np64(g), e) for g, e in zip(gb.fused_pass(p, *f), exp))
        for p, f in zip(plans, nan):
            gb.fused_pass(p, *f)
        assert all(np.array_equal(g, e) for g, e in zip(together(Phi), first))
    batch.close()


@pytest.mark.parametrize("dx,dy,k", [(40, 30, 5), (101, 37, 3), (5, 40, 3), (3, 3, 2)])
def test_warm_start_rounding_f32(gb, dx, dy, k):
    """The whitened cross matrix C of an FP32 plan's warm start, for views of
    condition about 1e4 and power iterations to their end: the pairs are
    singular pairs of C, up to sixteen times what the rounding of NumPy's FP64
    products of the same factors does to such a residual (their sums run in
    another order).  Products in double-float pairs are 2^9 times coarser."""
    import torch
    from synth import countsketch_draws
    big, lam, kap = np.longdouble, 1e-8, 1e4
    s = 4 * (dx + dy)
    n = 4 * s
    rng = np.random.default_rng(dx)
    m = min(dx, dy)
    z = rng.standard_normal((n, m)) * np.concatenate([np.linspace(3, 1, k), np.full(m - k, 0.1)])
    data = []
    for d in (dx, dy):
        A = 0.5 * rng.standard_normal((n, d))
        A[:, :m] += z
        A = (A * np.logspace(0, -np.log10(kap), d)) @ np.linalg.qr(rng.standard_normal((d, d)))[0]
        data.append(torch.from_numpy(A.astype(np.float32)).cuda())
    h, g = countsketch_draws(n, s, seed=3)
    plan = gb.cca_plan(n, dx, dy, k, "f32", gb.default_options(s=s, warm_iters=400))
    gb.cca_precondition(plan, *data, lam, lam, torch.from_numpy(h).cuda(), torch.from_numpy(g).cuda())
    S = [np64(gb.query(plan, q)).reshape(s, d) for q, d in ((gb.Q_SKETCH_X, dx), (gb.Q_SKETCH_Y, dy))]
    R = [np64(gb.query(plan, q)).reshape(d, d) for q, d in ((gb.Q_R_X, dx), (gb.Q_R_Y, dy))]
    A, B = (r.astype(big) @ np64(gb.query(plan, q)).reshape(-1, k).astype(big)
            for r, q in zip(R, (gb.Q_WARM_U, gb.Q_WARM_V)))

    def solve(r, M):  # r^{-T} M by forward substitution
        X = M.copy()
        for i in range(len(r)):
            X[i] = (X[i] - r[:i, i] @ X[:i]) / r[i, i]
        return X

    C = solve(R[0].astype(big), S[0].astype(big).T @ S[1].astype(big))
    C = solve(R[1].astype(big), C.T.copy()).T
    Ri = [np.linalg.inv(r) for r in R]
    E = Ri[0].T @ (S[0].T @ S[1]) @ Ri[1] - C
    sig = np.sum(A * (C @ B), axis=0)
    got = max(np.max(np.abs(C @ B - A * sig)), np.max(np.abs(C.T @ A - B * sig)))
    assert got <= 16 * max(np.max(np.abs(E @ B)), np.max(np.abs(E.T @ A)))


@pytest.mark.parametrize("dt", ["bf16", "f32"])
def test_two_sweep_long_ranges(gb, dt):
    """So many rows beside so few columns that a CTA's range of tiles is summed
    in several accumulations (alone and in a batch beside a short plan):
    entries of -1, 0 and 1 and a Phi that picks columns make every sum an
    integer below 2^24, so the products are exact."""
    import torch
    n, dx, dy, k = 350003, 32, 24, 20
    tdt = {"bf16": torch.bfloat16, "f32": torch.float32}[dt]
    g = torch.Generator(device="cuda").manual_seed(1)
    plans, data, Phi, exact = [], [], [], []
    for m in (n, 700):
        Z = [torch.randint(-1, 2, (m, d), generator=g, device="cuda").to(tdt) for d in (dx, dy)]
        P = [torch.zeros(d, 2 * k, dtype=torch.float64, device="cuda") for d in (dx, dy)]
        for p, step in zip(P, (7, 5)):
            c = torch.arange(2 * k, device="cuda")
            p[(c * step) % p.shape[0], c] = 1.0
        plan = gb.cca_plan(m, dx, dy, k, dt, gb.default_options())
        gb.cca_precondition(plan, *Z, 1.0, 1.0)
        W = torch.cat([z.double() @ p for z, p in zip(Z, P)], 1)
        plans.append(plan)
        data.append(Z)
        Phi.append(P)
        exact.append(([z.double().T @ W for z in Z], W.T @ W))
    batch = gb.Batch(plans)
    Gb, Mb = gb.batch_fused_pass(batch, [p[0] for p in Phi], [p[1] for p in Phi])
    for i, plan in enumerate(plans):
        (Ex, Ey), Em = exact[i]
        Gx, Gy, Gram = gb.fused_pass(plan, *Phi[i])
        assert torch.equal(Gx, Ex) and torch.equal(Gy, Ey) and torch.equal(Gram, Em)
        assert torch.equal(Gb[i], torch.cat([Ex, Ey])) and torch.equal(Mb[i], Em)
    batch.close()


@pytest.mark.parametrize("dt", ["f32", "bf16"])
def test_warm_start_range(gb, dt):
    """Cross products of the sketches that vanish in FP32 leave the warm start
    nothing to start from, whatever the ridge: both forms of the Gram report
    it, and neither does where the products are there."""
    import torch
    n, d = 300, 9
    tdt = {"f32": torch.float32, "bf16": torch.bfloat16}[dt]
    rng = np.random.default_rng(0)
    X = rng.standard_normal((n, d))
    Y = 0.5 * X + rng.standard_normal((n, d))
    for tc in (1, 0):
        for scale, lam, refused in ((1e-26, 1e-30, True), (1e-24, 1e-30, True), (1e-26, 1e-1, True),
                                    (1e-18, 1e-30, False), (1e-10, 1e-1, False), (1.0, 1e-1, False)):
            x, y = (torch.from_numpy(a * scale).to(tdt).cuda() for a in (X, Y))
            plan = gb.cca_plan(n, d, d, 2, dt, gb.default_options(tensor_cores=tc))
            assert _refused(lambda: gb.cca_precondition(plan, x, y, lam, lam)) == refused
