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
