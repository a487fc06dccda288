"""Macro-F1 at the sizes where its kernels change: 4 x 4 against 8 x 8 tiles
(d + 1 = 64 | 65), ragged tiles and 32-wide Cholesky panels, row blocks of 128
and stages of 32 rows with remainders, one label, and an ill-conditioned
Hessian (scaled features), which takes the FP64 factorisation. Against the
oracle: both solve the same strictly convex problem to convergence and score
the same rows; a margin within FP32 rounding (~1e-6 of the scores) of a tie may
fall either way, so one decision in the few hundred scored may differ:
tolerance 2 / (decisions per label)."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_07084_gb300 import lne

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2302_07084_gb300 import build
    build.build()
    c = lne.Context(0)
    yield c
    c.close()


def _case(n, d, L, seed, scale=1.0):
    rng = np.random.default_rng(seed)
    first = rng.integers(0, L, n)
    lab = np.zeros((n, L), np.uint8)
    lab[np.arange(n), first] = 1
    if L > 2:
        two = rng.random(n) < 0.3
        lab[np.arange(n)[two], rng.integers(0, L, n)[two]] = 1
    X = (0.7 * rng.normal(size=(L, d))[first] + rng.normal(size=(n, d))).astype(np.float32) * np.float32(scale)
    perm = rng.permutation(n).astype(np.int32)
    return X, lab, perm


@pytest.mark.parametrize("d,n_train,L", [(1, 40, 2), (7, 127, 3), (31, 128, 5), (32, 129, 4), (62, 300, 3),
                                         (63, 257, 2), (64, 300, 3), (95, 161, 2), (127, 300, 2), (128, 385, 3),
                                         (159, 400, 2), (20, 33, 1)])
def test_matches_oracle(ctx, d, n_train, L):
    n = n_train + 300
    X, lab, perm = _case(n, d, L, d + n_train)
    tr, te = perm[:n_train], perm[n_train:]
    ma, mi = ctx.macro_f1(torch.as_tensor(X).cuda(), torch.as_tensor(lab).cuda(), torch.as_tensor(tr).cuda(),
                          torch.as_tensor(te).cuda())
    wa, wi, _ = oracle.macro_f1(X, lab, tr, te)
    per_label = max(1, min(int(lab[te].sum(0).min()), len(te)))
    assert abs(ma - wa) <= 2.0 / per_label and abs(mi - wi) <= 2.0 / len(te), (ma, wa, mi, wi)


@pytest.mark.parametrize("scale,iters", [(3.0e3, 1), (3.0e3, 2), (1.0e5, 1)])
def test_ill_conditioned(ctx, scale, iters):
    """1 + C |X|^2 / 4 up to 1e12: the first Newton steps from 0 are compared
    (they are the solve with H = I + X^T X / 4)."""
    X, lab, perm = _case(700, 40, 3, 9, scale)
    X[:, 1] = X[:, 0] + X[:, 1] * np.float32(1e-3)   # nearly dependent columns
    tr, te = perm[:400], perm[400:]
    ma, mi = ctx.macro_f1(torch.as_tensor(X).cuda(), torch.as_tensor(lab).cuda(), torch.as_tensor(tr).cuda(),
                          torch.as_tensor(te).cuda(), iters=iters)
    wa, wi, _ = oracle.macro_f1(X, lab, tr, te, iters=iters)
    assert abs(mi - wi) <= 0.02 and abs(ma - wa) <= 0.02, (ma, wa, mi, wi)
