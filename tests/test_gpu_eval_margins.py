"""Macro-F1 on labels without signal, where the decisions hang on small differences of the
margins, at ragged Cholesky panels and tiles (d + 1 = 33, 65, 97, 129, 160). A row's
decision may differ from the FP64 oracle's only where its k-th and (k + 1)-th score are
closer than the margins' FP32 error: 1e-5 of the largest score (the products' rounding is
about 1e-6 of it). `ties` counts those rows, each of which moves one true positive, so
Micro-F1 by at most 1 / (decisions) and Macro-F1 by at most 2 / (L times the smallest F1
denominator / 2) twice. A weight matrix off by 1% past its first panel has to change more
rows than that, or the labels are too easy (checked on the oracle's own weights)."""
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


@pytest.mark.parametrize("d", [32, 64, 96, 128, 159])
def test_labels_without_signal(ctx, d):
    rng = np.random.default_rng(d)
    n_train, n_test, L = 700, 3000, 20
    n = n_train + n_test
    X = rng.normal(size=(n, d)).astype(np.float32)
    lab = np.zeros((n, L), np.uint8)
    lab[np.arange(n), rng.integers(0, L, n)] = 1
    lab[np.arange(n), rng.integers(0, L, n)] = 1
    perm = rng.permutation(n).astype(np.int32)
    tr, te = perm[:n_train], perm[n_train:]
    wa, wi, W = oracle.macro_f1(X, lab, tr, te)
    Xt, truth = np.hstack([X[te].astype(np.float64), np.ones((n_test, 1))]), lab[te].astype(bool)
    k = truth.sum(1)

    scores = Xt @ W
    order = -np.sort(-scores, axis=1)
    gap = order[np.arange(n_test), k - 1] - order[np.arange(n_test), k]
    ties = int((gap < 1e-5 * np.abs(scores).max()).sum())
    tol_micro = ties / k.sum()
    tol_macro = 2 * ties * 2.0 / (L * truth.sum(0).min())
    off = W.copy()
    off[min(32, d // 2):] *= 1.01
    changed = (oracle.predict_topk(Xt @ off, k) != oracle.predict_topk(scores, k)).any(1).sum()
    assert changed > ties, "labels too easy"
    ma, mi = ctx.macro_f1(torch.as_tensor(X).cuda(), torch.as_tensor(lab).cuda(), torch.as_tensor(tr).cuda(),
                          torch.as_tensor(te).cuda())
    assert abs(mi - wi) <= tol_micro + 1e-12 and abs(ma - wa) <= tol_macro + 1e-12, (ma, wa, mi, wi, ties)


@pytest.mark.parametrize("scale", [1.0, 5.0e17, 2.0e18])
def test_large_features(ctx, scale):
    """Features so large that the Hessian's sums pass FP32's range while every row block's
    partial sum is inside it: the scores are those of the same features at scale 1 (the
    penalty is negligible at either), as the oracle's are."""
    rng = np.random.default_rng(1)
    n, d, L = 12000, 24, 5
    first = rng.integers(0, L, n)
    lab = np.zeros((n, L), np.uint8)
    lab[np.arange(n), first] = 1
    X = ((0.3 * rng.normal(size=(L, d))[first] + rng.normal(size=(n, d))) * scale).astype(np.float32)
    perm = rng.permutation(n).astype(np.int32)
    tr, te = perm[:6000], perm[6000:]
    wa, wi, _ = oracle.macro_f1(X, lab, tr, te)
    ma, mi = ctx.macro_f1(torch.as_tensor(X).cuda(), torch.as_tensor(lab).cuda(), torch.as_tensor(tr).cuda(),
                          torch.as_tensor(te).cuda())
    # two decisions may fall the other way (ties within FP32 rounding)
    assert abs(mi - wi) <= 2.0 / len(te) and abs(ma - wa) <= 2.0 / lab[te].sum(0).min()
