"""Candidates scored together (batched tuning) against each scored alone: a batch runs
the same arithmetic per candidate, so the scores are equal. d = 16 and 60 take the
small tiles, 64 and 100 the large; 200 labels at d = 100 need more than the batch's
buffer bound, so five candidates run in several batches; k = 0 candidates join the
propagated ones; a bad row index is refused as before."""
import numpy as np
import pytest
import torch

from paper_2302_07084_gb300 import lne, synth
from gpu_common import make_params

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2302_07084_gb300 import build
    build.build()
    c = lne.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("d,L", [(16, 1), (16, 7), (60, 5), (64, 5), (100, 200)])
def test_scores_equal_single_runs(ctx, d, L):
    g = synth.sbm(1300, 5, 0.05, 0.01, seed=d + L)
    rng = np.random.default_rng(L)
    labels = (rng.random((g.n, L)) < 0.3).astype(np.uint8)
    labels[:, 0] |= labels.sum(1) == 0
    perm = rng.permutation(g.n)
    lab, tr, te = (torch.as_tensor(a).cuda() for a in (labels, perm[:1000], perm[1000:]))
    cands = [make_params(3, np.full(3, 1 / 3), 30.0 * g.n_arcs, d=d, oversample=8, q=1, k=k, theta=th, mu=0.2, seed=s)
             for k, th, s in [(3, 0.5, 1), (0, 0.5, 1), (5, 0.9, 1), (3, 0.4, 2), (0, 0.5, 2)]]
    dg = lne.DeviceGraph.from_graph(g)
    ma, mi, X = ctx.tune_batch(dg, cands, lab, tr, te, iters=3, want_embeddings=True)
    for j in range(len(cands)):
        assert ctx.macro_f1(X[j], lab, tr, te, iters=3) == (ma[j], mi[j]), j
    bad = tr.clone()
    bad[7] = g.n
    with pytest.raises(lne.LneError):
        ctx.tune_batch(dg, cands, lab, bad, te, iters=3)
    again = ctx.tune_batch(dg, cands, lab, tr, te, iters=3)
    assert np.array_equal(again[0], ma) and np.array_equal(again[1], mi)
