"""The batched propagation's timed tile choice is kept per what it was measured on: a graph
with a long row runs the merge kernel and must not take the choice timed on a graph of
short rows of the same size (a lane group per row, which ignores the CTA size). Counted in
traced products: the timing runs (three CTA sizes and a warm-up each, column blocks apart)
come on top of the chain's."""
import numpy as np
import pytest
import torch

from paper_2302_07084_gb300 import lne, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_07084_gb300 import build
    build.build()


def _graphs():
    n = 3000
    rng = np.random.default_rng(0)
    e = rng.integers(0, n, (26000, 2))
    e = np.unique(np.sort(e[e[:, 0] != e[:, 1]], axis=1), axis=0)
    short = synth.csr_from_edges(n, e[:, 0], e[:, 1])
    hub = np.stack([np.zeros(1000, np.int64), np.arange(1, 1001)], 1)
    e = np.unique(np.concatenate([e[1000:], hub]), axis=0)
    long = synth.csr_from_edges(n, e[:, 0], e[:, 1])
    assert np.diff(short[0]).max() <= 256 < np.diff(long[0]).max()
    assert int(np.log2(short[0][-1])) == int(np.log2(long[0][-1]))      # the same size buckets
    return [lne.DeviceGraph(p, i) for p, i in (short, long)]


def test_a_long_row_is_timed_by_itself():
    short, long = _graphs()
    n = 3000
    lab = torch.from_numpy((np.arange(n)[:, None] % 4 == np.arange(4)).astype(np.uint8)).cuda()
    idx = torch.arange(n, dtype=torch.int32, device="cuda")
    cands = [lne.Params(T=3, s=[1 / 3] * 3, samples=20.0 * short.nnz, d=32, k=k, seed=1) for k in (4, 6)]

    def products(ctx, g):
        ctx.trace(True)
        ctx.tune_batch(g, cands, lab, idx[::2].contiguous(), idx[1::2].contiguous())
        count = sum(t["regions"] for t in ctx.trace_read() if t["name"] == "graph_spmm")
        ctx.trace(False)
        return count

    a, b = lne.Context(0), lne.Context(0)
    alone = products(a, long)
    first = products(b, short)
    after = products(b, long)
    again = products(b, long)
    assert after == alone and again < alone and first > 0
    a.close()
    b.close()
