"""Key-sort aggregation at the sizes where its tiles and passes change.

The sorted keys, their run lengths and the assembled CSR are whole numbers (and
values that depend on them alone), so everything is compared exactly with the
CPU oracle, or with the dense-table aggregation where that is the general path:

* totals of one key pair up to several sort tiles (6144 keys), on either side of
  a tile's edge and of a run-length chunk (1024 keys);
* vertex counts whose key bits end in, before and after a whole byte, so the
  mirrored sort (over the row bits alone) starts in the middle of one;
* runs of equal keys of one and of many tiles (a star with few leaves);
* rows in which no pair is kept, and downsampled (weighted) sums.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_07084_gb300 import lne, synth
from gpu_common import make_params, oracle_counts, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2302_07084_gb300 import build
    build.build()
    c = lne.Context(0)
    c.set_option(lne.OPT_AGGREGATION, lne.AGG_SORT)
    yield c
    c.close()


def _star(leaves, n):
    u = np.zeros(leaves, dtype=np.int64)
    v = np.arange(1, leaves + 1, dtype=np.int64)
    indptr, indices = synth.csr_from_edges(n, u, v)
    return synth.Graph(n, indptr, indices, None, f"star{leaves}of{n}")


CASES = [
    (synth.ring(3), 1, 1.0),             # 6 keys
    (synth.ring(511), 3, 1.0),           # 1022 keys: below a run-length chunk
    (synth.ring(513), 3, 1.0),
    (synth.ring(3071), 5, 1.0),          # 6142, 6144 and 6146 keys: a sort tile's edge
    (synth.ring(3072), 5, 1.0),
    (synth.ring(3073), 5, 1.0),
    (synth.ring(257), 10, 97.0),         # 9 bits a vertex, many tiles
    (synth.ring(70001), 4, 1.5),         # 17 bits a vertex: 34-bit keys, a mirrored sort from bit 17
    (_star(1, 2), 2, 10000.0),           # one pair, repeated over several tiles
    (_star(3, 40), 3, 30000.0),          # long runs, isolated vertices
    (synth.chung_lu(2000, 12000, 2.1, seed=4, n_labels=5), 10, 6.3),
]


@pytest.mark.parametrize("g,T,rate", CASES, ids=lambda v: getattr(v, "name", str(v)))
def test_counts_and_csr(ctx, g, T, rate):
    p = make_params(T, np.full(T, 1.0 / T), rate * g.n_arcs, seed=11)
    dg = lne.DeviceGraph.from_graph(g)
    res = ctx.sparsifier_counts(dg, p)
    x, y, c = oracle_counts(g, p)
    assert np.array_equal(to_np(res["x"]).astype(np.int64), x)
    assert np.array_equal(to_np(res["y"]).astype(np.int64), y)
    assert np.array_equal(to_np(res["count"]).astype(np.int64), c)
    out = ctx.sparsifier_csr(dg, p)
    sp = oracle.sparsifier(g.indptr, g.indices, p.T, p.s, p.samples, p.seed, p.b)
    assert np.array_equal(to_np(out["indptr"]), sp["indptr"])
    assert np.array_equal(to_np(out["indices"]).astype(np.int64), sp["indices"])
    # one FP32 log against an FP64 log rounded to FP32: 8 ulp of the value and
    # of the log's argument's rounding (2^-24 absolute in the log)
    np.testing.assert_allclose(to_np(out["data"]), sp["data"], rtol=1e-6, atol=1e-7)


@pytest.mark.parametrize("T,rate", [(1, 1.0), (5, 0.4), (16, 0.5)])
def test_walk_without_arc_records(ctx, T, rate):
    """Graphs of more than 2^22 arcs walk through neighbours and vertex records
    instead of arc records: the oracle's pairs all the same."""
    g = synth.ring((1 << 21) + 3)
    p = make_params(T, np.full(T, 1.0 / T), rate * g.n_arcs, seed=5)
    res = ctx.sparsifier_counts(lne.DeviceGraph.from_graph(g), p)
    x, y, c = oracle_counts(g, p)
    assert np.array_equal(to_np(res["x"]).astype(np.int64), x)
    assert np.array_equal(to_np(res["y"]).astype(np.int64), y)
    assert np.array_equal(to_np(res["count"]).astype(np.int64), c)


@pytest.mark.parametrize("n,rate", [(513, 1.0), (3073, 4.0), (9001, 2.5)])
@pytest.mark.parametrize("C", [0.7, 4.0])
def test_downsampled_sums_equal_the_table(ctx, n, rate, C):
    """Weighted run sums are 64-bit integers: the same whichever way they are added up."""
    g = synth.chung_lu(n, 5 * n, 2.2, seed=6, n_labels=3)
    p = make_params(6, np.full(6, 1.0 / 6), rate * g.n_arcs, seed=3)
    p.downsample_C = C
    dg = lne.DeviceGraph.from_graph(g)
    table = lne.Context(0)
    table.set_option(lne.OPT_AGGREGATION, lne.AGG_TABLE)
    a = {k: to_np(v).copy() for k, v in ctx.sparsifier_csr(dg, p).items() if torch.is_tensor(v)}
    b = {k: to_np(v).copy() for k, v in table.sparsifier_csr(dg, p).items() if torch.is_tensor(v)}
    table.close()
    for k in ("indptr", "indices", "data"):
        assert np.array_equal(a[k], b[k]), k


def test_kept_buffers_serve_every_size(ctx):
    """Calls of changing sizes and kinds in one context equal those of fresh ones."""
    gs = [synth.ring(3000), synth.chung_lu(2000, 12000, 2.1, seed=4, n_labels=5), synth.ring(50)]
    ps = [make_params(5, np.full(5, 0.2), r * g.n_arcs, seed=2) for g, r in zip(gs, (9.0, 6.0, 300.0))]
    def run(c, i, C):
        ps[i].downsample_C = C
        return {k: to_np(v).copy() for k, v in c.sparsifier_csr(lne.DeviceGraph.from_graph(gs[i]), ps[i]).items()
                if torch.is_tensor(v)}
    for i, C in [(0, 0.0), (2, 0.0), (1, 0.0), (1, 2.0), (0, 2.0), (0, 0.0), (2, 0.0)]:
        fresh = lne.Context(0)
        fresh.set_option(lne.OPT_AGGREGATION, lne.AGG_SORT)
        a, b = run(ctx, i, C), run(fresh, i, C)
        fresh.close()
        for k in a:
            assert np.array_equal(a[k], b[k]), (i, C, k)
    before = ctx.workspace_bytes()
    run(ctx, 1, 0.0)
    assert ctx.workspace_bytes() == before   # nothing new for a size it has served


@pytest.mark.parametrize("rate", [0.3, 40.0, 900.0])
@pytest.mark.parametrize("hub", [False, True])
def test_table_values_sparse_and_dense(ctx, rate, hub):
    """The table's value passes (queued below three samples a pair, a value per lane
    above) against the oracle; hub: degree products beyond 2^24, where FP32 decides
    only what is dropped. One FP32 log of a quotient with a relative error of 1e-7:
    1e-6 as for every other value here."""
    n = 4200 if hub else 300
    if hub:      # two vertices joined to all the others: 4199^2 > 2^24
        u = np.concatenate([np.zeros(n - 1, np.int64), np.ones(n - 2, np.int64)])
        v = np.concatenate([np.arange(1, n), np.arange(2, n)])
        g = synth.Graph(n, *synth.csr_from_edges(n, u, v), None, "hubs")
    else:
        g = synth.chung_lu(n, 2000, 2.2, seed=8, n_labels=2)
    p = make_params(3, [0.2, 0.3, 0.5], rate * g.n_arcs, seed=4)
    with_table = lne.Context(0)
    with_table.set_option(lne.OPT_AGGREGATION, lne.AGG_TABLE)
    out = {k: to_np(v).copy() for k, v in with_table.sparsifier_csr(lne.DeviceGraph.from_graph(g), p).items()
           if torch.is_tensor(v)}
    with_table.close()
    sp = oracle.sparsifier(g.indptr, g.indices, p.T, p.s, p.samples, p.seed, p.b)
    assert np.array_equal(out["indptr"], sp["indptr"])
    assert np.array_equal(out["indices"].astype(np.int64), sp["indices"])
    np.testing.assert_allclose(out["data"], sp["data"], rtol=1e-6, atol=1e-7)
