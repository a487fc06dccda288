"""The propagation's products by a lane group per row (graphs with short rows,
taken by lne_embed, which knows the longest row) and by slices (lne_propagate,
which does not): every sum has the same order, so the two give the same bits.
Widths: every lane-group size and both column counts per lane; rows that cross
slices of 32 nonzeros, isolated vertices, weights, BF16 operands. A graph with a
hub takes the slices in both and is checked against the spectral filter in
FP64."""
import numpy as np
import pytest
import torch

import oracle
from paper_2302_07084_gb300 import lne, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2302_07084_gb300 import build
    build.build()
    c = lne.Context(0)
    c.set_option(4, 1)   # LNE_OPT_DENSE_PRODUCT: the CSR products, which lne_rsvd takes
    yield c
    c.close()


def _with_isolated(g, extra):
    """g with `extra` isolated vertices after every 7th vertex and at the end."""
    n = g.n + extra
    new = np.arange(g.n) + np.minimum(np.arange(g.n) // 7, extra - 1)
    src = new[np.repeat(np.arange(g.n), np.diff(g.indptr))]
    dst = new[g.indices]
    order = np.lexsort((dst, src))
    indptr = np.zeros(n + 1, np.int64)
    np.cumsum(np.bincount(src, minlength=n), out=indptr[1:])
    return synth.Graph(n, indptr, dst[order].astype(np.int32), None)


@pytest.mark.parametrize("d", [4, 12, 28, 48, 64, 100, 128, 140])
@pytest.mark.parametrize("kind", ["plain", "isolated", "weighted", "bf16"])
def test_short_rows_give_the_same_bits(ctx, d, kind):
    g = synth.sbm(1200, 5, 0.06, 0.006, seed=d)
    if kind == "isolated":
        g = _with_isolated(g, 60)
    assert 32 < np.diff(g.indptr).max() <= 256
    w = synth.edge_weights(g, 1, 9, seed=3) if kind == "weighted" else None
    dg = lne.DeviceGraph.from_graph(g, weights=w)
    p = lne.Params(T=3, s=[0.5, 0.3, 0.2], samples=40.0 * g.n_arcs, d=d, oversample=8, q=1, k=4, theta=0.6, mu=0.1,
                   seed=5, precision=lne.PREC_BF16_MIXED if kind == "bf16" else lne.PREC_FP32)
    X = ctx.embed(dg, p)
    X0 = ctx.rsvd(ctx.sparsifier_csr(dg, p), p)["X0"]
    assert torch.equal(ctx.propagate(dg, p, X0)["X"], X)


@pytest.mark.parametrize("d", [8, 128, 132])
def test_hub_rows_and_empty_rows(ctx, d):
    """A 3,000-leaf hub beside a sparse graph with isolated vertices: the hub's
    partial sums are added by the last slice to arrive. F and P against FP64:
    sums of up to 3,000 terms, 1e-5 of the largest entry."""
    base = synth.sbm(4000, 2, 0.002, 0.001, seed=1)
    src = np.repeat(np.arange(base.n), np.diff(base.indptr))
    keys = src.astype(np.int64) * base.n + base.indices
    leaves = np.arange(500, 3500)
    keys = np.unique(np.concatenate([keys, leaves, leaves * base.n]))   # vertex 0 joined to 3,000 others
    keys = keys[(keys // base.n != 3999) & (keys % base.n != 3999)]     # vertex 3,999 isolated
    indptr = np.zeros(base.n + 1, np.int64)
    np.cumsum(np.bincount(keys // base.n, minlength=base.n), out=indptr[1:])
    g = synth.Graph(base.n, indptr, (keys % base.n).astype(np.int32), None)
    X0 = np.random.default_rng(2).normal(size=(g.n, d)).astype(np.float32)
    p = lne.Params(T=1, s=[1.0], samples=1.0, d=d, k=5, theta=0.5, mu=0.2)
    out = ctx.propagate(lne.DeviceGraph.from_graph(g), p, torch.as_tensor(X0).cuda(), want_intermediates=True)
    ref = oracle.spectral_propagation(g.indptr, g.indices, X0.astype(np.float64), 5, 0.5, 0.2)
    for name in ("F", "P"):
        got = out[name].cpu().numpy()
        assert np.abs(got - ref[name]).max() <= 1e-5 * np.abs(ref[name]).max(), name
