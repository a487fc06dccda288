"""The key sort at the edges of its 4096-key tiles and of the 1024-key run-length chunks:
the sort and the run lengths by themselves (tests/cpp/sort_edges.cu), and whole calls of
just below, at and just above a full tile, plain and downsampled (the sort carries a
payload then), equal to the dense-table aggregation: whole numbers, and values that
depend on them alone."""
import numpy as np
import pytest
import torch

from paper_2302_07084_gb300 import lne, synth
from gpu_common import make_params, to_np
from test_gpu_bounded_waits import _run

pytestmark = pytest.mark.gpu


def test_sort_and_run_lengths(tmp_path):
    _run(tmp_path, "sort_edges")


@pytest.mark.parametrize("n", [512, 2047, 2048, 2049, 4096])   # 1024, 4094, 4096, 4098 and 8192 keys
@pytest.mark.parametrize("C", [0.0, 0.7])
def test_whole_calls(n, C):
    g = synth.ring(n)
    p = make_params(4, np.full(4, 0.25), float(g.n_arcs), seed=9)
    p.downsample_C = C
    dg = lne.DeviceGraph.from_graph(g)
    out = []
    for agg in (lne.AGG_SORT, lne.AGG_TABLE):
        c = lne.Context(0)
        c.set_option(lne.OPT_AGGREGATION, agg)
        m = c.sparsifier_csr(dg, p)
        out.append({k: to_np(v).copy() for k, v in m.items() if torch.is_tensor(v)})
        c.close()
    assert out[0]["indices"].size > 0
    for k in ("indptr", "indices", "data"):
        assert np.array_equal(out[0][k], out[1][k]), k
