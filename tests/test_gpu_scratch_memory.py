"""Device memory of the key-sort path between calls: what a call has handed back belongs to
whoever allocates next, another context or another allocator of the process, and calls in
several threads share it without disturbing each other."""
import threading

import pytest
import torch

from paper_2302_07084_gb300 import lne, synth

pytestmark = pytest.mark.gpu

GB = 1 << 30


@pytest.fixture(scope="module", autouse=True)
def built():
    from paper_2302_07084_gb300 import build
    build.build()


def _case(n, m, per_arc, seed):
    indptr, indices = synth.chung_lu_device(n, m, 2.2, seed)
    g = lne.DeviceGraph.from_tensors(indptr, indices)
    return g, lne.Params(T=5, s=[0.2] * 5, samples=per_arc * g.nnz, d=32, seed=seed)


def _free():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    return torch.cuda.mem_get_info()[0]


def test_other_allocators_get_the_scratch():
    g, p = _case(400000, 8000000, 12.5, 1)   # 2e8 samples: 7 GB of scratch
    a, b = lne.Context(0), lne.Context(0)
    before = _free()
    m = a.sparsifier_csr(g, p)
    nnz, total = m["nnz"], float(m["data"].double().sum())
    del m
    first = before - _free()
    b.sparsifier_csr(g, p)
    second = before - first - _free()
    # the second context takes its own results only, not a scratch of its own
    assert second <= b.workspace_bytes() + GB // 4 and second < 0.6 * first
    scratch = first - a.workspace_bytes()
    assert scratch > 3 * GB
    # another allocator: all but 2 GB of what is free, then 2 GB more than that; the call's
    # end is enough, without a synchronisation of the device
    a.sparsifier_csr(g, p, copy=False)
    held = torch.empty(torch.cuda.mem_get_info()[0] - 2 * GB, dtype=torch.uint8, device="cuda")
    try:
        torch.empty(4 * GB, dtype=torch.uint8, device="cuda")   # out of the scratch
    finally:
        del held
        _free()
    m = a.sparsifier_csr(g, p)   # and the next call takes its scratch again
    assert m["nnz"] == nnz and float(m["data"].double().sum()) == total
    del m
    a.close()
    b.close()
    assert before - _free() < GB // 4


def test_threads_share_the_scratch():
    cases = [_case(70000 + 4096 * i, 400000 + 10007 * i, 6.0, 3 + i) for i in range(4)]
    torch.cuda.synchronize()
    ref = []
    c = lne.Context(0)
    for g, p in cases:
        m = c.sparsifier_csr(g, p)
        ref.append((m["indptr"], m["indices"], m["data"]))
    c.close()
    bad = []

    def work(i):
        torch.cuda.set_device(0)
        c = lne.Context(0)
        with torch.cuda.stream(torch.cuda.Stream()):
            for k in range(8):
                j = (i + k) % len(cases)
                m = c.sparsifier_csr(*cases[j])
                if not all(torch.equal(m[key], r) for key, r in zip(("indptr", "indices", "data"), ref[j])):
                    bad.append((i, k))
        c.close()

    threads = [threading.Thread(target=work, args=(i,)) for i in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad, bad


def test_weighted_walk_without_memory_for_its_records():
    """The weighted step's records (16 bytes an arc) are left out where they do not fit:
    the walk searches the thresholds then, and draws the same pairs."""
    indptr, indices = synth.chung_lu_device(300000, 6000000, 2.1, 5)   # 12M arcs: 192 MB of records
    g = lne.DeviceGraph.from_tensors(indptr, indices)
    src = torch.repeat_interleave(torch.arange(300000, device="cuda"), torch.diff(indptr))
    g.weights = (1 + (src + indices.long()) % 9).to(torch.int32)       # equal on both arcs of an edge
    del src
    p = lne.Params(T=6, s=[1 / 6] * 6, samples=300000.0, d=32, seed=7)
    a = lne.Context(0)
    a.set_option(lne.OPT_AGGREGATION, lne.AGG_SORT)

    def counts():
        a.trace(True)
        r = a.sparsifier_counts(g, p)
        r = {k: r[k].cpu() for k in ("x", "y", "count")}   # nothing stays in the held memory's segment
        names = {t["name"] for t in a.trace_read()}
        a.trace(False)
        return r, names

    ref, names = counts()
    assert "build_wstep" in names
    lne.Context(0).close()   # unmaps the scratch
    held = torch.empty(_free() - 128 * (1 << 20), dtype=torch.uint8, device="cuda")
    try:
        got, names = counts()
    finally:
        del held
        _free()
    assert "build_wstep" not in names
    assert all(torch.equal(ref[k], got[k]) for k in ref)
    a.close()
