"""Weighted products (a CSR matrix with values) of few columns: several nonzeros a
warp step, four lanes' worth of columns (c <= 16) and more. Against FP64: a row of
m terms summed in any order in FP32 (one rounding a product and an addition, fused
or not) is off by at most m 2^-23 of the sum of the terms' sizes."""
import numpy as np
import pytest
import torch

from paper_2302_07084_gb300 import lne

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2302_07084_gb300 import build
    build.build()
    c = lne.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("c", [4, 8, 12, 16, 20, 32, 64])
@pytest.mark.parametrize("dtype", [torch.float32, torch.bfloat16])
def test_narrow_weighted_products(ctx, c, dtype):
    rng = np.random.default_rng(c)
    n = 3001
    deg = rng.choice([0, 1, 3, 31, 32, 33, 64, 97], size=n)
    deg[5], deg[n - 1] = 2900, 1025          # rows of several slices
    indptr = np.zeros(n + 1, np.int64)
    np.cumsum(deg, out=indptr[1:])
    idx = np.concatenate([np.sort(rng.choice(n, size=k, replace=False)) for k in deg]).astype(np.int32)
    val = rng.standard_normal(idx.size).astype(np.float32)
    X = torch.from_numpy(rng.standard_normal((n, c)).astype(np.float32)).to(ctx.dev).to(dtype)
    csr = dict(n=n, nnz=idx.size, indptr=torch.from_numpy(indptr).to(ctx.dev),
               indices=torch.from_numpy(idx).to(ctx.dev), data=torch.from_numpy(val).to(ctx.dev))
    Y = ctx.spmm(csr, X).cpu().numpy().astype(np.float64)
    x = X.float().cpu().numpy().astype(np.float64)
    terms = val.astype(np.float64)[:, None] * x[idx]
    rows = np.repeat(np.arange(n), deg)
    ref, size = np.zeros((n, c)), np.zeros((n, c))
    np.add.at(ref, rows, terms)
    np.add.at(size, rows, np.abs(terms))
    assert (np.abs(Y - ref) <= deg[:, None] * 2.0 ** -23 * size).all()
