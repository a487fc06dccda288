"""The small SVD of matrices whose singular values span many scales: a block diagonal
matrix whose second block is scaled down to 1e-12 of the first. Its singular values are
the blocks' own, each known to FP64 accuracy, however small the block (the blocks share
no row or column). The FP32 start leaves the cosines between columns below 0.4 c ulp
(1.2e-6 at c = 48), whatever the columns' lengths; a singular value is off by the square
of that times c (7e-11) before the FP64 refinement, the rows of U^T R by c of it (6e-5)."""
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


@pytest.mark.parametrize("c", [16, 32, 48])
@pytest.mark.parametrize("scale", [1e-6, 1e-9, 1e-10, 1e-12])
def test_blocks_of_two_scales(ctx, c, scale):
    rng = np.random.default_rng(c)
    h = c // 2
    A = np.triu(rng.normal(size=(h, h))) + 3 * np.eye(h)
    B = scale * (np.triu(rng.normal(size=(c - h, c - h))) + 3 * np.eye(c - h))
    R = np.zeros((c, c))
    R[:h, :h], R[h:, h:] = A, B
    U, s = ctx.svd_small(torch.from_numpy(R).cuda())
    U, s = U.cpu().numpy(), s.cpu().numpy()
    ref = np.concatenate([np.linalg.svd(A)[1], np.linalg.svd(B)[1]])
    assert np.abs(s / ref - 1.0).max() <= 1e-9
    rows = U.T @ R
    rows /= np.linalg.norm(rows, axis=1, keepdims=True)
    assert np.abs(rows @ rows.T - np.eye(c)).max() <= 6e-5
    assert np.abs(U.T @ U - np.eye(c)).max() <= 1e-9
