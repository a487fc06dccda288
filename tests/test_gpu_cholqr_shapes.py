"""CholeskyQR2 at the shapes where its kernels change: the Gram's chunks of 64
rows and padded 8-column tiles, 16-byte against 4-byte copies (c % 4), the row
solve's 16-column blocks and its tiles of 32 to 256 rows, and magnitudes near
FP32's limits (the Gram's per-column powers of two). Q is orthonormal and
Y = Q R to FP32 rounding of c-term sums (c 2^-24 and a few), and R equals the
FP64 Cholesky factor's to the FP32 rounding of the first pass' Q."""
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


def _check(ctx, Y):
    c = Y.shape[1]
    Q, R = ctx.cholqr2(Y)
    Y64, Q64 = Y.double(), Q.double()
    eye = torch.eye(c, dtype=torch.float64, device="cuda")
    assert (Q64.T @ Q64 - eye).abs().max() <= 1e-5
    scale = Y64.norm(dim=0, keepdim=True)
    assert ((Q64 @ R - Y64).norm(dim=0, keepdim=True) / scale).max() <= 1e-6 * np.sqrt(c)
    want = torch.linalg.cholesky((Y64 / scale).T @ (Y64 / scale)).T * scale
    assert ((R - want) / scale).abs().max() <= 1e-6 and torch.equal(R, torch.triu(R))


@pytest.mark.parametrize("n,c", [(1, 1), (63, 1), (70, 7), (65, 16), (300, 17), (4097, 30), (1000, 33), (20000, 45),
                                 (64, 64), (5000, 130), (10312, 144), (39000, 144), (39000, 145), (3000, 160),
                                 (40001, 100), (500, 240)])
def test_shapes(ctx, n, c):
    g = torch.Generator(device="cuda").manual_seed(n + c)
    Y = torch.randn(n, c, generator=g, device="cuda")
    if n == c:
        Y += 4.0 * torch.eye(n, device="cuda") * n ** 0.5
    _check(ctx, Y * torch.logspace(0, -2, c, device="cuda"))


@pytest.mark.parametrize("scale", [1e-15, 1e-12, 1e12, 1e15])
def test_magnitudes(ctx, scale):
    g = torch.Generator(device="cuda").manual_seed(3)
    _check(ctx, torch.randn(3000, 20, generator=g, device="cuda") * scale)


def test_zero_column_and_non_finite_rows_are_refused(ctx):
    Y = torch.randn(500, 24, device="cuda")
    Y[:, 5] = 0.0
    with pytest.raises(lne.LneError) as e:
        ctx.cholqr2(Y)
    assert e.value.code == -6
    Y = torch.randn(500, 24, device="cuda")
    Y[77, 3] = float("nan")
    with pytest.raises(lne.LneError) as e:
        ctx.cholqr2(Y)
    assert e.value.code == -6
