"""The surrogate's kernels at the row counts where their work split changes:
groups of 2, 4, 8 or 32 rows a CTA (152 CTAs), the staging chunks of 256 rows
and ragged tails, against the FP64 oracle. Tolerances: 256-term FP32 dot
products are within 256 2^-24 = 1.5e-5 of exact relative to the sum of their
terms' magnitudes; sums over up to 1,300 rows of a gradient within 1300 2^-24
= 8e-5 of it; a few times these are allowed."""
import numpy as np
import pytest
import torch

from oracle import surrogate as sg
from paper_2302_07084_gb300 import lne

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2302_07084_gb300 import build
    build.build()
    c = lne.Context(0)
    yield c
    c.close()


def _gapped(seed, rows):
    """Network and rows whose pre-activations keep clear of zero (biases of
    +-2, small weights), so no ReLU decision depends on rounding."""
    rng = np.random.default_rng(seed)
    theta = rng.normal(0.0, 0.005, sg.N_PARAMS)
    p = sg.unpack(theta)
    sign = np.where(np.arange(256) % 2 == 0, 1.0, -1.0)
    p["b1"][:], p["b2"][:] = 2.0 * sign, 2.0 * sign[::-1]
    p["W1"][:] *= 2.0
    p["w3"][:] = rng.normal(0.0, 0.1, 256)
    theta = theta.astype(np.float32)
    mean = rng.normal(0.0, 1.0, 30).astype(np.float32)
    std = rng.uniform(0.5, 2.0, 30).astype(np.float32)
    X = (mean + std * rng.normal(size=(rows, 30))).astype(np.float32)
    t = rng.normal(size=rows).astype(np.float32)
    th, Xs = sg.bf16_round(theta), (X.astype(np.float64) - mean) / std
    _, (_, z1, _, z2, _) = sg.forward(th, Xs)
    assert min(np.abs(z1).min(), np.abs(z2).min()) > 1e-3
    return theta, mean, std, X, t, th, Xs


@pytest.mark.parametrize("rows", [1, 2, 3, 304, 305, 1216, 1217, 5001])
def test_forward(ctx, rows):
    theta, mean, std, X, _, th, Xs = _gapped(rows, rows)
    ctx.surrogate_set_params(theta, mean, std)
    y = ctx.surrogate_predict(torch.as_tensor(X).cuda()).cpu().numpy()
    ref, _ = sg.forward(th, Xs)
    assert y.shape == (rows,) and np.abs(y - ref).max() <= 1e-4 * np.abs(ref).max()


@pytest.mark.parametrize("rows", [1, 255, 257, 305, 1300])
def test_gradient(ctx, rows):
    theta, mean, std, X, t, th, Xs = _gapped(10 + rows, rows)
    ctx.surrogate_set_params(theta, mean, std)
    g, loss = ctx.surrogate_grad(torch.as_tensor(X).cuda(), torch.as_tensor(t).cuda())
    assert abs(loss - sg.loss(th, Xs, t)) <= 1e-5 * sg.loss(th, Xs, t)
    got, want = sg.unpack(g.cpu().numpy().astype(np.float64)), sg.unpack(sg.grad(th, Xs, t))
    for name, _ in sg.LAYOUT:
        assert np.abs(got[name] - want[name]).max() <= 3e-4 * np.abs(want[name]).max(), name


@pytest.mark.parametrize("rows", [1, 37, 257, 305, 609, 1300])
def test_adam_step(ctx, rows):
    theta, mean, std, X, t, th, Xs = _gapped(20 + rows, rows)
    ctx.surrogate_set_params(theta, mean, std)
    ctx.surrogate_train(torch.as_tensor(X).cuda(), torch.as_tensor(t).cuda(), epochs=1, batch=rows, lr=1e-3, seed=1)
    got, _, _ = ctx.surrogate_get_params()
    g = sg.grad(th, Xs, t)
    want, _, _ = sg.adam_step(theta.astype(np.float64), np.zeros(sg.N_PARAMS), np.zeros(sg.N_PARAMS), g, 1)
    diff = np.abs(got - want)
    firm = np.abs(g) > 1e-3 * np.abs(g).max()   # lr g / (|g| + eps): well-determined where |g| >> rounding
    assert diff[firm].max() <= 2e-6 and diff.max() <= 2.1e-3


def test_many_passes_in_one_call(ctx):
    """Several launches of several passes (1, 2, 4, 8, ... of them), ragged
    last batches: the same call gives the same bits, and the loss falls."""
    rng = np.random.default_rng(5)
    X = rng.normal(size=(700, 30)).astype(np.float32)
    t = np.sin(X[:, 0]).astype(np.float32)
    Xd, td = torch.as_tensor(X).cuda(), torch.as_tensor(t).cuda()
    out = []
    for _ in range(2):
        ctx.surrogate_init(seed=2)
        loss = ctx.surrogate_train(Xd, td, epochs=21, batch=96, lr=1e-3, seed=4)
        out.append(ctx.surrogate_get_params()[0])
    assert np.array_equal(out[0], out[1]) and loss < 0.2 * t.var()
