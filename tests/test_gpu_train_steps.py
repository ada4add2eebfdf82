"""Training kernels at the edges of their work split: the Adam kernel brings 128 tiles' gradient
sums into shared memory at a time, the normalisation adds block sums of the whole device."""
import numpy as np
import pytest
import torch

from oracle import mlp as M
from paper_2203_15963_gb300 import native

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _lib():
    native.build()
    native.load()


def _data(n, seed):
    inp = torch.empty((n, 3), dtype=torch.float32, device=DEV)
    tg = torch.empty((n, 7), dtype=torch.float32, device=DEV)
    native.blacklight_mlp_dataset(n, seed, inp, tg)
    return inp, tg


@pytest.mark.parametrize("tiles", [1, 127, 128, 129, 300])
def test_adam_step_over_tile_counts(tiles):
    """From zero moments the first step moves each parameter by lr g / (|g| + eps) against its
    gradient; the loss is the gradient entry point's, summed in another order
    (FP32: n 2^-24 relative at most, and 1e-5 for n <= 300 tiles of sums)."""
    n = 128 * tiles
    inp, tg = _data(n, 11 + tiles)
    p = torch.empty(M.N_PARAMS, dtype=torch.float32, device=DEV)
    native.blacklight_mlp_init(p, 3)
    native.blacklight_mlp_normalise(inp, tg, p)
    g = torch.empty_like(p)
    loss = native.blacklight_mlp_grad(p, inp, tg, g)
    q = p.clone()
    hist = torch.zeros(1, dtype=torch.float32, device=DEV)
    native.blacklight_mlp_train(q, inp, tg, n, 1, 1e-3, 1e-3, loss_history=hist)
    gg = g[:M.OFF_MEAN].double().cpu().numpy()
    step = (q - p).double().cpu().numpy()
    big = np.abs(gg) > 1e-3 * np.abs(gg).max()
    # the first step is lr g / (|g| + eps), eps = 1e-8; q - p carries the rounding of q (2^-24 |q|)
    want = -1e-3 * gg[big] / (np.abs(gg[big]) + 1e-8)
    np.testing.assert_allclose(step[:M.OFF_MEAN][big], want, rtol=1e-3)
    assert np.all(step[M.OFF_MEAN:] == 0.0)
    assert float(hist[0]) == pytest.approx(loss, rel=1e-5)


@pytest.mark.parametrize("n", [64, 127, 129, 77825, 300001])
def test_normalise_matches_least_squares(n):
    """Against numpy's float64 least squares. Both are accurate to about cond^2 2^-53 < 1e-13;
    the stored floats may then differ by one rounding, 2^-23 of the vector's largest entry."""
    inp, tg = _data(n, n)
    p = torch.empty(M.N_PARAMS, dtype=torch.float32, device=DEV)
    native.blacklight_mlp_init(p, 3)
    native.blacklight_mlp_normalise(inp, tg, p)
    got = p.double().cpu().numpy()
    x, o = inp.double().cpu().numpy(), tg.double().cpu().numpy()
    f = M.features(x[:, 0], x[:, 1], x[:, 2]).astype(np.float32).astype(np.float64)[:, :3]
    A = np.concatenate([f, np.ones((n, 1))], 1)
    beta, *_ = np.linalg.lstsq(A, o, rcond=None)
    rms = np.sqrt(np.mean((o - A @ beta) ** 2, axis=0))
    for a, b in ((got[M.OFF_MEAN:M.OFF_SCALE], beta[3]), (got[M.OFF_SCALE:M.OFF_A], rms),
                 (got[M.OFF_A:].reshape(7, 3), beta[:3].T)):
        np.testing.assert_allclose(a, b, rtol=0, atol=2.0 ** -22 * np.abs(b).max())
