"""Training kernels at the edges of their work split: the normalisation adds block sums of the
whole device."""
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
