"""TensorMOEA/D pairs ruled out in float before FP64 (from 196,608 pairs on):
decisions bit-exact against the oracle where the float filter has least room
(offspring close to the solutions they compete with, huge and tiny penalties,
wide ranges), and on the routes without it (fewer pairs; fewer neighbours than
a record of the filter needs room for)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from tests.test_gpu_moead import _compare  # noqa: E402
from tests.test_gpu_moead import _built  # noqa: E402,F401

pytestmark = pytest.mark.gpu


def _random(n, m, t, seed):
    rng = np.random.default_rng(seed)
    X, O = rng.random((n, 3), dtype=np.float32), rng.random((n, 3), dtype=np.float32)
    F1, F2 = rng.random((n, m), dtype=np.float32), rng.random((n, m), dtype=np.float32)
    W = rng.random((n, m), dtype=np.float32) + np.float32(1e-3)
    I_nb = rng.integers(0, n, size=(n, t)).astype(np.int32)  # now and then a neighbour twice
    return X, F1, O, F2, F1.min(axis=0), W, I_nb


@pytest.mark.parametrize("n,m,t", [(2048, 3, 95), (2048, 3, 96), (2049, 3, 96), (2500, 2, 80), (1500, 4, 132),
                                   (2500, 5, 79), (1000, 8, 200), (400, 3, 400), (500, 16, 400), (9900, 16, 19),
                                   (9900, 16, 20)])
def test_routes(n, m, t):
    _compare(*_random(n, m, t, seed=n + t))


@pytest.mark.parametrize("theta", [0.0, 1e-30, 5.0, 1e30, 1e300])
@pytest.mark.parametrize("scale", [1e-6, 1e-3])
def test_close_competitors(theta, scale):
    X, F1, O, F2, z, W, I_nb = _random(2500, 3, 80, seed=4)
    rng = np.random.default_rng(8)
    F2 = (F1 * (1 + scale * rng.standard_normal(F1.shape))).astype(np.float32)
    F2[::5] = F1[::5]
    F2[1::7] = F2[0::7][: F2[1::7].shape[0]]
    W[:] = W[:1]  # one direction: neighbours compete for the same place
    _compare(X, F1, O, F2, z, W, I_nb, theta=theta)


def test_wide_ranges():
    X, F1, O, F2, z, W, I_nb = _random(2500, 3, 80, seed=5)
    rng = np.random.default_rng(9)
    f = np.float32(10.0) ** rng.integers(-30, 30, size=(F1.shape[0], 1)).astype(np.float32)
    _compare(X, F1 * f, O, F2 * np.roll(f, 1, 0), (F1 * f).min(0), W, I_nb)
