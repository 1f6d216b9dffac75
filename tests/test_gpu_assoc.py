"""The association's search over the tree of reference directions, bit-exact
against the oracle's exhaustive one: reference counts at the edges of leaves
(32) and nodes (1024), clustered, repeated and axis-parallel directions, one to
many lanes per point, every kind of grid (m <= 3 and beyond)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_20286_gb300 import _binding as emo  # noqa: E402
from paper_2503_20286_gb300 import build as _build  # noqa: E402
from paper_2503_20286_gb300 import workloads as wl  # noqa: E402
from tests import _gpu  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


@pytest.mark.parametrize("m", [2, 3, 4, 5, 6, 9])
@pytest.mark.parametrize("n_r", [1, 31, 32, 33, 1023, 1025, 2500])
def test_reference_counts(m, n_r):
    rng = np.random.default_rng(100 * m + n_r)
    R = rng.exponential(size=(n_r, m)).astype(np.float32)
    F = wl.population(1500, m, m + 9, "sphere" if n_r % 2 else "linear", seed=n_r + m)
    _gpu.compare_select(F, R, 700, seed=n_r)


@pytest.mark.parametrize("n2", [40, 6000, 30000])
def test_points_per_warp(n2):
    F = wl.population(n2, 3, 12, "sphere", seed=n2)
    _gpu.compare_select(F, wl.das_dennis(60, 3), n2 // 2, seed=3)


@pytest.mark.parametrize("m", [2, 3, 5])
def test_clustered_repeated_and_axis_directions(m):
    rng = np.random.default_rng(m)
    cone = (np.full((700, m), 1.0) + 1e-4 * rng.random((700, m))).astype(np.float32)
    R = np.concatenate([cone, np.eye(m, dtype=np.float32) * 3.0, cone[:200] * np.float32(2.0),
                        wl.das_dennis(6, m)]).astype(np.float32)
    F = wl.population(2000, m, m + 9, "sphere", seed=40 + m)
    info, t = _gpu.compare_select(F, R, 900, seed=m)
    assert info["n_recheck"] > 0          # directions repeated three times and more
    _gpu.compare_select(F, np.tile(R[:1], (300, 1)), 900, seed=m)


def test_point_at_the_ideal_point():
    F = wl.population(1200, 3, 9, "linear", seed=9)
    F[17] = 0.0
    info, t = _gpu.compare_select(F, wl.das_dennis(20, 3), 500, seed=2)
    assert info["n_recheck"] >= 1
