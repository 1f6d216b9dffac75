"""Points next to the ideal point: normalised objectives down to 1e-40, whose
squares underflow in float, are associated as the oracle does it (scales on
both sides of where the float search rescales them and of where every
reference is evaluated in FP64)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_20286_gb300 import build as _build  # noqa: E402
from paper_2503_20286_gb300 import workloads as wl  # noqa: E402
from tests import _gpu  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,h", [(2, 300), (3, 40), (5, 9), (8, 4)])
@pytest.mark.parametrize("scale", [1e-13, 1e-16, 1e-18, 1e-20, 1e-21, 1e-22, 3e-23, 1e-30, 1e-35, 1e-37, 1e-40])
def test_points_next_to_the_ideal_point(m, h, scale):
    _build.build()
    rng = np.random.default_rng(m)
    u = np.abs(rng.standard_normal((300, m)))
    u /= np.linalg.norm(u, axis=1, keepdims=True)
    u[:m] = np.eye(m)  # the ideal point is 0
    far = wl.population(1500, m, m + 9, "sphere", seed=m) + np.float32(0.01)
    F = np.concatenate([(u * scale).astype(np.float32), far]).astype(np.float32)
    _gpu.compare_select(F, wl.das_dennis(h, m), 900, 3, 1)
