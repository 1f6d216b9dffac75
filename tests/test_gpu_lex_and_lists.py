"""The lexicographic order by digits that span objectives (coarse, constant,
negative and tiny values side by side, sizes at the edges of a CTA's share of a
radix pass) and the picks from long candidate lists (1 to 4097 members, lists
emptied to the last), bit-exact against the oracle."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2503_20286_gb300 import build as _build  # noqa: E402
from paper_2503_20286_gb300 import _binding as emo  # noqa: E402
from tests import _gpu  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


@pytest.mark.parametrize("n2", [2047, 2048, 2049, 4097, 5000])
@pytest.mark.parametrize("values", [(2, 3, 65, 1, 5, 9), (1, 1, 2, 1, 1, 300), (64, 64, 64, 64, 64, 64)])
def test_order_of_coarse_objectives(n2, values):
    rng = np.random.default_rng(n2 + len(set(values)))
    scale = np.float32([1.0, -3.0, 1e-30, 7.0, 0.125, -1e30])
    F = np.stack([np.float32(rng.integers(0, v, n2) - v // 3) * s for v, s in zip(values, scale)], 1)
    r, last = _gpu.gpu_rank(np.ascontiguousarray(F, np.float32), 0)
    ref = oracle.nd_sort_deb(F)
    assert last == ref.max() and np.array_equal(r, ref)


@pytest.mark.parametrize("n,keep", [(33, 32), (129, 100), (1025, 1024), (4096, 3000), (4097, 4000), (6000, 2000)])
def test_picks_from_long_lists(n, keep):
    rng = np.random.default_rng(n)
    x = np.sort(rng.random(n)).astype(np.float32)
    F = np.stack([x, 1 - x], 1)                      # one front
    _gpu.compare_select(F, np.float32([[1, 0], [0, 1], [0.5, 0.5]]), keep, seed=n)
    _gpu.compare_select(F, np.float32([[0.5, 0.5]]), keep, seed=n + 1)
