"""Ranks by the z-order tree (problems of up to five objectives) against Deb's
sort: sizes at the edges of leaves (32 points), nodes (1024) and of the node
level (32,768), ties, duplicates, extreme values, one front, one point per
front, and CTA shares that keep their leaves in shared or in global memory."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2503_20286_gb300 import _binding as emo  # noqa: E402
from paper_2503_20286_gb300 import build as _build  # noqa: E402
from paper_2503_20286_gb300 import workloads as wl  # noqa: E402
from tests import _gpu  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


def _check(F, n_keep=0):
    r, last = _gpu.gpu_rank(F, n_keep)
    ref = oracle.nd_sort_deb(F)
    l = ref.max() if n_keep == 0 else np.sort(ref)[n_keep - 1]
    assert last == l
    assert np.array_equal(r, np.where(ref <= l, ref, emo.EMO_NOT_RANKED))


@pytest.mark.parametrize("m", [2, 3, 4, 5])
@pytest.mark.parametrize("n2", [1, 2, 31, 32, 33, 1023, 1024, 1025, 4097])
def test_ranks_at_leaf_and_node_edges(n2, m):
    _check(wl.population(n2, m, m + 5, "sphere" if n2 % 2 else "linear", seed=n2 + m))
    _check(wl.population(n2, m, m + 5, "sphere", seed=n2 + m, quantize=8.0), max(1, n2 // 3))


@pytest.mark.parametrize("n2,m", [(32769, 3), (33000, 2), (20000, 5)])
def test_ranks_over_many_nodes(n2, m):
    _check(wl.population(n2, m, m + 9, "sphere", seed=n2), n2 // 2)


def test_ranks_of_duplicates_and_extreme_values():
    rng = np.random.default_rng(3)
    F = rng.choice(np.float32([-3.4e38, -1.0, -1e-45, -0.0, 0.0, 1e-45, 1.0, 3.4e38]), size=(3000, 3))
    _check(F)
    _check(np.repeat(rng.random((40, 4), dtype=np.float32), 60, axis=0))
    _check(np.zeros((2100, 2), np.float32))
    F = rng.random((5000, 3), dtype=np.float32)
    F[:, 1] = 0.5                       # one constant objective
    F[:2500, 2] = F[0, 2]
    _check(F)
    x = rng.random(3000, dtype=np.float32)
    _check(np.stack([x, 1 - x, np.full_like(x, 2)], 1))          # one front
    _check(np.sort(rng.random((1500, 1), dtype=np.float32), 0)[::-1] * np.float32([1, 2, 3, 4]))  # one point per front


@pytest.mark.parametrize("cap_wide", [1, 2, 5])
@pytest.mark.parametrize("m", [2, 5])
def test_ranks_do_not_depend_on_the_group(tmp_path, m, cap_wide):
    """One CTA with more leaves than its shared memory keeps, and fewer."""
    n2 = 9000
    prop = torch.cuda.get_device_capability()
    path = tmp_path / "shape.txt"
    path.write_text(f"{prop[0] * 10 + prop[1]} {m} {int(np.log2(n2))} 8 64 {cap_wide} 0 0\n")
    try:
        emo.emo_autotune(m, n2, str(path))
        assert emo.emo_launch_shape(m, n2)["peel_ctas"] == cap_wide
        _check(wl.population(n2, m, m + 9, "linear", seed=7 + m))
    finally:
        emo.emo_autotune_reset()
