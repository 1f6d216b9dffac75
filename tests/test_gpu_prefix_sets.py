"""The prefix sets of column blocks by segments of 128 columns (up to seven
keys) and by halves (more): ranks of 6 to 9 objectives, the caller-order matrix
of 2 to 5 and HypE's dominator counts with 8 and 9 objectives, against Deb's
sort, the pairwise definition and the oracle's HypE, at sizes on both sides of
a segment, a column block and a block of rows, with ties and extreme values.
Everything compared is a whole number or a bit, or equal in every bit."""
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
from tests.test_gpu_hype import compare as _hype_compare  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


def _ranks(F):
    r, last = _gpu.gpu_rank(F, 0)
    ref = oracle.nd_sort_deb(F)
    assert last == ref.max()
    assert np.array_equal(r, ref)


@pytest.mark.parametrize("m", [6, 7, 8, 9])
@pytest.mark.parametrize("n2", [1, 127, 129, 1023, 1024, 1025, 2177])
def test_ranks_at_segment_and_block_edges(n2, m):
    _ranks(wl.population(n2, m, m + 5, "sphere", seed=n2 + m))
    _ranks(wl.population(n2, m, m + 5, "linear", seed=n2 + m, quantize=2.0))


@pytest.mark.parametrize("m", [6, 8])
def test_ranks_of_extreme_and_equal_values(m):
    rng = np.random.default_rng(m)
    _ranks(rng.choice(np.float32([-3.4e38, -1.0, -0.0, 0.0, 1e-45, 3.4e38]), size=(1500, m)))
    F = rng.random((1300, m), dtype=np.float32)
    F[:, 1:] = np.float32(0.25)  # every key equal: whole prefixes
    _ranks(F)


@pytest.mark.parametrize("m", [2, 3, 4, 5])
@pytest.mark.parametrize("n2", [127, 128, 129, 1024, 1153])
def test_caller_matrix_at_segment_edges(n2, m):
    for q in (None, 4.0):
        F = wl.population(n2, m, m + 5, "sphere", seed=n2 + m, quantize=q)
        D, c = emo.emo_dominance_ws(torch.from_numpy(F).cuda())
        torch.cuda.synchronize()
        assert np.array_equal(D.cpu().numpy().view(np.uint32), oracle.dominance_bits(F))
        assert np.array_equal(c.cpu().numpy(), oracle.domination_counts(F))


@pytest.mark.parametrize("m", [2, 4, 8, 9])
def test_hype_counts_by_segments_and_halves(m):
    F = wl.population(1200, m, m + 4, "sphere", seed=m, quantize=8.0)
    U = np.random.default_rng(m).random((257, m)).astype(np.float32)
    _hype_compare(F, (F.max(axis=0) * 1.05 + 0.02).astype(np.float32), U, 600)
