"""The tuner leaves the shapes of stages that a problem does not run at their
defaults: up to five objectives nothing builds a dominance matrix, and the group that ranks by the
tree is sized by its leaves."""
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

from paper_2503_20286_gb300 import _binding as emo  # noqa: E402
from paper_2503_20286_gb300 import build as _build  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


@pytest.mark.parametrize("m,n2", [(2, 1500), (3, 5000), (3, 20000), (5, 3000)])
def test_tree_ranked_sizes_keep_the_matrix_shapes(m, n2):
    emo.emo_autotune_reset()
    default = emo.emo_launch_shape(m, n2)
    try:
        emo.emo_autotune(m, n2)
        tuned = emo.emo_launch_shape(m, n2)
        for key in ("dom_rowblocks_per_item", "peel_wavefront", "peel_ctas"):
            assert tuned[key] == default[key]
    finally:
        emo.emo_autotune_reset()
