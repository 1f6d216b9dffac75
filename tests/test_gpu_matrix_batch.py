"""Batches that hold problems ranked from the dominance matrix (six objectives
and more): several of them in one call, with prefix sets by segments (up to
eight objectives) and by halves, and beside problems ranked by the tree. Uneven
sizes, ties and duplicates; survivors and info equal the oracle's."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2503_20286_gb300 import _binding as emo  # noqa: E402
from paper_2503_20286_gb300 import build as _build  # noqa: E402
from paper_2503_20286_gb300 import workloads as wl  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


def _problem(b, n2, m, q):
    F = wl.population(n2, m, m + 9, "sphere" if b % 2 else "linear", seed=300 + b, quantize=q)
    if b % 3 == 0:
        F[n2 // 2:n2 // 2 + n2 // 8] = F[:n2 // 8]  # duplicates
    return F, wl.das_dennis(wl.h_for_count(min(n2 // 2, 400), m), m)


@pytest.mark.parametrize("shapes", [
    [(1500, 6, 0), (1023, 6, 8.0), (700, 8, 4.0), (1025, 8, 0), (900, 9, 16.0), (2100, 16, 0), (2, 16, 0), (33, 7, 0)],
    [(3000, 2, 0), (1500, 3, 16.0), (1100, 7, 8.0), (2049, 9, 0), (800, 5, 0), (64, 12, 4.0), (1, 2, 0), (2500, 6, 0)]])
@pytest.mark.parametrize("mode", [0, 1])
def test_batches_of_the_matrix_route(shapes, mode):
    problems, refs = [], []
    for b, (n2, m, q) in enumerate(shapes):
        F, R = _problem(b, n2, m, q)
        keep = max(1, n2 // 2)
        refs.append(oracle.nsga3_select(F, R, keep, 11, b, mode=mode))
        problems.append(dict(F=torch.from_numpy(F).cuda(), R=torch.from_numpy(R).cuda(), n_keep=keep, seed=11,
                             generation=b, niche_mode=mode,
                             survivors=torch.full((keep,), -1, dtype=torch.int32, device="cuda"),
                             info=torch.full((8,), -7, dtype=torch.int32, device="cuda")))
    emo.emo_nsga3_select_batch(problems)
    torch.cuda.synchronize()
    for p, (surv, t) in zip(problems, refs):
        info = p["info"].cpu().numpy()
        assert info[0] == 0 and list(info[1:4]) == [t["last_rank"], t["n_before"], t["n_last"]]
        assert np.array_equal(p["survivors"].cpu().numpy(), surv)
