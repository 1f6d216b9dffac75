"""Selections on two streams at once, each with its own workspace: while the
CTAs of one share the GPU with the other's, those of a group reach and leave
their barriers at uneven times, and every result stays what it is alone."""
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


@pytest.mark.parametrize("sizes", [((2000, 3), (1800, 2)), ((1500, 6), (3000, 5)), ((20000, 3), (1200, 7))])
def test_two_streams(sizes):
    runs = []
    for i, (n2, m) in enumerate(sizes):
        F = wl.population(n2, m, m + 9, "sphere", seed=40 + i)
        R = wl.das_dennis(wl.h_for_count(n2 // 2, m), m)
        keep = n2 // 2
        ref, t = oracle.nsga3_select(F, R, keep, 5, 1)
        nbytes = emo.emo_workspace_size(emo.EMO_OP_NSGA3_SELECT, n2, m, R.shape[0])
        runs.append(dict(F=torch.from_numpy(F).cuda(), R=torch.from_numpy(R).cuda(), keep=keep, ref=ref, t=t,
                         stream=torch.cuda.Stream(), ws=torch.empty(nbytes, dtype=torch.uint8, device="cuda"),
                         out=torch.full((64, keep), -1, dtype=torch.int32, device="cuda"),
                         info=torch.full((64, 8), -7, dtype=torch.int32, device="cuda")))
    torch.cuda.synchronize()
    for rep in range(64):
        for r in runs:
            emo.emo_nsga3_select(r["F"], r["R"], r["keep"], 5, 1, survivors=r["out"][rep], info=r["info"][rep],
                                 ws=r["ws"], stream=r["stream"])
    torch.cuda.synchronize()
    for r in runs:
        info, t = r["info"].cpu().numpy(), r["t"]
        assert np.all(info[:, 0] == 0)
        assert np.all(info[:, 1:4] == [t["last_rank"], t["n_before"], t["n_last"]])
        assert np.all(r["out"].cpu().numpy() == r["ref"][None])
