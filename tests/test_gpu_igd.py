"""IGD on the GPU: the grouped route (reference points along a Hilbert curve, far
population points skipped per group) and the direct one return the same
distances -- the same float minimum for every reference point -- at the edges
of their tiles and on the layouts that could break the skipping bound."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA GPU", allow_module_level=True)

import oracle  # noqa: E402
from paper_2503_20286_gb300 import _binding as emo  # noqa: E402
from paper_2503_20286_gb300 import build as _build  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    _build.build()
    emo.lib()


def _dists(F, Ref, grouped):
    """The IGD and the minima (float bits, the head of the workspace)."""
    n_ref, m = Ref.shape
    nbytes = emo.emo_workspace_size(emo.EMO_OP_IGD, n_ref, m, 0) if grouped else 8 * n_ref
    ws = torch.full((nbytes,), 0xAB, dtype=torch.uint8, device="cuda")
    out = torch.empty(1, dtype=torch.float64, device="cuda")
    L = emo.lib()
    s = torch.cuda.current_stream().cuda_stream
    assert L.emo_igd(F.data_ptr(), F.shape[0], m, Ref.data_ptr(), n_ref, out.data_ptr(), ws.data_ptr(), nbytes, s) == 0
    torch.cuda.synchronize()
    return float(out.item()), ws[:4 * n_ref].view(torch.int32).cpu().numpy()


def _cloud(kind, n, m, g):
    x = torch.rand(n, m, generator=g, device="cuda")
    if kind == "far":        # every point about equally far from every reference point
        return x * 1e-3 + 50.0
    if kind == "line":
        return x[:, :1].expand(n, m).contiguous() * 2.0 - 0.5
    if kind == "equal":
        return torch.full((n, m), 0.25, device="cuda")
    return x


@pytest.mark.parametrize("n,n_ref,m,kind", [
    (700001, 1024, 3, "cloud"), (690000, 1025, 2, "cloud"), (685001, 1031, 5, "line"), (175001, 4099, 3, "far"),
    (88000, 8193, 4, "cloud"), (240011, 3001, 8, "cloud"), (360000, 2049, 3, "equal"), (350100, 2000, 16, "far")])
def test_grouped_route_equals_direct(n, n_ref, m, kind):
    assert n * n_ref >= 7e8  # pairs from which the grouped route is taken
    g = torch.Generator(device="cuda").manual_seed(n + m)
    F = _cloud(kind, n, m, g)
    Ref = torch.rand(n_ref, m, generator=g, device="cuda")
    if kind == "equal":
        Ref[::3] = 0.25
    a, da = _dists(F, Ref, True)
    b, db = _dists(F, Ref, False)
    assert np.array_equal(da, db)
    assert a == b
    # float32 squared distances against FP64: (m + 3) / 2 roundings of each distance
    assert a == pytest.approx(oracle.igd(F.cpu().numpy(), Ref.cpu().numpy(), parallel=oracle.has_parallel()),
                              rel=(m + 3) * 2.0 ** -24, abs=1e-300)


def test_grouped_route_with_non_finite_values():
    g = torch.Generator(device="cuda").manual_seed(3)
    F, Ref = torch.rand(500001, 3, generator=g, device="cuda"), torch.rand(1500, 3, generator=g, device="cuda")
    F[5, 1], F[77, 0], F[300] = float("nan"), float("inf"), -float("inf")
    Ref[7, 2], Ref[400, 0] = float("nan"), float("inf")
    assert np.array_equal(_dists(F, Ref, True)[1], _dists(F, Ref, False)[1])


@pytest.mark.parametrize("n,n_ref,m", [(1, 1, 2), (3, 1, 3), (5, 255, 3), (255, 257, 2), (1023, 513, 5), (1, 1023, 16),
                                       (3000, 300, 6), (1025, 512, 4)])
def test_direct_route_edges(n, n_ref, m):
    g = torch.Generator(device="cuda").manual_seed(n)
    F, Ref = torch.rand(n, m, generator=g, device="cuda"), torch.rand(n_ref, m, generator=g, device="cuda")
    a, d = _dists(F, Ref, False)
    assert a == pytest.approx(oracle.igd(F.cpu().numpy(), Ref.cpu().numpy()), rel=(m + 3) * 2.0 ** -24)
