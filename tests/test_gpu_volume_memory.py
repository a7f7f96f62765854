"""Device memory of a volume plan: the k-space copy of the adjoint lies in the plan's own workspace where
it has the room, and the partial tiles of the spreading are bounded, whatever the points are."""
import numpy as np
import pytest

import synth
from helpers import to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,shared", [(120000, True), (140000, False)])
def test_points_cost_what_the_header_says(M, shared):
    """32^3 x 32 coils: 131,072 points fit the workspace.  Points at random touch about 4 tiles each, so
    pieces of 256 entries would need 2,048 partial tiles of 128 KiB.  The operators stay adjoint: bound
    1e-5 on <A x, y> against <x, A^H y>, float32 rounding."""
    import paper_2411_01955_gb300 as hq
    n, L = 32, 32
    S = to_dev(synth.coil_maps3d(2, (n, n, n), L))
    k = np.random.default_rng(1).uniform(-np.pi, np.pi, size=(M, 3)).astype(np.float32)
    held = []
    for m in (0, M):
        plan = hq.plan3d_create(to_dev(k[:m]), (n, n, n), S, 6, 2.0)
        held.append(plan.info()["device_bytes"])
    per_point = 116 + 8 * (1 + 8) + (0 if shared else 8 * L)
    # 64 KiB: work items and tickets of the 512 tiles
    assert held[1] - held[0] <= per_point * M + (128 << 20) + (64 << 10)
    x, y = to_dev(synth.phantom3d(1, (n, n, n))), to_dev(synth.complex_noise(3, (L, M)))
    Ax, Ahy = torch.empty_like(y), torch.empty_like(x)
    hq.forward3d(plan, x, Ax)
    hq.adjoint3d(plan, y, Ahy)
    a = np.vdot(to_host(Ax), to_host(y))
    b = np.vdot(to_host(x), to_host(Ahy))
    assert abs(a - b) <= 1e-5 * np.linalg.norm(to_host(Ax)) * np.linalg.norm(to_host(y))


def test_info_counts_the_spreading_items():
    """One item for each of the 64 tiles of the 32^3 grid, and 4 more where 5,000 equal points (1,250 units
    of 4, pieces of 256) lie in one tile."""
    import paper_2411_01955_gb300 as hq
    n = 16
    S = to_dev(synth.coil_maps3d(2, (n, n, n), 1))
    k = np.full((5000, 3), 5.5 * 2 * np.pi / (2 * n), dtype=np.float32)   # taps 4 .. 7 at W 4
    for m, items in ((0, 64), (5000, 68)):
        assert hq.plan3d_create(to_dev(k[:m]), (n, n, n), S, 4, 2.0).info()["nsub"] == items
