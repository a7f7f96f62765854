"""Re-binning a 2D plan's points: accepted whatever the bins hold, since the spreading's lists and
partial tiles belong to the 8 x 8 tiles of the grid and do not depend on the bin size."""
import numpy as np
import pytest

import synth
from helpers import rel, to_dev, to_host

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_rebin_of_many_points():
    """120,000 points x 32 coils on the 128^2 grid: by bins of 32, each of the 16 bins has 9 / 16
    of the points as neighbours; a partial tile of 32 x 32 x 32 coils for every 256 of those would
    be 1.03 GiB.  Bound: the float32 sums of one grid cell in another order, far below 1e-5."""
    import paper_2411_01955_gb300 as hq
    n, L, M = 64, 32, 120000
    traj = np.random.default_rng(3).uniform(-np.pi, np.pi, size=(M, 2)).astype(np.float32)
    plan = hq.plan_create(to_dev(traj), n, n, to_dev(synth.coil_maps(2, n, L)), 4, 2.0)
    y = to_dev(synth.complex_noise(7, (L, M)))
    out = {}
    for tile in (8, 32, 16):
        hq.plan_retile(plan, tile)
        assert plan.info().tile == tile
        x = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        hq.adjoint(plan, y, x)
        out[tile] = to_host(x)
    assert rel(out[32], out[8]) <= 1e-5 and rel(out[16], out[8]) <= 1e-5
