"""Volume interpolation by footprint units and tile-owned spreading against the FP64 oracle, at the coil
counts and widths where their variants change (1, 2 and 4 coils per lane, odd counts, a ragged last chunk),
with repeated points (units of 1 to 4), tiles of several items, and grids of one and two tiles per axis.
Bound as in test_gpu_volume.py: float32 rounding of the transforms and the tap sums, below 1e-5."""
import numpy as np
import pytest

import synth
from helpers import rel, to_dev, to_host
from oracle import nufft3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,L,W", [((8, 8, 16), 1, 4), ((16, 8, 16), 4, 8), ((16, 16, 8), 5, 6), ((16, 16, 16), 6, 5),
                                       ((8, 16, 32), 16, 7), ((16, 16, 16), 20, 6), ((8, 8, 8), 17, 6)])
def test_units_and_tiles(shape, L, W):
    import paper_2411_01955_gb300 as hq
    rng = np.random.default_rng(L)
    k = rng.uniform(-np.pi, np.pi, size=(2603, 3))
    k[:1900] *= 0.04                   # a dense centre: many points a footprint, several items a tile
    k[1900:1907] = k[1900]             # a run of equal points, not a multiple of a unit
    k[1907] = [-np.pi, np.pi, 0.0]
    traj = k.astype(np.float32)
    x = synth.phantom3d(1, shape).astype(np.complex64).astype(np.complex128)
    S = synth.coil_maps3d(2, shape, L).astype(np.complex64).astype(np.complex128)
    plan = hq.plan3d_create(to_dev(traj, np.float32), shape, to_dev(S), W, 2.0)
    y = torch.full((L, len(traj)), float("nan"), dtype=torch.complex64, device="cuda")
    hq.forward3d(plan, to_dev(x), y)
    assert rel(to_host(y), nufft3d.forward(x, S, traj, W, 2.0)) <= 1e-5
    yin = synth.complex_noise(5, y.shape).astype(np.complex64)
    out = [torch.empty(shape, dtype=torch.complex64, device="cuda") for _ in range(2)]
    for o in out:
        hq.adjoint3d(plan, to_dev(yin), o)
    assert torch.equal(out[0], out[1])
    assert rel(to_host(out[0]), nufft3d.adjoint(yin.astype(np.complex128), S, traj, W, 2.0)) <= 1e-5
