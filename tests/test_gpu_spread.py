"""Tile-owned spreading and the interpolation of the 2D operators against the FP64 oracle: 1, 2 and 4 coils
per lane, odd counts and a ragged last chunk, every width, light tiles, tiles of one whole CTA and of several,
taps that wrap, on the smallest grid and after re-binning (the lists follow the points' order).
Bound: float32 rounding of the transforms and the tap sums, below 1e-5."""
import numpy as np
import pytest

import synth
from helpers import make_plan, quantised, rel, to_dev, to_host
from oracle import nufft

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,L,W", [(16, 1, 4), (16, 5, 8), (32, 3, 2), (32, 8, 7), (64, 13, 6), (64, 20, 3), (64, 16, 5)])
def test_spread_and_interp(n, L, W):
    import paper_2411_01955_gb300 as hq
    rng = np.random.default_rng(L)
    k = rng.uniform(-np.pi, np.pi, size=(2601, 2))
    k[:1500] *= 0.05                  # one tile of several CTAs
    k[1500:1700] = rng.uniform(2.0, 2.0 + 6 * np.pi / n, size=(200, 2))   # tiles of one whole CTA
    k[1700:1705] = [[-np.pi, -np.pi], [np.pi, 0.0], [0.0, np.pi], [-np.pi, 3.1], [0.0, 0.0]]
    case = quantised(dict(n=n, L=L, W=W, sigma=2.0, x=synth.phantom(1, n), smaps=synth.coil_maps(1, n, L),
                          traj=k.astype(np.float32)))
    plan, _, _ = make_plan(case)
    y = torch.full((L, len(k)), float("nan"), dtype=torch.complex64, device="cuda")
    hq.forward(plan, to_dev(case["x"]), y)
    assert rel(to_host(y), nufft.forward(case["x"], case["smaps"], case["traj"], W, 2.0)) <= 1e-5
    yin = synth.complex_noise(5, y.shape).astype(np.complex64)
    want = nufft.adjoint(yin.astype(np.complex128), case["smaps"], case["traj"], W, 2.0)
    for tile in (8, 16, 8):
        hq.plan_retile(plan, tile)
        out = [torch.empty((n, n), dtype=torch.complex64, device="cuda") for _ in range(2)]
        for o in out:
            hq.adjoint(plan, to_dev(yin), o)
        assert torch.equal(out[0], out[1])
        assert rel(to_host(out[0]), want) <= 1e-5
