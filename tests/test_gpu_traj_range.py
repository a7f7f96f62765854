"""Trajectories of any real value: periodic in 2 pi, and values that are not finite stay inside the
plan's arrays (their point counts as zero in the gridded operators, the others are not touched).
Bound: float32 rounding against the FP64 oracle, 1e-5."""
import numpy as np
import pytest

import synth
from helpers import make_plan, quantised, rel, to_dev, to_host
from oracle import nufft, nufft3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def points(dim, seed):
    """Points up to 40 pi either way."""
    rng = np.random.default_rng(seed)
    k = rng.uniform(-40 * np.pi, 40 * np.pi, size=(301, dim)).astype(np.float32)
    k[:20] = rng.uniform(-np.pi, np.pi, size=(20, dim))
    return k


def wild(k):
    """The same with three points that are not finite in one coordinate, and their indices."""
    out = k.copy()
    for j, v in ((3, np.nan), (50, np.inf), (51, -np.inf)):
        out[j, j % k.shape[1]] = v
    return out, [3, 50, 51]


def test_plane():
    import paper_2411_01955_gb300 as hq
    n, L, W = 32, 3, 6
    k = points(2, 1)
    case = quantised(dict(n=n, L=L, W=W, sigma=2.0, x=synth.phantom(1, n), smaps=synth.coil_maps(1, n, L), traj=k))
    yin = synth.complex_noise(5, (L, len(k))).astype(np.complex64)
    for traj, bad in ((k, []), wild(k)):
        plan, _, _ = make_plan(dict(case, traj=traj))
        y = torch.empty((L, len(k)), dtype=torch.complex64, device="cuda")
        hq.forward(plan, to_dev(case["x"]), y)
        good = np.setdiff1d(np.arange(len(k)), bad)
        want = nufft.forward(case["x"], case["smaps"], k, W, 2.0)
        assert rel(to_host(y)[:, good], want[:, good]) <= 1e-5
        x = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        hq.adjoint(plan, to_dev(yin), x)
        want = nufft.adjoint(yin[:, good].astype(np.complex128), case["smaps"], k[good], W, 2.0)
        assert rel(to_host(x), want) <= 1e-5


def test_volume():
    import paper_2411_01955_gb300 as hq
    nz, ny, nx, L, W = 8, 16, 16, 2, 4
    k = points(3, 2)
    rng = np.random.default_rng(9)
    x = (rng.normal(size=(nz, ny, nx)) + 1j * rng.normal(size=(nz, ny, nx))).astype(np.complex64)
    maps = (rng.normal(size=(L, nz, ny, nx)) + 1j * rng.normal(size=(L, nz, ny, nx))).astype(np.complex64)
    yin = synth.complex_noise(5, (L, len(k))).astype(np.complex64)
    for traj, bad in ((k, []), wild(k)):
        plan = hq.plan3d_create(to_dev(traj), (nz, ny, nx), to_dev(maps), W, 2.0)
        y = torch.empty((L, len(k)), dtype=torch.complex64, device="cuda")
        hq.forward3d(plan, to_dev(x), y)
        good = np.setdiff1d(np.arange(len(k)), bad)
        want = nufft3d.forward(x.astype(np.complex128), maps.astype(np.complex128), k, W, 2.0)
        assert rel(to_host(y)[:, good], want[:, good]) <= 1e-5
        out = torch.empty((nz, ny, nx), dtype=torch.complex64, device="cuda")
        hq.adjoint3d(plan, to_dev(yin), out)
        want = nufft3d.adjoint(yin[:, good].astype(np.complex128), maps.astype(np.complex128), k[good], W, 2.0)
        assert rel(to_host(out), want) <= 1e-5
