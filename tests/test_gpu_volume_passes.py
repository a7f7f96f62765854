"""The volume passes on axes of 64 and 128 points (two-stage transforms) in the forms that the other volume
tests do not reach: coil counts that do not divide 16 (a product per coil and a separate sum), 1, 2 and 4
coils (the sum over 4 to 16 rows of one round at once), a last round with fewer than 16 lines, and volumes
whose other axes run the general passes and hand their buffers over.  Against the FP64 oracle; bounds as in
test_gpu_volume.py: 1e-5 for the operators, the solve's true residual."""
import numpy as np
import pytest

import synth
from helpers import rel, to_dev, to_host
from oracle import nufft3d

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,L", [((8, 16, 64), 3), ((64, 8, 16), 5), ((16, 64, 8), 1), ((8, 8, 64), 2), ((8, 8, 64), 4),
                                     ((8, 64, 64), 8), ((16, 64, 32), 6), ((8, 8, 128), 13), ((128, 8, 8), 1)])
def test_mixed_axes(shape, L):
    import paper_2411_01955_gb300 as hq
    W, mu = 4, 1.0
    rng = np.random.default_rng(L)
    traj = rng.uniform(-np.pi, np.pi, size=(701, 3)).astype(np.float32)
    x = synth.phantom3d(1, shape).astype(np.complex64).astype(np.complex128)
    S = synth.coil_maps3d(2, shape, L).astype(np.complex64).astype(np.complex128)
    plan = hq.plan3d_create(to_dev(traj, np.float32), shape, to_dev(S), W, 2.0)
    y = torch.full((L, len(traj)), float("nan"), dtype=torch.complex64, device="cuda")
    hq.forward3d(plan, to_dev(x), y)
    assert rel(to_host(y), nufft3d.forward(x, S, traj, W, 2.0)) <= 1e-5
    yin = synth.complex_noise(5, y.shape).astype(np.complex64)
    out = torch.full(shape, float("nan"), dtype=torch.complex64, device="cuda")
    hq.adjoint3d(plan, to_dev(yin), out)
    rhs = nufft3d.adjoint(yin.astype(np.complex128), S, traj, W, 2.0)
    assert rel(to_host(out), rhs) <= 1e-5
    K = nufft3d.khat(nufft3d.kernel(traj, shape))
    out.fill_(float("nan"))
    hq.toeplitz_normal3d(plan, to_dev(x), out)
    assert rel(to_host(out), nufft3d.normal(x, S, K)) <= 1e-5
    # the solve's applies run with the epilogue a A^H A p + b p and under the stop flag
    rhs = rhs.astype(np.complex64).astype(np.complex128)
    u = torch.zeros(shape, dtype=torch.complex64, device="cuda")
    info = hq.dc_solve3d(plan, 1.0, mu, to_dev(rhs), u, max_iter=100, rel_tol=1e-4, precond=hq.HQS_PRECOND_NONE)
    got = to_host(u)
    assert info.rc == hq.HQS_OK
    assert np.linalg.norm(rhs - nufft3d.normal(got, S, K) - mu * got) <= 2e-4 * np.linalg.norm(rhs)
