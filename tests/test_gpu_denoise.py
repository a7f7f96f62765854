"""The conv net's last layer (32 x 4 pixel tiles) and the denoiser's fused first and last layers against the
FP64 oracle at ragged sizes, in FP32 precision; in place equals out of place.  Bound as for the FP32 network."""
import numpy as np
import pytest

from helpers import rel, to_dev, to_host
from oracle import convnet

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,H,W", [(1, 4, 32), (2, 5, 33), (1, 9, 1), (1, 3, 70), (3, 1, 31)])
def test_forward_and_denoise(N, H, W):
    import paper_2411_01955_gb300 as hq
    rng = np.random.default_rng(H)
    vec = (rng.normal(size=convnet.num_params()) * 0.1).astype(np.float32)
    params = convnet.unflatten(vec)
    net = hq.Net()
    net.set_params(vec)
    net.set_precision(hq.HQS_PREC_FP32)
    x = rng.normal(size=(N, 2, H, W)).astype(np.float32)
    got = net.forward(torch.from_numpy(x).cuda()).cpu().numpy()
    assert rel(got, convnet.forward(params, x)[0]) <= 1e-5
    v = (rng.normal(size=(H, W)) + 1j * rng.normal(size=(H, W))).astype(np.complex64)
    sigma = 0.3
    t = to_dev(v)
    out = net.denoise(t, torch.empty_like(t), sigma)
    o = convnet.forward(params, np.stack([v.real, v.imag])[None].astype(np.float64) / sigma)[0]
    assert rel(to_host(out), v - sigma * (o[0, 0] + 1j * o[0, 1])) <= 1e-5
    assert torch.equal(net.denoise(t, t, sigma), out)
