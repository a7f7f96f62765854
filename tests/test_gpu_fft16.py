"""The two-stage 16 x R transforms of the Toeplitz and NUFFT passes against the FP64 oracle, at every size they
cover and at coil counts on either side of the 4-, 8- and 16-line items, of full and ragged chunks.
Bound: float32 transforms of N points carry a relative error of a few u log2 N (u = 6e-8), below 1e-5."""
import numpy as np
import pytest

import synth
from helpers import make_plan, quantised, rel, to_dev, to_host
from oracle import toeplitz

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _case(n, L, seed):
    traj = synth.traj_radial(24, 2 * n)
    return dict(n=n, L=L, W=4, sigma=2.0, x=synth.phantom(seed, n), smaps=synth.coil_maps(seed, n, L), traj=traj)


@pytest.mark.parametrize("n,coils", [(64, (1, 4, 5, 17)), (128, (3, 8, 16)), (256, (4, 9, 20)), (320, (2, 7, 13, 33)),
                                     (384, (5, 8, 16))])
def test_normal_operator_and_batch(n, coils):
    import paper_2411_01955_gb300 as hq
    plans, xs, want = [], [], []
    for i, L in enumerate(coils):
        case = quantised(_case(n, L, 3 + i))
        plan, _, _ = make_plan(case)
        x = to_dev(case["x"])
        out = torch.empty_like(x)
        hq.toeplitz_normal(plan, x, out)
        want.append(toeplitz.normal(case["x"], case["smaps"], toeplitz.khat(toeplitz.kernel(case["traj"], n, n))))
        assert rel(to_host(out), want[-1]) <= 1e-5, L
        plans.append(plan)
        xs.append(x)
    outs = [torch.empty_like(x) for x in xs]
    hq.Batch(plans).toeplitz_normal(xs, outs)
    for L, o, w in zip(coils, outs, want):
        assert rel(to_host(o), w) <= 1e-5, L


@pytest.mark.parametrize("n,coils", [(64, (1, 5, 16)), (128, (4, 9)), (256, (3, 17)), (320, (8, 13)), (384, (2, 20))])
def test_forward_and_adjoint(n, coils):
    import paper_2411_01955_gb300 as hq
    from oracle import nufft
    for i, L in enumerate(coils):
        case = quantised(_case(n, L, 11 + i))
        plan, _, _ = make_plan(case)
        y = torch.empty((L, len(case["traj"])), dtype=torch.complex64, device="cuda")
        hq.forward(plan, to_dev(case["x"]), y)
        assert rel(to_host(y), nufft.forward(case["x"], case["smaps"], case["traj"], 4, 2.0)) <= 1e-5, L
        yin = synth.complex_noise(7, y.shape).astype(np.complex64).astype(np.complex128)
        out = torch.empty((n, n), dtype=torch.complex64, device="cuda")
        hq.adjoint_axpy(plan, to_dev(yin), 0.5, to_dev(case["x"]), out)
        want = nufft.adjoint(yin, case["smaps"], case["traj"], 4, 2.0) + 0.5 * case["x"]
        assert rel(to_host(out), want) <= 1e-5, L
