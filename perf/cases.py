"""Workloads of the reconstruction library, measured through its public Python entry points.

Each case is one call that a reconstruction program makes: the multicoil NUFFT and its adjoint, the
Toeplitz normal operator, the data-consistency step of one slice and of a batch of slices, an annealed
HQS run over slices of uneven size, the conv-net denoiser, and the volume operators and solve.  Images
are ellipse phantoms with a smooth phase seen through Gaussian-bump coil maps, sampled on golden-angle
spokes, variable-density spirals or stacks of them, with Gaussian noise; the seed sets the phantom, the
maps' phases, the trajectory's rotation and the noise.

Systems are solved for a fixed number of iterations (the outer loop's five, or the first ones of a
longer solve), so that every pass does the same work.  The weight mu is 1 or more against
||A^H A|| of about 440: conjugate gradients amplify the rounding of their operator by ||A^H A|| / mu, and
two correct programs should still agree.
"""
from __future__ import annotations

import math
import random

import numpy as np
import torch

import paper_2411_01955_gb300 as hq

SIZES = (64, 128, 256, 320, 384)         # image edges that every 2D entry point takes
VOL_SIZES = (16, 32, 64)                 # volume edges with a density preconditioner


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest operator call: one apply of A^H A on a 64^2 image, 4 coils, 16 spokes x 128;
        # launches and latency count
        dict(name="normal_64x4", op="normal", n=64, L=4, W=4, kind="radial", a=16, b=128),
        # a brain slice: 320^2, 16 coils, spiral 16 x 2048 (the library's benchmark size)
        dict(name="normal_320x16", op="normal", n=320, L=16, W=6, kind="spiral", a=16, b=2048),
        dict(name="forward_320x16", op="forward", n=320, L=16, W=6, kind="spiral", a=16, b=2048),
        dict(name="adjoint_320x16", op="adjoint", n=320, L=16, W=6, kind="spiral", a=16, b=2048),
        # the largest image with a coil count that fills no 16-coil chunk, radial spokes
        dict(name="adjoint_384x13", op="adjoint", n=384, L=13, W=6, kind="radial", a=73, b=768),
        # the data-consistency step of one slice inside an outer loop: right-hand side and 5 iterations
        dict(name="step_320x16", op="step", n=320, L=16, W=6, kind="spiral", a=16, b=2048, its=5, mu=1.0),
        # a scan's slices solved together: right-hand sides and 6 iterations of every slice
        dict(name="batch_step_16x320x16", op="batch_step", count=16, n=320, L=16, W=6, kind="spiral", a=16, b=2048,
             its=6, mu=1.0),
        # annealed HQS over slices of uneven size, coil count and trajectory (a whole call)
        dict(name="batch_hqs_9_uneven", op="batch_hqs", count=9, n=384, L=20, W=6, kind="mixed", a=64, b=0, its=5,
             outer=2, mu=2.0),
        # the conv-net denoiser on one slice (once per outer iteration)
        dict(name="denoise_320", op="denoise", n=320, m=320, sigma=0.05),
        # a volume: 64^3, 16 coils, 64 spirals of 8 x 1024 (the library's volume benchmark)
        dict(name="vol_forward_64x16", op="vol_forward", nz=64, ny=64, nx=64, L=16, W=6, a=8, b=1024),
        dict(name="vol_adjoint_64x16", op="vol_adjoint", nz=64, ny=64, nx=64, L=16, W=6, a=8, b=1024),
        # the volume's data-consistency solve inside an outer loop: 5 iterations
        dict(name="vol_solve_64x16", op="vol_solve", nz=64, ny=64, nx=64, L=16, W=6, a=8, b=1024, its=5, mu=1.0),
    ]


def draw(rng: random.Random):
    """A case between the smallest and the largest listed ones: any operator, any supported image edge,
    1 to 20 coils, radial or spiral sampling of uneven length, widths 4 to 6."""
    op = rng.choice(("normal", "forward", "adjoint", "adjoint", "forward", "step", "batch_step", "batch_hqs", "denoise",
                     "vol_forward", "vol_adjoint", "vol_normal", "vol_solve"))
    if op == "denoise":
        return dict(op=op, n=_log_int(rng, 48, 400), m=_log_int(rng, 48, 400), sigma=round(rng.uniform(0.02, 0.2), 4))
    if op.startswith("vol_"):
        nz, ny, nx = (rng.choice(VOL_SIZES) for _ in range(3))
        case = dict(op=op, nz=nz, ny=ny, nx=nx, L=_log_int(rng, 1, 16), W=rng.choice((4, 5, 6, 6)),
                    a=_log_int(rng, 2, 8), b=_log_int(rng, 100, 1024))
        if op == "vol_solve":
            case.update(its=rng.randint(2, 5), mu=round(10 ** rng.uniform(0, 1), 4))
        return case
    n = rng.choice(SIZES)
    case = dict(op=op, n=n, L=_log_int(rng, 2, 20), W=rng.choice((4, 5, 6, 6)), kind=rng.choice(("radial", "spiral")))
    if case["kind"] == "radial":
        case.update(a=_log_int(rng, 16, 96), b=2 * n)
    else:
        case.update(a=_log_int(rng, 8, 24), b=_log_int(rng, 500, 2048))
    if op == "step":
        case.update(its=rng.randint(2, 5), mu=round(10 ** rng.uniform(0, 1), 4))
    elif op == "batch_step":
        case.update(count=rng.randint(2, 12), its=rng.randint(3, 6), mu=round(10 ** rng.uniform(0, 1), 4))
    elif op == "batch_hqs":
        case.update(count=rng.randint(2, 9), kind="mixed", a=rng.randint(48, 64), b=0, its=rng.randint(3, 5), outer=2,
                    mu=2.0)
    return case


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


# ------------------------------------------------------------------ inputs
def _coords(n):
    return (torch.arange(n, dtype=torch.float64) - n // 2) / (n / 2.0)


def _phantom(shape, r):
    """Ellipsoids with a smooth random phase, complex64 on the GPU."""
    ax = torch.meshgrid(*[_coords(n) for n in shape], indexing="ij")
    ax = [a.cuda() for a in ax]
    head = sum((a / s) ** 2 for a, s in zip(ax, (0.85, 0.8, 0.9)[-len(shape):])) <= 1.0
    mag = 0.25 * head.double()
    for _ in range(10):
        c = [r.uniform(-0.55, 0.55) for _ in shape]
        s = [r.uniform(0.06, 0.4) for _ in shape]
        mag = mag + r.uniform(0.1, 1.0) * (sum(((a - ci) / si) ** 2 for a, ci, si in zip(ax, c, s)) <= 1.0)
    mag = mag * head
    p = sum(r.uniform(-1, 1) * a + r.uniform(-1, 1) * a * a for a in ax)
    return torch.polar(mag, math.pi * p / len(shape)).to(torch.complex64).contiguous()


def _coil_maps(shape, L, r):
    """Gaussian bumps on a ring with linear phases, root-sum-of-squares 1, complex64 (L, *shape)."""
    ax = [a.cuda() for a in torch.meshgrid(*[_coords(n) for n in shape], indexing="ij")]
    maps = []
    for l in range(L):
        ang = 2 * math.pi * l / L + r.uniform(-0.2, 0.2)
        c = [math.sin(ang) * 1.4, math.cos(ang) * 1.4]
        if len(shape) == 3:
            c = [0.5 * (-1) ** l] + c
        d2 = sum((a - ci) ** 2 for a, ci in zip(ax, c))
        ph = 2 * math.pi * l / L + sum(r.uniform(-0.5, 0.5) * a for a in ax)
        maps.append(torch.polar(torch.exp(-d2 / (2 * 0.8 ** 2)), ph))
    m = torch.stack(maps)
    return (m / m.abs().square().sum(0).sqrt()).to(torch.complex64).contiguous()


def _wrap(k):
    return (k + math.pi) % (2 * math.pi) - math.pi


def _plane(kind, a, b, n, turn):
    """(a b, 2) float64: a golden-angle spokes of b samples, or a spiral interleaves of b samples
    (8-fold undersampled at the edge), turned by `turn` radians."""
    if kind == "radial":
        th = np.arange(a)[:, None] * (math.pi * (math.sqrt(5.0) - 1.0) / 2.0) + turn
        kr = -math.pi + 2 * math.pi * np.arange(b)[None, :] / b
        k = kr * np.exp(1j * th)
    else:
        T = 1.5 * n / (16.0 * a)
        t = np.arange(b) / b
        il = np.arange(a)[:, None]
        k = math.pi * t ** 1.5 * np.exp(1j * (2 * math.pi * (T * t + il / a) + turn))
    k = k.reshape(-1)
    return np.stack([_wrap(k.real), _wrap(k.imag)], axis=1)


def _traj(case, r):
    turn = r.uniform(0, 2 * math.pi)
    if "nz" in case:   # a stack of spirals: one plane of spirals per kz
        n, out = max(case["ny"], case["nx"]), []
        for p in range(case["nz"]):
            k = _plane("spiral", case["a"], case["b"], n, turn + p * math.pi * (3.0 - math.sqrt(5.0)))
            kz = 2 * math.pi * (p - case["nz"] / 2) / case["nz"]
            out.append(np.concatenate([k, np.full((len(k), 1), kz)], axis=1))
        return torch.from_numpy(np.concatenate(out).astype(np.float32)).cuda()
    return torch.from_numpy(_plane(case["kind"], case["a"], case["b"], case["n"], turn).astype(np.float32)).cuda()


def _noise(seed, shape, std, dtype=torch.complex64):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return (torch.randn(tuple(shape) + (2,), generator=g, device="cuda") * (std / math.sqrt(2))).view(torch.complex64) \
        .squeeze(-1).to(dtype)


def _shape(case):
    return (case["nz"], case["ny"], case["nx"]) if "nz" in case else (case["n"], case["n"])


def _slice_case(case, i):
    """The i-th slice of a batch: alike, or of uneven size, coil count and trajectory."""
    if case["op"] != "batch_hqs":
        return case
    n = (320, 256, 384)[i % 3]
    L = 8 + (5 * i + case["L"]) % 13
    kind = ("spiral", "radial")[i % 2]
    a, b = (12 + 5 * i % 13, 1024 + 317 * i) if kind == "spiral" else (case["a"] - 5 * i % 17, 2 * n)
    return dict(case, n=n, L=L, kind=kind, a=a, b=b)


def _scan(case, seed):
    """What a program holds for one slice or volume: maps, trajectory, k-space data, an image."""
    r = random.Random(seed * 1009 + 17)
    shape = _shape(case)
    x, S, k = _phantom(shape, r), _coil_maps(shape, case["L"], r), _traj(case, r)
    y = _nudft(x, S, k, case) + _noise(seed + 5, (case["L"], k.shape[0]), 0.01)
    return dict(x=x, S=S, k=k, y=y.contiguous())


# ------------------------------------------------------------- the operators as sums
# A x and A^H y by their definition, as matrix products over the axes, in the type of x: for the data
# (complex64) and for exact() (complex128).  A volume's trajectory is a stack of planes of one kz each.
def _axis(k, n, sign, dtype):
    d = torch.arange(n, device="cuda", dtype=torch.float64) - n // 2
    return torch.polar(torch.ones((), device="cuda", dtype=torch.float64), sign * k.double()[:, None] * d).to(dtype)


def _planes(k, case):
    m = k.shape[0] // case["nz"]
    return [(k[p * m, 2:3], k[p * m:(p + 1) * m, :2], slice(p * m, (p + 1) * m)) for p in range(case["nz"])]


def _nudft(x, S, k, case, dtype=torch.complex64):
    S, x = S.to(dtype), x.to(dtype)
    if x.dim() == 3:
        out = torch.empty((S.shape[0], k.shape[0]), dtype=dtype, device="cuda")
        for kz, kp, at in _planes(k, case):
            ez = _axis(kz, x.shape[0], -1.0, dtype)[0]
            v = torch.einsum("z,lzyx->lyx", ez, S * x)
            ex, ey = _axis(kp[:, 0], x.shape[2], -1.0, dtype), _axis(kp[:, 1], x.shape[1], -1.0, dtype)
            out[:, at] = ((v @ ex.T) * ey.T).sum(1)
        return out / math.sqrt(x.numel())
    ex, ey = _axis(k[:, 0], x.shape[1], -1.0, dtype), _axis(k[:, 1], x.shape[0], -1.0, dtype).T.contiguous()
    return torch.stack([(((s * x) @ ex.T) * ey).sum(0) for s in S]) / math.sqrt(x.numel())


def _nudft_adjoint(y, S, k, case, dtype=torch.complex128):
    S, y = S.to(dtype), y.to(dtype)
    shape = S.shape[1:]
    if len(shape) == 3:
        out = torch.zeros(tuple(S.shape), dtype=dtype, device="cuda")
        for kz, kp, at in _planes(k, case):
            ez = _axis(kz, shape[0], 1.0, dtype)[0]
            ex, ey = _axis(kp[:, 0], shape[2], 1.0, dtype), _axis(kp[:, 1], shape[1], 1.0, dtype)
            plane = (ey.T * y[:, None, at]) @ ex
            out += ez[None, :, None, None] * plane[:, None]
        return (S.conj() * out).sum(0) / math.sqrt(out[0].numel())
    ex, ey = _axis(k[:, 0], shape[1], 1.0, dtype), _axis(k[:, 1], shape[0], 1.0, dtype)
    x = torch.zeros(tuple(shape), dtype=dtype, device="cuda")
    for s, v in zip(S, y):
        x += s.conj() * ((ey.T * v) @ ex)
    return x / math.sqrt(x.numel())


def _kernel(k, shape, case):
    """The first column of A^H A's circulant embedding: t(d) = Npix^-1 sum_j exp(i k_j d), zero at d = -N."""
    off = [torch.cat([torch.arange(n), torch.arange(-n, 0)]).double().cuda() for n in shape]
    ax = lambda kk, d: torch.polar(torch.ones((), device="cuda", dtype=torch.float64), kk.double()[:, None] * d)
    if len(shape) == 3:
        c = torch.zeros([2 * n for n in shape], dtype=torch.complex128, device="cuda")
        for kz, kp, _ in _planes(k, case):
            plane = ax(kp[:, 1], off[1]).T @ ax(kp[:, 0], off[2])
            c += ax(kz, off[0])[0][:, None, None] * plane
    else:
        c = ax(k[:, 1], off[0]).T @ ax(k[:, 0], off[1])
    for d, n in enumerate(shape):
        c.select(d, n).zero_()
    return c / math.prod(shape)


def _normal(x, S, kh):
    """A^H A x through the circulant embedding, kh = FFT of the kernel (real)."""
    dims, out = tuple(range(x.dim())), torch.zeros_like(x)
    for s in S:
        v = torch.fft.fftn(s * x, s=kh.shape, dim=dims)
        v = torch.fft.ifftn(v * kh, dim=dims)[tuple(slice(0, n) for n in x.shape)]
        out += s.conj() * v
    return out


def _density(c, shape):
    """Symbol of the density preconditioner: eigenvalues of the circulant nearest the Toeplitz part."""
    for d, n in enumerate(shape):
        q = torch.arange(n, device="cuda").double() / n
        sh = [1] * len(shape)
        sh[d] = n
        c = c.narrow(d, 0, n) * (1 - q).view(sh) + c.narrow(d, n, n) * q.view(sh)
    return torch.fft.fftn(c).real


def _exact_system(scan, case):
    shape = _shape(case)
    S = scan["S"].to(torch.complex128)
    c = _kernel(scan["k"], shape, case)
    kh, lam = torch.fft.fftn(c).real, _density(c, shape)
    return S, kh, lam


def _pcg(S, kh, lam, a, b, rhs, x, its):
    """`its` conjugate-gradient iterations on (a A^H A + b I) x = rhs with the density preconditioner."""
    H = lambda v: a * _normal(v, S, kh) + b * v
    m = (a * lam.clamp(min=0) + b).clamp(min=0.25 * b).rsqrt()
    M = lambda v: torch.fft.ifftn(torch.fft.fftn(v) * m)
    dot = lambda u, v: (u.conj() * v).real.sum()
    r = rhs - H(x) if bool(x.abs().max() > 0) else rhs.clone()
    z = M(r)
    p, rz = z.clone(), dot(r, z)
    for _ in range(its):
        q = H(p)
        al = rz / dot(p, q)
        x, r = x + al * p, r - al * q
        z = M(r)
        rz, old = dot(r, z), rz
        p = z + (rz / old) * p
    return x


def _blur(x, s):
    """Periodic Gaussian smoothing, std s pixels, radius ceil(3 s); identity below 0.1."""
    if s < 0.1:
        return x
    r = int(math.ceil(3 * s))
    g = [math.exp(-i * i / (2 * s * s)) for i in range(-r, r + 1)]
    for d in range(x.dim()):
        x = sum(w / sum(g) * torch.roll(x, r - i, dims=d) for i, w in enumerate(g))
    return x


# ------------------------------------------------------------------ the calls
def _schedule(case):
    K = case["outer"]
    mu = [case["mu"] * 0.6 ** k for k in range(K)]
    return mu, list(mu)


def _net_params(r):
    layers, out = ((2, 32), (32, 32), (32, 32), (32, 2)), []
    g = np.random.default_rng(r.randrange(1 << 30))
    for ci, co in layers:
        out.append((g.normal(size=(co, ci, 3, 3)) * math.sqrt(2.0 / (9 * ci)), g.normal(size=co) * 0.05))
    return np.concatenate([np.concatenate([w.ravel(), b]) for w, b in out]).astype(np.float32)


def prepare(case, seed):
    op, seed = case["op"], int(seed)
    s = dict(case=case)
    if op == "denoise":
        r = random.Random(seed)
        s["net"] = hq.Net()
        s["params"] = _net_params(r)
        s["net"].set_params(s["params"])
        x = _phantom((case["n"], case["m"]), r)
        s["x"] = (x + _noise(seed, x.shape, case["sigma"])).contiguous()
        s["out"] = torch.empty_like(s["x"])
        return s
    if op in ("batch_step", "batch_hqs"):
        cs = [_slice_case(case, i) for i in range(case["count"])]
        scans = [_scan(c, seed * 131 + i) for i, c in enumerate(cs)]
        s["plans"] = [hq.plan_create(v["k"], c["n"], c["n"], v["S"], c["W"], 2.0) for v, c in zip(scans, cs)]
        s["batch"] = hq.Batch(s["plans"])
        s["y"], s["z"] = [v["y"] for v in scans], [v["x"] for v in scans]
        s["rhs"] = [torch.empty_like(z) for z in s["z"]]
        s["out"] = [torch.empty_like(z) for z in s["z"]]
        return s
    v = _scan(case, seed)
    if op.startswith("vol_"):
        s["plan"] = hq.plan3d_create(v["k"], _shape(case), v["S"], case["W"], 2.0)
    else:
        s["plan"] = hq.plan_create(v["k"], case["n"], case["n"], v["S"], case["W"], 2.0)
    s.update(x=v["x"], y=v["y"], out=torch.empty_like(v["y"] if "forward" in op else v["x"]))
    if op == "step":
        s["rhs"] = torch.empty_like(v["x"])
    if op == "vol_solve":
        b0 = _nudft_adjoint(v["y"], v["S"], v["k"], case, torch.complex64)
        s["rhs"] = (b0 + case["mu"] * v["x"]).contiguous()
    return s


def run(s):
    case, op = s["case"], s["case"]["op"]
    if op == "forward":
        return hq.forward(s["plan"], s["x"], s["out"])
    if op == "adjoint":
        return hq.adjoint(s["plan"], s["y"], s["out"])
    if op == "normal":
        return hq.toeplitz_normal(s["plan"], s["x"], s["out"])
    if op == "step":
        hq.adjoint_axpy(s["plan"], s["y"], case["mu"], s["x"], s["rhs"])
        hq.dc_solve(s["plan"], 1.0, case["mu"], s["rhs"], s["out"], max_iter=case["its"], rel_tol=0.0,
                    mode=hq.HQS_SOLVE_FUSED | hq.HQS_SOLVE_X0_ZERO, want_info=False)
        return s["rhs"], s["out"]
    if op == "batch_step":
        s["batch"].adjoint_axpy(s["y"], case["mu"], s["z"], s["rhs"])
        s["batch"].dc_solve(s["rhs"], s["out"], 1.0, case["mu"], max_iter=case["its"], rel_tol=0.0)
        return s["rhs"], s["out"]
    if op == "batch_hqs":
        mu, sigma = _schedule(case)
        for o, z in zip(s["out"], s["z"]):
            o.copy_(z)
        s["batch"].run(s["y"], s["out"], mu, sigma, cg_iters=case["its"])
        return s["out"]
    if op == "denoise":
        return s["net"].denoise(s["x"], s["out"], case["sigma"])
    if op == "vol_forward":
        return hq.forward3d(s["plan"], s["x"], s["out"])
    if op == "vol_adjoint":
        return hq.adjoint3d(s["plan"], s["y"], s["out"])
    if op == "vol_normal":
        return hq.toeplitz_normal3d(s["plan"], s["x"], s["out"])
    s["out"].zero_()
    hq.dc_solve3d(s["plan"], 1.0, case["mu"], s["rhs"], s["out"], max_iter=case["its"], rel_tol=0.0)
    return s["out"]


# ------------------------------------------------------------------ work and exact values
def _points(case):
    return case["a"] * case["b"] * case.get("nz", 1)


def _work(case, op):
    shape, L = _shape(case), case["L"]
    n, d, M, W = math.prod(shape), len(shape), _points(case), case["W"]
    # one pruned pair of transforms to and from the doubled grid, and the coil multiply and sum
    G = 2 ** d * n
    half = 5.0 * L * sum(2 ** (i + 1) * n * math.log2(2 * shape[i]) for i in range(d))
    coils = 14.0 * L * n
    maps, image, data, traj = 8.0 * L * n, 8.0 * n, 8.0 * L * M, 4.0 * d * M
    if op == "forward":
        return maps + image + data + traj, half + coils + 4.0 * L * M * W ** d
    if op == "adjoint":
        return maps + image + data + traj, half + coils + 4.0 * L * M * W ** d
    aha = 2 * half + 2 * coils + 2.0 * L * G
    if op == "normal":
        return maps + 2 * image + 4.0 * G, aha
    it = aha + 10.0 * n * math.log2(n) + 24.0 * n
    return maps + 2 * image + 4.0 * G + 4.0 * n, case["its"] * it


def work(case):
    op = case["op"].replace("vol_", "")
    if op == "denoise":
        n = case["n"] * case["m"]
        return dict(bytes=16.0 * n, flops=2.0 * n * 9 * (2 * 32 + 32 * 32 + 32 * 32 + 32 * 2))
    count = case.get("count", 1)
    total = [0.0, 0.0]
    for i in range(count):
        c = _slice_case(case, i)
        parts = [("solve", 1)]
        if op in ("forward", "adjoint", "normal"):
            parts = [(op, 1)]
        elif op in ("step", "batch_step"):
            parts = [("adjoint", 1), ("solve", 1)]
        elif op == "batch_hqs":
            # the iterations of every outer step and the apply that starts it
            parts = [("adjoint", 1), ("solve", case["outer"] * (1 + 1.0 / case["its"]))]
        for p, k in parts:
            b, f = _work(c, p)
            total[0] += b
            total[1] += k * f
    return dict(bytes=total[0], flops=total[1])


def exact(case, seed):
    op, seed = case["op"], int(seed)
    if op == "denoise":
        r = random.Random(seed)
        vec = torch.from_numpy(_net_params(r)).double().cuda()
        x = _phantom((case["n"], case["m"]), r)
        x = (x + _noise(seed, x.shape, case["sigma"])).to(torch.complex128)
        sig = float(np.float32(case["sigma"]))
        h, at = torch.stack([x.real, x.imag])[None] / sig, 0
        for i, (ci, co) in enumerate(((2, 32), (32, 32), (32, 32), (32, 2))):
            w = vec[at:at + 9 * ci * co].view(co, ci, 9)
            b = vec[at + 9 * ci * co:at + 9 * ci * co + co]
            at += 9 * ci * co + co
            p = torch.nn.functional.unfold(h, 3, padding=1).view(ci, 9, -1)
            h = (torch.einsum("oct,ctp->op", w, p) + b[:, None]).view(1, co, *x.shape)
            h = h.relu() if i < 3 else h
        return x - sig * torch.complex(h[0, 0], h[0, 1])
    f32 = lambda v: float(np.float32(v))
    if op in ("batch_step", "batch_hqs"):
        rhss, outs = [], []
        for i in range(case["count"]):
            c = _slice_case(case, i)
            v = _scan(c, seed * 131 + i)
            S, kh, lam = _exact_system(v, c)
            b0, x = _nudft_adjoint(v["y"], v["S"], v["k"], c), v["x"].to(torch.complex128)
            if op == "batch_step":
                rhss.append(b0 + f32(case["mu"]) * x)
                outs.append(_pcg(S, kh, lam, 1.0, f32(case["mu"]), rhss[-1], torch.zeros_like(x), case["its"]))
                continue
            mu, sigma = _schedule(case)
            for m, sg in zip(mu, sigma):
                u = _pcg(S, kh, lam, 1.0, f32(m), b0 + f32(m) * x, x, case["its"])
                x = _blur(u, 1.5 * f32(sg) / f32(sigma[0]))
            outs.append(x)
        return (rhss, outs) if op == "batch_step" else outs
    v = _scan(case, seed)
    x = v["x"].to(torch.complex128)
    if op.endswith("forward"):
        return _nudft(v["x"], v["S"], v["k"], case, torch.complex128)
    if op.endswith("adjoint"):
        return _nudft_adjoint(v["y"], v["S"], v["k"], case)
    S, kh, lam = _exact_system(v, case)
    if op.endswith("normal"):
        return _normal(x, S, kh)
    if op == "step":
        rhs = _nudft_adjoint(v["y"], v["S"], v["k"], case) + f32(case["mu"]) * x
        return rhs, _pcg(S, kh, lam, 1.0, f32(case["mu"]), rhs, torch.zeros_like(x), case["its"])
    b0 = _nudft_adjoint(v["y"], v["S"], v["k"], case, torch.complex64)
    rhs = (b0 + case["mu"] * v["x"]).to(torch.complex128)
    return _pcg(S, kh, lam, 1.0, f32(case["mu"]), rhs, torch.zeros_like(x), case["its"])
