"""Scenarios of tests/test_host_faults.py, each run in a process of its own:

    python tests/host_fault_runs.py <stand-in .so> <library .so> <scenario>

The stand-in replaces the CUDA runtime (fake_cudart.cpp), so device pointers are host memory
and kernels do nothing; what is checked is the host code around them.
"""
import ctypes as C
import sys

OOM = -2
VP, LONG = C.c_void_p, C.c_long


class Fake:
    def __init__(self, path):
        self.lib = C.CDLL(path, mode=C.RTLD_GLOBAL)
        for name, ret in [("fake_calls", LONG), ("fake_bad", LONG), ("fake_live", LONG), ("fake_bytes", C.c_size_t),
                          ("fake_hash", C.c_ulonglong), ("fake_launches", C.c_char_p)]:
            getattr(self.lib, name).restype = ret
        self.lib.fake_fail_call.argtypes = self.lib.fake_fail_malloc.argtypes = [LONG]

    def __getattr__(self, name):
        return getattr(self.lib, "fake_" + name)

    def device(self, nbytes):
        p = VP()
        assert self.lib.cudaMalloc(C.byref(p), C.c_size_t(nbytes)) == 0
        return p


def net_scratch_holds_the_samples(fake, hqs):
    """One large image first, then many small ones with fewer pixels and tiles in all: the
    per-sample losses need room for the second count."""
    net = VP()
    assert hqs.hqs_net_create(C.byref(net)) == 0
    x = fake.device(2 * 256 * 256 * 4)
    loss = C.c_double()
    lr = C.c_float(1e-3)
    assert hqs.hqs_net_train_step(net, x, x, 1, 256, 256, lr, C.byref(loss), None) == 0
    assert hqs.hqs_net_train_step(net, x, x, 128, 4, 4, lr, C.byref(loss), None) == 0
    assert fake.bad() == 0, "per-sample losses copied from beyond their buffer"
    hqs.hqs_net_destroy(net)


def net_scratch_after_failed_growth(fake, hqs):
    """A growth that runs out of memory leaves no buffer behind; the next, smaller call has
    to allocate what it needs (not launch on the pointers that were freed)."""
    for k in range(1, 8):
        net = VP()
        assert hqs.hqs_net_create(C.byref(net)) == 0
        x = fake.device(2 * 128 * 128 * 4)
        base = fake.bytes()
        assert hqs.hqs_net_forward(net, x, x, 1, 64, 64, None) == 0
        fake.fail_malloc(k)
        assert hqs.hqs_net_forward(net, x, x, 1, 128, 128, None) == OOM
        fake.fail_malloc(-1)
        fake.lib.cudaGetLastError()
        assert hqs.hqs_net_forward(net, x, x, 1, 32, 32, None) == 0
        # activations and gradients: 5 x 32 + 2 planes of the image
        assert fake.bytes() - base >= (5 * 32 + 2) * 32 * 32 * 4, k
        hqs.hqs_net_destroy(net)


def make_plan(fake, hqs, n, M=300, L=4, W=4):
    plan = VP()
    traj, smaps = fake.device(M * 8), fake.device(L * n * n * 8)
    assert hqs.hqs_plan_create(C.byref(plan), traj, C.c_int64(M), n, n, L, smaps, W, C.c_float(2.0), None) == 0
    return plan


def learned_scratch_after_failed_growth(fake, hqs):
    """The same for the learned preconditioner's image buffers."""
    small, mid, big = (make_plan(fake, hqs, n) for n in (32, 64, 128))
    r = fake.device(128 * 128 * 8)
    one = C.c_float(1.0)
    for k in range(1, 4):
        net = VP()
        assert hqs.hqs_net_create(C.byref(net)) == 0
        for p in (small, mid, big):
            assert hqs.hqs_plan_set_net(p, net) == 0
        # the network's own scratch at its largest, so that only the image buffers grow
        assert hqs.hqs_net_forward(net, r, r, 1, 128, 128, None) == 0
        base = fake.bytes()
        assert hqs.hqs_learned_precond_apply(mid, one, one, r, r, None) == 0
        fake.fail_malloc(k)
        assert hqs.hqs_learned_precond_apply(big, one, one, r, r, None) == OOM
        fake.fail_malloc(-1)
        fake.lib.cudaGetLastError()
        assert hqs.hqs_learned_precond_apply(small, one, one, r, r, None) == 0
        assert fake.bytes() - base >= (2 + 4) * 32 * 32 * 4, k
        hqs.hqs_net_destroy(net)


def next_call_after_oom(fake, hqs):
    """Every allocation of the creating calls fails once; the refusal must not be reported
    again by the next call, which has nothing to do with it."""
    good = make_plan(fake, hqs, 32)
    img, ksp = fake.device(64 * 64 * 8), fake.device(64 * 1024 * 8)
    traj, maps3 = fake.device(3 * 500 * 4), fake.device(2 * 16 ** 3 * 8)
    two, zero, h = C.c_float(2.0), C.c_float(0.0), VP()

    def plan():
        return hqs.hqs_plan_create(C.byref(h), traj, C.c_int64(200), 32, 32, 4, ksp, 4, two, None)

    def volume():
        return hqs.hqs_plan3d_create(C.byref(h), traj, C.c_int64(200), 16, 16, 16, 2, maps3, 4, two, None)

    def batch():
        return hqs.hqs_batch_create(C.byref(h), (VP * 1)(plan64), 1, 4)

    def retile():
        return hqs.hqs_plan_retile(good, 16, None)

    def smaps():
        return hqs.hqs_estimate_smaps(traj, C.c_int64(200), ksp, None, 32, 2, 4, two, C.c_float(8.0), zero, img, None)

    plan64 = make_plan(fake, hqs, 64)
    destroy = {plan: hqs.hqs_plan_destroy, volume: hqs.hqs_plan3d_destroy, batch: hqs.hqs_batch_destroy}
    for call in (plan, volume, batch, retile, smaps):
        refused = 0
        while True:
            live = fake.live()
            fake.fail_malloc(refused + 1)
            rc = call()
            fake.fail_malloc(-1)
            if rc == 0:
                break
            refused += 1
            assert rc == OOM and refused < 100, (call.__name__, rc)
            assert fake.live() == live, (call.__name__, refused, "memory lost")
            assert hqs.hqs_adjoint(good, ksp, img, None) == 0, (call.__name__, refused)
        assert refused > 0, call.__name__
        if call in destroy:
            destroy[call](h)


class PlanInfo(C.Structure):
    _fields_ = [("ny", C.c_int), ("nx", C.c_int), ("coils", C.c_int), ("kernel_width", C.c_int),
                ("oversamp", C.c_float), ("grid", C.c_int), ("npoints", C.c_int64), ("kb_beta", C.c_double),
                ("device_bytes", C.c_size_t), ("nsub", C.c_int), ("tile", C.c_int)]


def retile_fails_whole(fake, hqs):
    """Every call that hqs_plan_retile makes fails once: a refusal leaves the plan's arrays and
    its bin size as they were."""
    plan, info = make_plan(fake, hqs, 32), PlanInfo()
    # new blocks look different, so that a copy into the plan's shows
    fake.mark()
    fake.pattern(0x5a)
    before, live, k = fake.hash(), fake.live(), 0
    while True:
        k += 1
        fake.clear_launches()
        fake.fail_call(k)
        rc = hqs.hqs_plan_retile(plan, 16, None)
        fake.fail_call(-1)
        assert hqs.hqs_plan_get_info(plan, C.byref(info)) == 0
        replaced = b"k_replace_points" in fake.launches()
        assert fake.live() == live and fake.hash() == before, (k, rc)
        assert replaced == (info.tile == 16), (k, rc)
        if replaced:
            break
        assert rc != 0 and k < 200
    assert k > 10


if __name__ == "__main__":
    fake = Fake(sys.argv[1])
    hqs = C.CDLL(sys.argv[2])
    hqs.hqs_net_destroy.restype = hqs.hqs_plan_destroy.restype = hqs.hqs_plan3d_destroy.restype = None
    hqs.hqs_batch_destroy.restype = None
    globals()[sys.argv[3]](fake, hqs)
    assert fake.bad() == 0
