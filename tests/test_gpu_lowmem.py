"""Low-memory plans: what they hold, what is live while they are made, and the precision of
their depth sums."""
import ctypes

import numpy as np
import pytest

import oracle
from paper_2301_09710_gb300 import synthetic

from gpu_helpers import assert_close, dev, host, make_plan, need_gpu, torch

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _gpu():
    need_gpu()


# nx, nz, nview, taps, separable: MB that the bound of a plan on the general low-memory kernels
# comes to (image, projections, compressed adjacency lists and a slab of at most 256 MiB)
GENERAL_MB = [
    (96, 64, 60, 21, True, 170.1),
    (128, 80, 128, 37, True, 364.0),
    (160, 96, 120, 29, True, 413.0),
    (192, 128, 128, 37, True, 503.5),
    (256, 64, 128, 21, True, 629.3),
    (512, 64, 120, 11, True, 1618.1),
    (96, 64, 60, 21, False, 171.7),
    (64, 32, 64, 11, True, 45.1),
    (192, 5, 128, 3, True, 267.0),
]


@pytest.mark.parametrize("case", GENERAL_MB, ids=[f"{c[0]}x{c[1]}v{c[2]}p{c[3]}{'' if c[4] else 'full'}" for c in GENERAL_MB])
def test_low_memory_bound_does_not_exceed_the_general_kernels(case):
    from paper_2301_09710_gb300.projector import plan_bytes
    nx, nz, nview, p, separable, mb = case
    assert plan_bytes(nx, nz, nview, p, p, separable=separable, low_memory=True) <= 1e6 * (mb + 0.05)


def _pool_high():
    """Read and reset the high-water mark of the device's memory pool (bytes in use)."""
    rt = ctypes.CDLL("libcudart.so.13")
    pool, high, zero = ctypes.c_void_p(), ctypes.c_uint64(), ctypes.c_uint64(0)
    assert rt.cudaDeviceGetDefaultMemPool(ctypes.byref(pool), torch.cuda.current_device()) == 0
    used_now, used_high = 7, 8  # cudaMemPoolAttrUsedMemCurrent, cudaMemPoolAttrUsedMemHigh
    assert rt.cudaMemPoolGetAttribute(pool, used_high, ctypes.byref(high)) == 0
    assert rt.cudaMemPoolSetAttribute(pool, used_high, ctypes.byref(zero)) == 0  # to the bytes now in use
    now = ctypes.c_uint64()
    assert rt.cudaMemPoolGetAttribute(pool, used_now, ctypes.byref(now)) == 0
    return high.value, now.value


@pytest.mark.parametrize("kind", ["lowmem", "default", "recompute"])
@pytest.mark.parametrize("nx,nz,nview,p", [(96, 64, 60, 21), (64, 5, 90, 3), (129, 7, 100, 5)])
def test_plan_creation_stays_within_plan_bytes(kind, nx, nz, nview, p):
    """The bound covers what is live while the plan is made, not only what it keeps: the pool's
    high-water mark over creation and one EM update.  Up to 256 bytes per allocation are rounding."""
    from paper_2301_09710_gb300 import SpectPlan
    from paper_2301_09710_gb300.projector import plan_bytes
    kw = {"lowmem": {"low_memory": True}, "default": {}, "recompute": {"recompute_attenuation": True}}[kind]
    taps = np.full((1, nx, p), 1.0 / p, np.float32)
    x, y = dev(np.ones((nz, nx, nx))), dev(np.ones((nview, nz, nx)))
    torch.cuda.synchronize()
    _, before = _pool_high()
    plan = SpectPlan(nx, nz, nview, mu=dev(np.full((nz, nx, nx), 0.01)), fx=taps, fz=taps, **kw)
    plan.em_step(x, y, None, niter=1)
    torch.cuda.synchronize()
    high, _ = _pool_high()
    bound = plan_bytes(nx, nz, nview, p, p, **kw)
    held = plan.info()["device_bytes"]
    plan.check()
    plan.close()
    assert held <= bound and high - before <= bound + 64 * 256, (held, high - before, bound)


@pytest.mark.parametrize("path,nx,nz,nview", [("lowmem", 32, 16, 300), ("lowmem", 16, 600, 300), ("direct_lowmem", 32, 16, 3)])
def test_low_memory_depth_sums_are_compensated_over_all_depths(path, nx, nz, nview):
    """Planes 2^24, 1, 0 ..., -2^24, 0 ... under a one-tap PSF at angle 0: every term and every
    compensation term is a whole number that FP32 holds, so the compensated sum over all depths is
    exact (one per sixteen planes), while a sum that drops the 1, within a group of planes or
    between groups, gives 0.  16x600: more work items than a block has threads.
    Enough views that several planes go to a block."""
    from paper_2301_09710_gb300 import SpectPlan
    x = np.zeros((nz, nx, nx), np.float32)
    x[:, 0::16], x[:, 1::16], x[:, 8::16] = 2.0 ** 24, 1.0, -2.0 ** 24
    one = np.ones((1, nx, 1), np.float32)
    kw = {"fx": one, "fz": one} if path == "lowmem" else {"psf": one[..., None]}
    plan = SpectPlan(nx, nz, nview, angles=[0.0] * nview, low_memory=True, **kw)
    got = host(plan.forward(dev(x)))
    plan.check()
    plan.close()
    assert np.array_equal(got, np.full((nview, nz, nx), nx // 16, np.float64))


def test_flat_low_memory_plan_makes_its_tables_in_each_pass():
    """160x160x5: one view per pass, the rotation tables of the pass made in it; A, A' and an EM
    step against the oracle."""
    prob = synthetic.random_problem(3, nx=160, nz=5, nview=20, px=9, pz=9, mu_scale=0.02)
    ang = oracle.default_angles(20)
    plan = make_plan(prob, ang, "lowmem")
    assert plan.info()["view_chunk"] == 1
    psf = oracle.psf_from_factors(prob.fx, prob.fz)
    assert_close(host(plan.forward(dev(prob.x))), oracle.forward(prob.x, prob.mu, psf, prob.dy, ang), what="A x")
    y = np.random.default_rng(3).uniform(0.5, 1.5, plan.proj_shape).astype(np.float32)
    assert_close(host(plan.back(dev(y))), oracle.back(y, prob.mu, psf, prob.dy, ang), what="A' y")
    x0 = np.full(prob.x.shape, 0.5, np.float32)
    xg = dev(x0)
    plan.em_step(xg, dev(y), None, niter=1)
    assert_close(host(xg), oracle.em_step(x0, y, None, prob.mu, psf, prob.dy, ang), what="EM step")
    plan.check()
    plan.close()


def test_low_memory_plan_that_fits_only_the_general_kernels():
    """A full PSF of its own for each of 218 views of a tiny volume: the tap records of the fused
    kernels would take more than the general kernels' plan, which serves it within its bound."""
    from paper_2301_09710_gb300.projector import plan_bytes
    nx, nz, nview, px, pz = 8, 2, 218, 9, 31
    prob = synthetic.random_problem(5, nx=nx, nz=nz, nview=nview, px=px, pz=pz, nview_psf=nview, mu_scale=0.05)
    ang = oracle.default_angles(nview)
    plan = make_plan(prob, ang, "direct_lowmem")
    assert plan.info()["device_bytes"] <= plan_bytes(nx, nz, nview, px, pz, nview, separable=False, low_memory=True)
    psf = prob.full_psf().astype(np.float64)
    assert_close(host(plan.forward(dev(prob.x))), oracle.forward(prob.x, prob.mu, psf, prob.dy, ang), what="A x")
    y = np.random.default_rng(5).uniform(0.5, 1.5, plan.proj_shape).astype(np.float32)
    assert_close(host(plan.back(dev(y))), oracle.back(y, prob.mu, psf, prob.dy, ang), what="A' y")
    plan.check()
    plan.close()
