"""The blur kernels at the edges of their launch shapes, A and A' against the FP64 oracle:
planes of more rows than one tensor box (256), more work items than threads (sums in shared
memory), a last tile of one column, tiles narrower than the PSF's halo, one-plane groups.
Tolerance: the 2e-6 / 1e-4 bars of the other parity tests (FP32 FIR of at most 37 terms per
pass, the depth sum in groups)."""
import numpy as np
import pytest

import oracle
from paper_2301_09710_gb300 import synthetic

from gpu_helpers import assert_close, dev, host, make_plan, need_gpu

pytestmark = pytest.mark.gpu

# nx, nz, nview, px, pz, nview_psf, seed, (fused_J, adj_J, tiles) or None for the defaults
SHAPES = [
    (16, 300, 3, 5, 5, 1, 1, None),        # two boxes per plane
    (16, 600, 2, 3, 3, 1, 2, None),        # 608 k-pass items: accumulators in shared memory, three boxes
    (33, 17, 5, 21, 9, 5, 3, None),        # last tile: one column; a partial k run of one row
    (65, 16, 3, 37, 37, 1, 4, (1, 1, 5)),  # one plane per group; tiles of 16 columns under a 37-tap PSF
    (40, 47, 4, 11, 13, 4, 5, (7, 5, 2)),  # ragged groups, the padding of a wider bucket on one axis
    (100, 66, 2, 29, 29, 1, 6, (32, 32, 1)),  # whole planes
]


@pytest.mark.parametrize("case", SHAPES, ids=[f"{c[0]}x{c[1]}p{c[3]}x{c[4]}" for c in SHAPES])
def test_blur_launch_shapes(case):
    need_gpu()
    nx, nz, nview, px, pz, nvp, seed, shape = case
    prob = synthetic.random_problem(seed, nx=nx, nz=nz, nview=nview, px=px, pz=pz, nview_psf=nvp, mu_scale=0.05)
    rng = np.random.default_rng(seed)
    ang = rng.uniform(0, 2 * np.pi, nview)
    plan = make_plan(prob, ang, "fused")
    assert plan.info()["fused"]
    if shape:
        plan.set_tuning(*shape)
    psf = oracle.psf_from_factors(prob.fx, prob.fz)
    assert_close(host(plan.forward(dev(prob.x))), oracle.forward(prob.x, prob.mu, psf, prob.dy, ang), what="A x")
    yy = rng.uniform(0, 1, plan.proj_shape).astype(np.float32)
    assert_close(host(plan.back(dev(yy))), oracle.back(yy, prob.mu, psf, prob.dy, ang), what="A' y")
    plan.check()
    plan.close()


# nx, nz, nview, px, pz, nview_psf, seed: the full-PSF kernels' tiles
DIRECT = [
    (33, 17, 5, 21, 9, 5, 3),   # last tile: one column; zero tap rows of the bucket
    (50, 5, 7, 13, 13, 1, 4),   # PSF taller than the plane
    (16, 300, 2, 5, 5, 1, 5),   # two boxes per plane
    (19, 40, 3, 37, 37, 1, 6),  # PSF wider than the plane: both halos in one tile
]


@pytest.mark.parametrize("case", DIRECT, ids=[f"{c[0]}x{c[1]}p{c[3]}x{c[4]}" for c in DIRECT])
def test_full_psf_launch_shapes(case):
    need_gpu()
    nx, nz, nview, px, pz, nvp, seed = case
    prob = synthetic.random_problem(seed, nx=nx, nz=nz, nview=nview, px=px, pz=pz, nview_psf=nvp, mu_scale=0.05)
    rng = np.random.default_rng(seed)
    ang = rng.uniform(0, 2 * np.pi, nview)
    plan = make_plan(prob, ang, "direct")
    assert plan.info()["fused"]
    psf = prob.full_psf().astype(np.float64)
    assert_close(host(plan.forward(dev(prob.x))), oracle.forward(prob.x, prob.mu, psf, prob.dy, ang), what="A x")
    yy = rng.uniform(0, 1, plan.proj_shape).astype(np.float32)
    assert_close(host(plan.back(dev(yy))), oracle.back(yy, prob.mu, psf, prob.dy, ang), what="A' y")
    plan.check()
    plan.close()


@pytest.mark.parametrize("path", ["lowmem", "direct_lowmem"])
def test_psf_wider_than_the_fused_kernels(path):
    """A 41-tap PSF: the low-memory kernels (a low-memory plan of up to 37 taps runs the
    fused kernels in view chunks), A, A' and one EM step."""
    need_gpu()
    nx, nz, nview, p = 40, 18, 5, 41
    prob = synthetic.random_problem(7, nx=nx, nz=nz, nview=nview, px=p, pz=p, mu_scale=0.05)
    ang = oracle.default_angles(nview)
    plan = make_plan(prob, ang, path)
    assert not plan.info()["fused"]
    psf = oracle.psf_from_factors(prob.fx, prob.fz) if path == "lowmem" else prob.full_psf().astype(np.float64)
    v_o = oracle.forward(prob.x, prob.mu, psf, prob.dy, ang)
    assert_close(host(plan.forward(dev(prob.x))), v_o, what="A x")
    yy = np.random.default_rng(8).uniform(0.5, 1.5, plan.proj_shape).astype(np.float32)
    assert_close(host(plan.back(dev(yy))), oracle.back(yy, prob.mu, psf, prob.dy, ang), what="A' y")
    x0 = np.full(prob.x.shape, 0.5, np.float32)
    xg = dev(x0)
    plan.em_step(xg, dev(yy), None, niter=1)
    assert_close(host(xg), oracle.em_step(x0, yy, None, prob.mu, psf, prob.dy, ang), what="EM step")
    plan.check()
    plan.close()


def test_low_memory_plan_in_view_chunks(monkeypatch):
    """A low-memory plan of up to 37 taps runs the fused kernels in view chunks: A and A' over
    several passes, and its memory bound."""
    need_gpu()
    from paper_2301_09710_gb300.projector import plan_bytes
    prob = synthetic.random_problem(9, nx=48, nz=21, nview=14, px=11, pz=9, mu_scale=0.05)
    ang = oracle.default_angles(14)
    monkeypatch.setenv("SPECT_SLAB_MB", "2")
    plan = make_plan(prob, ang, "lowmem")
    info = plan.info()
    assert not info["fused"] and 1 <= info["view_chunk"] < 14
    assert info["device_bytes"] <= plan_bytes(48, 21, 14, 11, 9, low_memory=True)
    monkeypatch.delenv("SPECT_SLAB_MB")
    one = make_plan(prob, ang, "lowmem")
    assert one.info()["view_chunk"] == 14
    psf = oracle.psf_from_factors(prob.fx, prob.fz)
    v_o = oracle.forward(prob.x, prob.mu, psf, prob.dy, ang)
    assert_close(host(plan.forward(dev(prob.x))), v_o, what="A x")
    yy = np.random.default_rng(9).uniform(0.5, 1.5, plan.proj_shape).astype(np.float32)
    xb = host(plan.back(dev(yy)))
    assert_close(xb, oracle.back(yy, prob.mu, psf, prob.dy, ang), what="A' y")
    # each pass resumes the compensated view sums of the last one
    assert np.array_equal(xb, host(one.back(dev(yy)))), "A' depends on how the views are split"
    x0 = np.full(prob.x.shape, 0.5, np.float32)
    xg = dev(x0)
    plan.em_step(xg, dev(yy), None, niter=1)
    assert_close(host(xg), oracle.em_step(x0, yy, None, prob.mu, psf, prob.dy, ang), what="EM step")
    plan.check()
    plan.close()
    one.close()


@pytest.mark.parametrize("nx", [25, 24])  # A' begins with the row padding, or with the blur adjoint right behind the caller's kernel
@pytest.mark.parametrize("path", ["fused", "direct", "lowmem"])
def test_chained_launches_keep_their_order(path, nx):
    """Small kernels back to back, each reading what the one before wrote and overwriting what
    it read: a run of calls queued at once equals the same calls with a wait after each.  (Both
    runs chain the launches within a call; that each kernel waits for the one before it is read
    from the sources, test_chained_launches_cpu.py.)"""
    need_gpu()
    import torch
    prob = synthetic.random_problem(10, nx=nx, nz=7, nview=3, px=7, pz=5, mu_scale=0.05)
    plan = make_plan(prob, oracle.default_angles(3), path)
    yy = dev(np.random.default_rng(10).uniform(0.5, 1.5, plan.proj_shape).astype(np.float32))

    def run(wait):
        x, out = dev(np.full(prob.x.shape, 0.5, np.float32)), []
        for _ in range(8):
            for f in (lambda: plan.em_step(x, yy, None, niter=2), lambda: plan.forward(x), lambda: plan.back(yy * x.sum())):
                out.append(f().clone())
                if wait:
                    torch.cuda.synchronize()
        torch.cuda.synchronize()
        return [host(o) for o in out]

    for a, b in zip(run(False), run(True)):
        assert np.array_equal(a, b)
    plan.check()
    plan.close()


@pytest.mark.parametrize("nx,nz", [(8, 5), (9, 1), (65, 3), (130, 4)])
def test_attenuation_runs_of_depths(nx, nz):
    """The attenuation factors at the edges of their runs of eight depths and rounds of 64
    (one plane past a round, a last run of one plane), a strong mu: A and A' against the oracle."""
    need_gpu()
    prob = synthetic.random_problem(nx, nx=nx, nz=nz, nview=3, px=3, pz=3, mu_scale=0.2)
    ang = np.random.default_rng(nx).uniform(0, 2 * np.pi, 3)
    plan = make_plan(prob, ang, "fused")
    psf = oracle.psf_from_factors(prob.fx, prob.fz)
    assert_close(host(plan.forward(dev(prob.x))), oracle.forward(prob.x, prob.mu, psf, prob.dy, ang), what="A x")
    yy = np.random.default_rng(11).uniform(0, 1, plan.proj_shape).astype(np.float32)
    assert_close(host(plan.back(dev(yy))), oracle.back(yy, prob.mu, psf, prob.dy, ang), what="A' y")
    plan.check()
    plan.close()


@pytest.mark.parametrize("i,k", [(0, 4), (47, 4), (20, 20)])
def test_an_infinite_voxel_reaches_only_its_psf(i, k):
    """Replicate padding multiplies the edge columns by folded taps: an infinity there reaches the
    outputs that its PSF reaches, not the rest of a run of 16 (at angle 0 the bilinear rotation
    hands it on to the column before it with weight 0)."""
    need_gpu()
    import torch
    from paper_2301_09710_gb300 import SpectPlan
    nx, nz, p = 48, 40, 5
    taps = np.full((1, nx, p), 1.0 / p, np.float32)
    plan = SpectPlan(nx, nz, 1, fx=taps, fz=taps, angles=[0.0])
    x = np.ones((nz, nx, nx), np.float32)
    x[k, 20, i] = np.inf
    v = plan.forward(dev(x))
    finite = torch.isfinite(v)[0].cpu().numpy()
    plan.check()
    plan.close()
    ii, kk = np.meshgrid(np.arange(nx), np.arange(nz))
    reached = (ii >= i - 1 - p // 2) & (ii <= i + p // 2) & (abs(kk - k) <= p // 2)
    assert finite[~reached].all()
    assert not finite[(abs(ii - i) <= p // 2) & (abs(kk - k) <= p // 2)].any()


def test_a_depth_sum_that_overflows_is_infinite():
    """Partial sums of depth groups that are finite and add up to more than FP32 holds: the
    projection is +inf, as a plain sum gives it, not NaN."""
    need_gpu()
    import torch
    from paper_2301_09710_gb300 import SpectPlan
    nx, nz = 64, 8
    taps = np.full((1, nx, 3), 1.0 / 3, np.float32)
    plan = SpectPlan(nx, nz, 1, fx=taps, fz=taps, angles=[0.0])
    v = plan.forward(torch.full((nz, nx, nx), 1e37, device="cuda"))
    assert torch.isposinf(v).all()
    plan.check()
    plan.close()


def test_launch_shape_round_trips():
    """The two blurs may have different tile counts: what a plan reports, set on it again or on
    another plan, gives the same shape, also by the call that takes one count."""
    need_gpu()
    prob = synthetic.random_problem(12, nx=96, nz=9, nview=3, px=5, pz=5, mu_scale=0.05)
    ang = oracle.default_angles(3)
    plan, other = make_plan(prob, ang, "fused"), make_plan(prob, ang, "fused")
    plan.set_tuning(4, 8, 2, adj_tiles=6)
    t = plan.tuning
    assert t == {"fused_J": 4, "adj_J": 8, "tiles": 2, "adj_tiles": 6}
    plan.set_tuning(4, 8, 2)
    assert plan.tuning == t
    other.set_tuning(**t)
    assert other.tuning == t
    other.set_tuning(4, 8, 3)
    assert other.tuning == {"fused_J": 4, "adj_J": 8, "tiles": 3, "adj_tiles": 3}
    yy = dev(np.random.default_rng(12).uniform(0, 1, plan.proj_shape))
    assert np.array_equal(host(plan.back(yy)), host(other.back(yy)))
    for p in (plan, other):
        p.check()
        p.close()
