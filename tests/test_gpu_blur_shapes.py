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
