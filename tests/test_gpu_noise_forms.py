"""The noise-grid scorer's forms (inlier counts per radius with two or four radii compiled in,
and the general form) against the single-setting score kernel, setting by setting."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import gpu_context, jitter_poses, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

RADII = [0.003, 0.009, 0.0045, 0.02]  # not sorted
WIDE = [0.003, 0.7]                   # half a metre or more: the general form
POUT = [0.01, 0.2, 0.05, 0.5]


@pytest.mark.parametrize("kind,radii,np_,w,miss_mode", [
    (0, RADII[:1], 1, 0, 0), (0, RADII[:2], 3, 1, 1), (0, RADII[:3], 4, 2, 0), (0, RADII, 4, 1, 0), (0, RADII, 2, 2, 1),
    (0, RADII, 1, 0, 1), (0, WIDE, 2, 1, 0), (0, WIDE, 2, 1, 1), (1, RADII[:3], 2, 1, 0), (1, RADII, 4, 2, 1)])
def test_every_setting_equals_the_single_setting_score(orc, kind, radii, np_, w, miss_mode):
    """The two kernels form every term from the same expressions and differ in the order of
    the FP32 sums: 2e-6 of the log-likelihood (as the single-setting test). The object is wider
    than a CTA of the noise kernel is of threads, and the image of odd size; tile_w 256 gives it
    a tile wider than the CTA."""
    from paper_2312_08715_gb300 import b3d
    wl = synth.tabletop_workload(3, n_objects=2, width=203, height=151, f=420.0, vox_lo=3000, vox_hi=8000)
    ctx = gpu_context(wl.scene, observed(orc, wl))
    poses = jitter_poses(np.random.default_rng(2), wl.hidden, 24, trans=0.03, rot_deg=20)
    pout = POUT[:np_]
    b3d.b3d_set_tuning(ctx.h, 256, 256, 0, 0)
    ll, marg = ctx.score_noise(wl.slot, poses, b3d.noise_grid(kind, radii, pout, w, miss_mode=miss_mode))
    for i, r in enumerate(radii):
        for j, p in enumerate(pout):
            one = ctx.score(wl.slot, poses, dict(kind=kind, radius=r, p_outlier=p, half_window=w, miss_mode=miss_mode))
            ctx.sync()
            np.testing.assert_allclose(ll[:, i * np_ + j].cpu().numpy(), one.cpu().numpy(), rtol=2e-6)
    ref = np.logaddexp.reduce(ll.cpu().numpy().astype(np.float64), axis=1)
    np.testing.assert_allclose(marg.cpu().numpy(), ref, rtol=1e-6)
    ctx.close()
