"""The launch shape a score call takes when none was set follows the size of the work: every
CTA size it can pick, single and batched, against the scores of one fixed shape."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import gpu_context, jitter_poses, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,vox,n", [(64, 600, 5000), (64, 600, 1500), (161, 3500, 3000), (150, 12000, 1200),
                                         (320, 12000, 300), (64, 600, 40)])
@pytest.mark.parametrize("lik", [dict(kind=0, half_window=1), dict(kind=1, half_window=2), dict(kind=0, half_window=3)])
def test_default_shape_scores(orc, width, vox, n, lik):
    """Shapes differ in the order of the FP32 sums only: 2e-6 of the log-likelihood."""
    from paper_2312_08715_gb300 import b3d
    lik = dict(lik, radius=0.004, p_outlier=0.02)
    wl = synth.tabletop_workload(6, n_objects=1, width=width, height=width * 3 // 4 + 1, f=0.9375 * width,
                                 vox_lo=int(0.7 * vox), vox_hi=int(1.4 * vox))
    obs = observed(orc, wl)
    poses = jitter_poses(np.random.default_rng(1), wl.hidden, n, trans=0.03, rot_deg=15)
    ctx, fixed = gpu_context(wl.scene, obs), gpu_context(wl.scene, obs)
    before = b3d.b3d_get_tuning(ctx.h)
    b3d.b3d_set_tuning(fixed.h, 64, 256, 0, 0)
    got, ref = ctx.score(wl.slot, poses, lik), fixed.score(wl.slot, poses, lik)
    P = torch.as_tensor(poses, device="cuda")
    outs = [torch.empty(k, device="cuda") for k in (n, max(1, n // 3))]
    owner = b3d.Context(0)
    b3d.b3d_score_multi(owner.h, [(c.h, wl.slot, o.numel(), P, o) for c, o in zip((ctx, fixed), outs)],
                        b3d.lik_params(**lik), ctx.stream)
    ctx.sync()
    ref = ref.cpu().numpy()
    np.testing.assert_allclose(got.cpu().numpy(), ref, rtol=2e-6)
    for o in outs:
        np.testing.assert_allclose(o.cpu().numpy(), ref[:o.numel()], rtol=2e-6)
    assert b3d.b3d_get_tuning(ctx.h) == before
    for c in (ctx, fixed, owner):
        c.close()
