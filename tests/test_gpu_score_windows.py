"""Scores of every window size, likelihood and miss mode against the oracle: footprints of
several tiles, at the image's border and beyond it, over fixed objects and over misses."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import check_ll, gpu_context, jitter_poses, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_objects", [1, 3])
@pytest.mark.parametrize("kind,half_window", [(0, 1), (0, 2), (0, 3), (1, 1), (1, 2), (1, 3)])
@pytest.mark.parametrize("miss_mode", [0, 1])
def test_scores_match_oracle(orc, n_objects, kind, half_window, miss_mode):
    """Each within 1e-4 of the summed |l_i| plus the oracle's bound for FP32 decisions; the depth
    images and their scores likewise, by shapes of 32 and 128 threads with tiles of 16 pixels."""
    from paper_2312_08715_gb300 import b3d
    wl = synth.tabletop_workload(9, n_objects=n_objects, width=73, height=58, f=90.0, vox_lo=500, vox_hi=1500)
    obs = observed(orc, wl)
    poses = jitter_poses(np.random.default_rng(2), wl.hidden, 14, trans=0.03, rot_deg=25)
    poses[9:12, 0, 3] += np.float32([0.25, -0.3, 0.28])  # over the border
    poses[12, 1, 3] += np.float32(2.0)  # off the image
    poses[13, :3, 3] = np.float32([0.0, 0.0, 0.4])  # large
    lik = dict(kind=kind, radius=0.004 if kind else 0.006, p_outlier=0.02, half_window=half_window, miss_mode=miss_mode)
    ref = orc.score(wl.scene, wl.slot, poses, lik, obs)
    ctx = gpu_context(wl.scene, obs)
    for tile, nt in ((64, 256), (16, 32), (16, 128)):
        b3d.b3d_set_tuning(ctx.h, tile, nt, 0, 0)
        ll = ctx.score(wl.slot, poses, lik)
        depth, tid = ctx.render(wl.slot, poses)
        image_ll = ctx.score_depth(depth, lik, tid, slot=wl.slot)
        ctx.sync()
        check_ll(ll.cpu().numpy(), ref, f"tile {tile}, {nt} threads", tight_frac=0.0)
        check_ll(image_ll.cpu().numpy(), ref, f"images, tile {tile}, {nt} threads", tight_frac=0.0)
    ctx.close()
