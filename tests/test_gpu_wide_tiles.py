"""Tiles requested wider than the CTA has threads: every column of a wide footprint is scored
(tile_w may be up to 256 with CTAs of 32 threads)."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import gpu_context, jitter_poses, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nt", [32, 64, 128, 256])
@pytest.mark.parametrize("half_window", [1, 2])
def test_wide_tile_scores_every_column(orc, nt, half_window):
    """The fused kernel and the image scorer under a 256-pixel tile against tiles of 32 pixels:
    the order of the FP32 sums differs (2e-6 of the log-likelihood)."""
    from paper_2312_08715_gb300 import b3d
    wl = synth.tabletop_workload(2, n_objects=1, width=300, height=200, f=700.0, vox_lo=6000, vox_hi=9000)
    lik = dict(wl.lik, half_window=half_window)
    ctx = gpu_context(wl.scene, observed(orc, wl))
    poses = jitter_poses(np.random.default_rng(3), wl.hidden, 12, trans=0.02, rot_deg=15)
    depth, _ = ctx.render(wl.slot, poses, want_tid=False)
    got = []
    for tile in (32, 256):
        b3d.b3d_set_tuning(ctx.h, tile, nt, 0, 0)
        got.append([x.cpu().numpy() for x in (ctx.score(wl.slot, poses, lik), ctx.score_depth(depth, lik, slot=wl.slot))])
        ctx.sync()
    for a, b in zip(*got):
        np.testing.assert_allclose(a, b, rtol=2e-6)
    ctx.close()
