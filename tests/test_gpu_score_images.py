"""Scoring of materialised images under the 3x3 inlier ball: images that differ from the
reference background at chosen places of their border (an image differing in its first and
last rows and both outer columns is scored whole, without a pass to find its box), over image
sizes with and without vector access."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import gpu_context, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(97, 61), (64, 48), (3, 2), (1, 5), (4, 1)])
@pytest.mark.parametrize("miss_mode", [0, 1])
def test_border_differences(orc, width, height, miss_mode):
    """Within 1e-4 of the summed |l_i| of the oracle's per-pixel terms (the FP32 tolerance of
    the log-likelihood tests; a borderline pair moves one term by a few nats at most)."""
    wl = synth.tabletop_workload(4, n_objects=1, width=width, height=height, f=0.9375 * width, vox_lo=500, vox_hi=900)
    sc, cam = wl.scene, wl.scene.camera
    obs = observed(orc, wl)
    ctx = gpu_context(sc, obs)
    base, tid = ctx.render(wl.slot, sc.poses[wl.slot][None])
    ctx.sync()
    base, tid = base[0].cpu().numpy(), tid[0].cpu().numpy()
    H, W = base.shape
    rng = np.random.default_rng(5)
    spots = [[], [(0, W // 2)], [(0, 0)], [(H - 1, W - 1)], [(0, 0), (H - 1, W - 1)], [(0, W - 1), (H - 1, 0)],
             [(0, W // 2), (H - 1, W // 3)], [(H // 2, 0), (H // 2, W - 1)], [(H // 2, W // 2)]]
    imgs = []
    for s in spots:
        im = base.copy()
        for y, x in s:
            im[y, x] += np.float32(0.05)
        imgs.append(im)
    imgs.append((base + rng.normal(0, 0.003, size=base.shape)).astype(np.float32))
    imgs = np.stack(imgs)
    ids = np.repeat(tid[None], len(imgs), 0)
    ids[-1][rng.random((H, W)) < 0.3] = -1
    lk = dict(kind=0, radius=0.005, p_outlier=0.01, half_window=1, miss_mode=miss_mode)
    ref, scale = [], []
    for im, i in zip(imgs, ids):
        ell = orc.pixel_loglik(cam, lk, im.astype(np.float64), i if miss_mode else None, obs)[0]
        ref.append(ell.sum())
        scale.append(np.abs(ell).sum())
    ref, tol = np.array(ref), 1e-4 * np.array(scale)
    for slot in (-1, wl.slot):
        got = ctx.score_depth(torch.as_tensor(imgs, device="cuda"), lk, torch.as_tensor(ids, device="cuda"), slot=slot)
        ctx.sync()
        assert (np.abs(got.cpu().numpy().astype(np.float64) - ref) <= tol).all(), slot
    ctx.close()
