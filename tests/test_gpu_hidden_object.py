"""An object wholly behind the fixed ones changes no pixel, so every term of its box equals the
background's and cancels: the score is the background's, the same bits wherever the object is."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("half_window", [1, 2, 3])
def test_hidden_object_scores_the_background(orc, kind, half_window):
    """The observed pixels are chosen so that the background's terms nearly sum to 0: a residue of
    a part in 10^8 of one term shows in the score."""
    from paper_2312_08715_gb300 import b3d
    cam = synth.Camera(97, 71, 90.0, 90.0, 48.0, 35.0, 0.01, 4.0)
    rng = np.random.default_rng(4)
    cells = np.array(np.unravel_index(rng.permutation(512)[:300], (8, 8, 8))).T
    meshes = [synth.table_mesh(5.0), synth.voxel_mesh(cells, 0.08, origin=(-0.32, -0.32, -0.32))]
    poses = np.stack([synth.rigid(np.eye(3), [0, 0, 1.0]), synth.rigid(np.eye(3), [0, 0, 2.0])]).astype(np.float32)
    lik = dict(kind=kind, radius=0.004, p_outlier=0.02, half_window=half_window, miss_mode=0)
    sigma = np.where(rng.random((cam.height, cam.width)) < 0.5, 0.004, 0.05)
    full = (1.0 + sigma * rng.normal(size=sigma.shape)).astype(np.float32)
    ell = orc.pixel_loglik(cam, lik, np.ones(full.shape), None, full)[0]
    box = [(y, x) for y in range(28, 44) for x in range(40, 57)]
    up = [p for p in box if ell[p] > 0]
    down = [p for p in box if ell[p] < 0]
    chosen, total = [], 0.0
    while len(chosen) < 80 and up and down:
        chosen.append((up if total <= 0 else down).pop())
        total += ell[chosen[-1]]
    chosen += min(((p, q) for p in up for q in down), key=lambda pq: abs(total + ell[pq[0]] + ell[pq[1]]))
    obs = np.zeros_like(full)
    for p in chosen:
        obs[p] = full[p]
    P = np.stack([synth.rigid(synth.random_rotation(rng), [x, y, 2.0]) for x, y in
                  ((0, 0), (0.1, 0.05), (-0.1, 0.03), (0.04, -0.1), (0.0, 0.1), (-0.05, -0.05), (60.0, 0.0))]).astype(np.float32)
    ctx, owner = b3d.Context(0), b3d.Context(0)
    ctx.set_scene(cam, [ctx.load_mesh(meshes[0], closed=False), ctx.load_mesh(meshes[1], closed=True)], poses, obs)
    Pd, out = torch.as_tensor(P, device="cuda"), torch.empty(len(P), device="cuda")
    for tile, nt in ((96, 128), (64, 256), (16, 32)):
        b3d.b3d_set_tuning(ctx.h, tile, nt, 0, 0)
        ll = ctx.score(1, P, lik)
        b3d.b3d_score_multi(owner.h, [(ctx.h, 1, len(P), Pd, out)], b3d.lik_params(**lik), ctx.stream)
        ctx.sync()
        # the last pose is off the image: its score is the background's sum
        assert (ll == ll[-1]).all() and torch.equal(out, ll), (tile, nt, ll - ll[-1])
    for c in (ctx, owner):
        c.close()
