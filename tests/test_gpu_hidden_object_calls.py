"""An object wholly behind the fixed ones, in the calls besides the score (test_gpu_hidden_object):
every term and derivative of its box equals the background's and cancels, so each result is the
same bits wherever the object is."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CAM = synth.Camera(97, 71, 90.0, 90.0, 48.0, 35.0, 0.01, 4.0)


def _setup(orc, lik):
    """A table before a hidden voxel object, observed pixels whose background terms nearly sum to
    0 (a residue of a part in 10^8 of one term shows in the sum), and poses behind the table, the
    last one off the image."""
    from paper_2312_08715_gb300 import b3d
    rng = np.random.default_rng(4)
    cells = np.array(np.unravel_index(rng.permutation(512)[:300], (8, 8, 8))).T
    meshes = [synth.table_mesh(5.0), synth.voxel_mesh(cells, 0.08, origin=(-0.32, -0.32, -0.32))]
    poses = np.stack([synth.rigid(np.eye(3), [0, 0, 1.0]), synth.rigid(np.eye(3), [0, 0, 2.0])]).astype(np.float32)
    sigma = np.where(rng.random((CAM.height, CAM.width)) < 0.5, 0.004, 0.05)
    full = (1.0 + sigma * rng.normal(size=sigma.shape)).astype(np.float32)
    ell = orc.pixel_loglik(CAM, lik, np.ones(full.shape), None, full)[0]
    box = [(y, x) for y in range(28, 44) for x in range(40, 57)]
    up, down = [p for p in box if ell[p] > 0], [p for p in box if ell[p] < 0]
    chosen, total = [], 0.0
    while len(chosen) < 80 and up and down:
        chosen.append((up if total <= 0 else down).pop())
        total += ell[chosen[-1]]
    obs = np.zeros_like(full)
    for p in chosen:
        obs[p] = full[p]
    P = np.stack([synth.rigid(synth.random_rotation(rng), [x, y, 2.0]) for x, y in
                  ((0, 0), (0.1, 0.05), (-0.1, 0.03), (0.04, -0.1), (0.0, 0.1), (-0.05, -0.05), (60.0, 0.0))]).astype(np.float32)
    ctx = b3d.Context(0)
    ctx.set_scene(CAM, [ctx.load_mesh(meshes[0], closed=False), ctx.load_mesh(meshes[1], closed=True)], poses, obs)
    return ctx, torch.as_tensor(P, device="cuda")


def _same(t):
    assert (t == t[-1]).all(), t - t[-1]


@pytest.mark.parametrize("half_window", [1, 2, 3])
def test_gradient(orc, half_window):
    lik = dict(kind=1, radius=0.004, p_outlier=0.02, half_window=half_window, miss_mode=0)
    ctx, P = _setup(orc, lik)
    ll, dpose, dsigma, dpout = ctx.score_grad(1, P, lik)
    ctx.sync()
    for t in (ll, dsigma, dpout):
        _same(t)
    assert (dpose == 0).all()
    ctx.close()


@pytest.mark.parametrize("kind,radii", [(0, [0.004, 0.01]), (0, [0.004, 0.7]), (1, [0.004, 0.01])])
@pytest.mark.parametrize("half_window", [0, 1, 2])
def test_noise_grid(orc, kind, radii, half_window):
    from paper_2312_08715_gb300 import b3d
    lik = dict(kind=kind, radius=0.004, p_outlier=0.02, half_window=half_window, miss_mode=0)
    ctx, P = _setup(orc, lik)
    ll, marg = ctx.score_noise(1, P, b3d.noise_grid(kind, radii, [0.02, 0.1], half_window))
    ctx.sync()
    _same(ll)
    _same(marg)
    ctx.close()


@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("half_window", [1, 2, 3])
def test_images(orc, kind, half_window):
    """Against the full scene's background, which holds the hidden object behind the table: the
    images equal it, so each is scored by its difference from it, which has no pixel; and images
    whose corner pixels were changed where nothing is observed, whose box is the whole image."""
    lik = dict(kind=kind, radius=0.004, p_outlier=0.02, half_window=half_window, miss_mode=0)
    ctx, P = _setup(orc, lik)
    depth, _ = ctx.render(1, P, want_tid=False)
    for slot in (1, -1):
        plain = ctx.score_depth(depth, lik, slot=slot)
        marked = depth.clone()
        marked[:-1, 0, 0] += 0.5
        marked[:-1, -1, -1] += 0.5
        got = ctx.score_depth(marked, lik, slot=slot)
        ctx.sync()
        _same(plain)
        _same(got)
    ctx.close()
