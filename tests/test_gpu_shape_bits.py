"""A score with half window 1 or 2 is the same bits however its launch was shaped: every CTA size,
tile width and register build, alone, in a part of its list, in a batch with other scenes, with
and without a tuning. So are the draws of an enumeration, alone and in a batch."""
import math

import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import check_ll, gpu_context, jitter_poses, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SHAPES = [(64, 256, 0), (128, 256, 1), (96, 128, 0), (8, 128, 0), (16, 128, 1), (64, 64, 0), (256, 64, 1), (32, 32, 0), (9, 32, 1)]


def _scene(orc, width, vox, seed=6):
    wl = synth.tabletop_workload(seed, n_objects=2, width=width, height=width * 3 // 4 + 1, f=0.9375 * width,
                                 vox_lo=int(0.7 * vox), vox_hi=int(1.4 * vox))
    return wl, observed(orc, wl)


@pytest.mark.parametrize("width,vox", [(64, 600), (161, 3500), (301, 9000)])
@pytest.mark.parametrize("lik", [dict(kind=0, half_window=1), dict(kind=0, half_window=2), dict(kind=1, half_window=1),
                                 dict(kind=1, half_window=2)])
def test_scores_are_the_same_bits(orc, width, vox, lik):
    """And within the parity tolerance of the oracle."""
    from paper_2312_08715_gb300 import b3d
    lik = dict(lik, radius=0.004, p_outlier=0.02)
    n = 700
    wl, obs = _scene(orc, width, vox)
    small, small_obs = _scene(orc, 64, 500, seed=7)
    poses = jitter_poses(np.random.default_rng(1), wl.hidden, n, trans=0.03, rot_deg=15)
    P = torch.as_tensor(poses, device="cuda")
    ctx, other, owner = gpu_context(wl.scene, obs), gpu_context(small.scene, small_obs), b3d.Context(0)
    Ps = torch.as_tensor(jitter_poses(np.random.default_rng(2), small.hidden, 3000), device="cuda")
    ref = ctx.score(wl.slot, P, lik)
    ref_small = other.score(small.slot, Ps, lik)
    for at in (0, 3, n - 40):  # parts of the list, untuned
        assert torch.equal(ctx.score(wl.slot, P[at:at + 40].contiguous(), lik), ref[at:at + 40])
    outs = [torch.empty(n, device="cuda"), torch.empty(3000, device="cuda")]
    items = [(ctx.h, wl.slot, n, P, outs[0]), (other.h, small.slot, 3000, Ps, outs[1])]

    def batch():
        for o in outs:
            o.fill_(float("nan"))
        b3d.b3d_score_multi(owner.h, items, b3d.lik_params(**lik), owner.stream)
        assert torch.equal(outs[0], ref) and torch.equal(outs[1], ref_small)

    batch()
    for tile, nt, hi in SHAPES:
        for c in (ctx, owner):
            b3d.b3d_set_tuning(c.h, tile, nt, 0, hi, 3)
        assert torch.equal(ctx.score(wl.slot, P, lik), ref), (tile, nt, hi)
        batch()
    sel = np.arange(0, n, 35)
    check_ll(ref.cpu().numpy()[sel], orc.score(wl.scene, wl.slot, poses[sel], lik, obs), "sample", tight_frac=0.0)
    for c in (ctx, other, owner):
        c.close()


@pytest.mark.parametrize("scenes,n_rot", [([(64, 500), (320, 9000), (97, 1500)], 9), ([(64, 500), (72, 700)], 40)])
def test_untuned_enumerations_equal_batched_ones(orc, scenes, n_rot):
    """Particles, weights and densities of scenes whose single calls and whose batch take different
    launch shapes: uneven ones (256 threads for the batch), and small ones of many hypotheses (32)."""
    from paper_2312_08715_gb300 import b3d
    stages = [synth.StageSpec(7, 0.01, 1, n_rot, math.radians(6)), synth.StageSpec(9, 0.003, 1, 3, math.radians(2))]
    lik, M = dict(kind=0, radius=0.004, p_outlier=0.02, half_window=1), 24
    owner, ctxs, items, singles, outs = b3d.Context(0), [], [], [], []
    for k, (width, vox) in enumerate(scenes):
        wl, obs = _scene(orc, width, vox, seed=20 + k)
        ctx = gpu_context(wl.scene, obs)
        centre = wl.hidden.astype(np.float32)
        singles.append([x.clone() for x in ctx.enumerate_c2f(wl.slot, centre, stages, lik, M, 50 + k, wl.grid_frame)])
        out = (torch.empty((M, 4, 4), device="cuda"), torch.empty(M, device="cuda"), torch.empty(M, device="cuda"))
        items.append(b3d.c2f_item(ctx.h, wl.slot, centre, b3d.schedule(stages, M, 50 + k, wl.grid_frame), *out))
        ctxs.append(ctx)
        outs.append(out)
    b3d.b3d_enumerate_multi(owner.h, items, b3d.lik_params(**lik), owner.stream)
    owner.sync()
    for out, single in zip(outs, singles):
        assert all(torch.equal(a, b) for a, b in zip(out, single))
    for c in ctxs + [owner]:
        c.close()


@pytest.mark.parametrize("radius", [1e-14, 0.004])
def test_extreme_gaussian_terms(orc, radius):
    """A standard deviation whose normaliser overflows gives NaN scores as it did in plain floats,
    the same under every shape; an ordinary one none."""
    from paper_2312_08715_gb300 import b3d
    wl, obs = _scene(orc, 64, 600)
    ctx = gpu_context(wl.scene, obs)
    lik = dict(kind=1, half_window=1, radius=radius, p_outlier=0.02)
    P = torch.as_tensor(jitter_poses(np.random.default_rng(3), wl.hidden, 20), device="cuda")
    for tile, nt, hi in SHAPES[::2]:
        b3d.b3d_set_tuning(ctx.h, tile, nt, 0, hi)
        assert bool(torch.isnan(ctx.score(wl.slot, P, lik)).all()) == (radius < 1e-10)
    ctx.close()
