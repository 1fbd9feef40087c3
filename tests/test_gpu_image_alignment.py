"""Materialised images of any size and at any 4-byte offset: the 16-byte accesses lie between an
image's own 16-byte boundaries, the pixels before and after them are accessed one by one."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import gpu_context, jitter_poses, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SIZES = [(97, 61), (64, 48), (66, 49), (3, 2), (1, 5), (3, 1), (1, 1)]
PAD = 8


def _scene(orc, width, height, n):
    wl = synth.tabletop_workload(4, n_objects=2, width=width, height=height, f=0.9375 * max(width, 16), vox_lo=500, vox_hi=900)
    obs = observed(orc, wl)
    return wl, gpu_context(wl.scene, obs), jitter_poses(np.random.default_rng(3), wl.scene.poses[wl.slot], n)


def _buffer(n, off, dtype):
    """(whole buffer, the view of n elements that starts `off` elements past a 16-byte boundary)"""
    b = torch.full((n + 2 * PAD,), 77, dtype=dtype, device="cuda")
    return b, b[PAD + off:PAD + off + n]


def _untouched(b, off, n):
    return bool((b[:PAD + off] == 77).all()) and bool((b[PAD + off + n:] == 77).all())


@pytest.mark.parametrize("width,height", SIZES)
def test_renders_with_ids(orc, width, height):
    """Ids and depths are the oracle's (ids except at flagged pixels, depths within 1e-5 relative
    where ids agree and the depth is well conditioned), the same bits at every offset, and nothing
    around the images is written."""
    from paper_2312_08715_gb300 import b3d
    wl, ctx, P = _scene(orc, width, height, 5)
    Pd = torch.as_tensor(P, device="cuda")
    n = len(P) * width * height
    first = None
    for od, ot in [(0, 0), (1, 1), (2, 2), (3, 3), (0, 1), (2, 3)]:
        (bd, d), (bt, t) = _buffer(n, od, torch.float32), _buffer(n, ot, torch.int32)
        b3d.b3d_render_batch(ctx.h, wl.slot, len(P), Pd, d, t, ctx.stream)
        ctx.sync()
        assert _untouched(bd, od, n) and _untouched(bt, ot, n)
        first = first or (d.clone(), t.clone())
        assert torch.equal(d, first[0]) and torch.equal(t, first[1]), (od, ot)
    d, t = (a.reshape(len(P), height, width).cpu().numpy() for a in first)
    for k in range(len(P)):
        poses = wl.scene.poses.copy()
        poses[wl.slot] = P[k]
        sc = synth.Scene(wl.scene.camera, wl.scene.meshes, poses)
        od, ot, of = orc.render(sc, edge_tol=1e-4, z_tol=1e-5, want_flags=True)
        mis = ot != t[k]
        assert not (mis & ((of & 1) == 0)).any(), f"pose {k}: unflagged id mismatches"
        ok = ~mis & ((of & 4) == 0)
        assert (np.abs(d[k][ok] - od[ok]) <= 1e-5 * od[ok]).all()
    ctx.close()


def test_few_and_many_large_images(orc):
    """Fewer than 100 images of more than 40,000 pixels are filled by a launch of their own."""
    wl, ctx, P = _scene(orc, 211, 197, 101)
    many = ctx.render(wl.slot, P)
    few = ctx.render(wl.slot, P[:99])
    ctx.sync()
    assert all(torch.equal(a[:99], b) for a, b in zip(many, few))
    ctx.close()


@pytest.mark.parametrize("width,height", SIZES)
def test_depth_renders_and_scores(orc, width, height):
    """The depth render is the same bits at every offset and writes nothing around the images;
    its scores, and those of images changed at their first and last pixels, are the same bits at
    every offset and within 1e-4 of the summed |l_i| of the oracle's per-pixel terms."""
    from paper_2312_08715_gb300 import b3d
    wl, ctx, P = _scene(orc, width, height, 5)
    Pd = torch.as_tensor(P, device="cuda")
    n = len(P) * width * height
    obs = observed(orc, wl)
    rng = np.random.default_rng(7)
    first = ids = None
    for off in range(4):
        bd, d = _buffer(n, off, torch.float32)
        b3d.b3d_render_batch(ctx.h, wl.slot, len(P), Pd, d, None, ctx.stream)
        ctx.sync()
        assert _untouched(bd, off, n)
        if first is None:
            first = d.clone()
            ids = torch.as_tensor(np.where(rng.random(n) < 0.2, -1, 3).astype(np.int32), device="cuda")
        assert torch.equal(d, first), off
    imgs = first.clone().reshape(len(P), -1)
    imgs[1:, 0] += 0.05
    imgs[2:, -1] -= 0.05
    for half_window in (1, 2):
        for miss_mode in (0, 1):
            lk = dict(kind=0, radius=0.005, p_outlier=0.01, half_window=half_window, miss_mode=miss_mode)
            got = []
            for od, ot in [(0, 0), (1, 1), (2, 2), (3, 3), (0, 3), (2, 1)]:
                (_, d), (_, t) = _buffer(n, od, torch.float32), _buffer(n, ot, torch.int32)
                d.copy_(imgs.reshape(-1))
                t.copy_(ids)
                shape = (len(P), height, width)
                got.append(ctx.score_depth(d.view(shape), lk, t.view(shape) if miss_mode else None, slot=wl.slot))
            ctx.sync()
            assert all(torch.equal(g, got[0]) for g in got)
            for k in range(len(P)):
                im = imgs[k].reshape(height, width).cpu().numpy().astype(np.float64)
                i = ids.reshape(len(P), height, width)[k].cpu().numpy() if miss_mode else None
                ell = orc.pixel_loglik(wl.scene.camera, lk, im, i, obs)[0]
                assert abs(float(got[0][k]) - ell.sum()) <= 1e-4 * np.abs(ell).sum()
    ctx.close()
