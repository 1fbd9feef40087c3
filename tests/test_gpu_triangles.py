"""The triangle rasteriser of the renders with ids and of the camera renders shares triangles
out by their pixel count (a lane's own, the warp's, the CTA's queue) and skips the face classes
of a voxel mesh turned away from the camera: each branch, and the limits between them, against
the oracle."""
import math

import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _sheets(n):
    """n parallel 1 m squares, 2 mm apart: every triangle covers hundreds of pixels, and more of
    them than the CTA's queue holds."""
    one = synth.table_mesh(1.0)
    verts = np.concatenate([one.verts + np.float32([0, 0, 0.002 * k]) for k in range(n)])
    faces = np.concatenate([one.faces + 4 * k for k in range(n)])
    return synth.Mesh(verts.astype(np.float32), faces.astype(np.int32))


def _case(name):
    """(mesh, closed, poses) seen by a 67x45 camera."""
    rng = np.random.default_rng(8)
    R = [synth.random_rotation(rng) for _ in range(6)]
    if name == "voxels":  # from under a pixel a triangle to a few hundred
        cells = np.array(np.unravel_index(rng.permutation(216)[:90], (6, 6, 6))).T
        mesh = synth.voxel_mesh(cells, 0.01, origin=(-0.03, -0.03, -0.03))
        return mesh, True, [synth.rigid(R[k], [0.0, 0.0, z]) for k, z in enumerate((0.09, 0.15, 0.3, 0.8, 2.0, 3.5))]
    if name == "edge-on":  # the camera within the margin of a lattice plane, on either side
        cells = np.argwhere(np.ones((4, 3, 5), bool))
        mesh = synth.voxel_mesh(cells, 0.01, origin=(0.0, 0.0, 0.0))
        return mesh, True, [synth.rigid(np.eye(3), [-0.02 + d, -0.01 + e, 0.2])
                            for d in (0.0, 3e-5, -3e-5, 3e-4) for e in (2e-5, -2e-4)]
    if name == "box":
        mesh = synth.box_mesh((0.2, 0.15, 0.1))
        return mesh, True, [synth.rigid(R[k], [0.02 * k, 0.0, 0.25 + 0.2 * k]) for k in range(6)]
    mesh = _sheets(60)
    return mesh, False, [synth.rigid(synth.yaw(0.3 * k), [0.1, 0.0, 0.5 + 0.3 * k]) for k in range(3)]


@pytest.mark.parametrize("name", ["voxels", "edge-on", "box", "sheets"])
def test_triangle_branches_match_oracle(orc, name):
    """Ids identical except at flagged pixels (coverage within 1e-4 px of an edge or depths
    within 1e-5 relative), depth within 1e-5 relative where ids agree and the depth is well
    conditioned; the same keys from the object renderer and the camera renderer."""
    from paper_2312_08715_gb300 import b3d
    mesh, closed, poses = _case(name)
    cam = synth.Camera(67, 45, 60.0, 62.0, 33.0, 22.0, 0.01, 4.0)
    P = np.stack(poses).astype(np.float32)
    ctx = b3d.Context(0)
    ctx.set_scene(cam, [ctx.load_mesh(mesh, closed=closed)], np.eye(4, dtype=np.float32)[None],
                  np.zeros((cam.height, cam.width), np.float32))
    d, t = ctx.render(0, P)
    dc, tc = ctx.render_camera(P)
    do, _ = ctx.render_camera(P, want_tid=False)
    ctx.sync()
    assert torch.equal(t, tc) and torch.equal(d, dc) and torch.equal(d, do)
    d, t = d.cpu().numpy(), t.cpu().numpy()
    seen = 0
    for k in range(len(P)):
        od, ot, of = orc.render(synth.Scene(cam, [mesh], P[k:k + 1]), edge_tol=1e-4, z_tol=1e-5, want_flags=True)
        mis = ot != t[k]
        assert not (mis & ((of & 1) == 0)).any(), f"pose {k}: unflagged id mismatches"
        ok = ~mis & ((of & 4) == 0)
        assert (np.abs(d[k][ok] - od[ok]) / od[ok]).max() <= 1e-5
        seen += int((ot >= 0).sum())
    assert seen > 0
    ctx.close()
