"""Renders with ids skip the face classes of a voxel mesh that are turned away from the camera;
where a plane is so nearly edge-on that the sign of its triangles' screen area is rounding, they
must not be skipped: the ids are those of the background raster, which tests every triangle."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _poses(rng, cam, half, z, n):
    """n poses before the middle of the image with the camera 1 to 4 times (0.1 mm + 0.01%) inside
    one face's plane."""
    d = np.array([(cam.width / 2 - cam.cx) / cam.fx, (cam.height / 2 - cam.cy) / cam.fy, 1.0])
    u = d / np.linalg.norm(d)
    out = np.zeros((n, 4, 4))
    for P in out:
        a, sign = rng.integers(3), rng.choice([-1, 1])
        dist = rng.uniform(*z) * np.linalg.norm(d)
        s = sign * (half - 1e-4 * (1 + dist) * rng.uniform(1.0, 4.0)) / dist
        v = rng.normal(size=3)
        v -= v.dot(u) * u
        axis = -s * u + np.sqrt(1 - s * s) * v / np.linalg.norm(v)
        w = np.cross(axis, u + 0.3 * rng.normal(size=3))
        w /= np.linalg.norm(w)
        cols = [None] * 3
        cols[a], cols[(a + 1) % 3], cols[(a + 2) % 3] = axis, w, np.cross(axis, w)
        R = np.stack(cols, 1)
        if np.linalg.det(R) < 0:
            R[:, (a + 2) % 3] *= -1
        P[:3, :3], P[:3, 3], P[3, 3] = R, u * dist, 1.0
    return out.astype(np.float32)


@pytest.mark.parametrize("f,cx,pitch,z,n", [(150.0, 32.0, 0.005, (0.5, 1.5), 3000), (1000.0, -4000.0, 0.002, (3, 8), 10000),
                                            (1000.0, -6000.0, 0.002, (3, 8), 10000), (1000.0, -4000.0, 0.001, (3, 8), 20000)])
def test_ids_equal_the_background_raster(f, cx, pitch, z, n):
    """A window of 64x64 pixels of a large image (the principal point far outside it), over a cube
    of 12^3 cells of about a pixel and less."""
    from paper_2312_08715_gb300 import b3d
    rng = np.random.default_rng(1)
    cam = synth.Camera(64, 64, f, f, cx, cx * 0.3, 0.01, 20.0)
    mesh = synth.voxel_mesh(np.argwhere(np.ones((12, 12, 12), bool)), pitch, origin=(-6 * pitch,) * 3)
    P = _poses(rng, cam, 6 * pitch, z, n)
    away = synth.rigid(np.eye(3), [0, 0, -5.0]).astype(np.float32)
    ctx = b3d.Context(0)
    ctx.set_scene(cam, [ctx.load_mesh(mesh, closed=True), ctx.load_mesh(synth.box_mesh((0.01, 0.01, 0.01)), closed=True)],
                  np.stack([P[0], away]), np.zeros((64, 64), np.float32))
    depth, ids = ctx.render(0, P)
    Pd, A = torch.as_tensor(P, device="cuda"), torch.as_tensor(away[None], device="cuda")
    differ = torch.zeros((), dtype=torch.int64, device="cuda")
    for k in range(n):
        b3d.b3d_set_object_pose_dev(ctx.h, 0, Pd[k], ctx.stream)
        bd, bt = ctx.render(1, A)
        differ += (bt[0] != ids[k]).sum() + (bd[0] != depth[k]).sum()
    assert int((ids >= 0).sum()) > 10 * n
    assert int(differ) == 0
    ctx.close()
