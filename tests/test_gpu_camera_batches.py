"""Camera depth renders whose z-buffer takes a CTA of 32 warps hand out an object's triangles 8
or 32 at a time by their size on the screen: the depths are the tiled renderer's bits and the
oracle's, for objects on either side of that line in one scene, near, far and out of view."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("width,height", [(131, 127), (181, 173), (223, 201)])
def test_depths_match_tiled_renderer_and_oracle(orc, width, height):
    """Depth within 1e-5 relative of the oracle's where no pixel is flagged (coverage within 1e-4
    px of an edge or depths within 1e-5 relative of each other)."""
    from paper_2312_08715_gb300 import b3d
    rng = np.random.default_rng(6)
    n = 20  # a table of 20 x 20 squares
    g = np.linspace(-0.5, 0.5, n + 1)
    verts = np.stack([a.ravel() for a in np.meshgrid(g, g, [0.0], indexing="ij")], 1).astype(np.float32)
    i, j = (a.ravel() for a in np.meshgrid(np.arange(n), np.arange(n), indexing="ij"))
    q = i * (n + 1) + j
    faces = np.concatenate([np.stack([q, q + n + 1, q + n + 2], 1), np.stack([q, q + n + 2, q + 1], 1)]).astype(np.int32)
    cells = np.array(np.unravel_index(rng.permutation(512)[:230], (8, 8, 8))).T
    meshes = [synth.Mesh(verts, faces), synth.voxel_mesh(cells, 0.01, origin=(-0.04, -0.04, -0.04)), synth.box_mesh((0.2, 0.15, 0.1))]
    world = np.stack([synth.rigid(np.eye(3), [0, 0, 0.1]), synth.rigid(synth.yaw(0.4), [0.1, 0.05, 0.0]),
                      synth.rigid(synth.yaw(-0.7), [-0.2, 0.1, 0.0])]).astype(np.float32)
    cams = [synth.rigid(np.eye(3), [0.0, 0.0, z]) for z in (0.3, 0.6, 1.2, 3.0)]
    cams += [synth.rigid(synth.random_rotation(rng), [0.1 * k, 0.0, 0.9]) for k in range(4)]
    cams.append(synth.rigid(np.eye(3), [9.0, 0.0, 1.0]))
    H = np.stack(cams).astype(np.float32)
    cam = synth.Camera(width, height, 0.9 * width, 0.9 * width, width / 2 - 0.3, height / 2 + 0.2, 0.01, 4.0)
    ctx = b3d.Context(0)
    ids = [ctx.load_mesh(m, closed=c) for m, c in zip(meshes, (False, True, True))]
    ctx.set_scene(cam, ids, world, np.zeros((height, width), np.float32))
    d, _ = ctx.render_camera(H, want_tid=False)
    dt, _ = ctx.render_camera(H)
    ctx.sync()
    assert torch.equal(d, dt)
    d = d.cpu().numpy()
    for k in range(len(H)):
        poses = np.stack([H[k].astype(np.float64) @ P for P in world.astype(np.float64)])
        od, _, of = orc.render(synth.Scene(cam, meshes, poses), edge_tol=1e-4, z_tol=1e-5, want_flags=True)
        ok = of == 0
        assert ok.mean() > 0.9 and (np.abs(d[k][ok] - od[ok]) <= 1e-5 * od[ok]).all(), k
    ctx.close()
