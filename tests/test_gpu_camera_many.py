"""Camera renders of scenes with more objects than a CTA sets up at a time (16): every object is
drawn, and the depths and ids are the oracle's."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_obj", [16, 17, 35])
def test_many_objects(orc, n_obj):
    """Ids equal except at flagged pixels (coverage within 1e-4 px of an edge or depths within 1e-5
    relative of each other), depth within 1e-5 relative where ids agree and the depth is well
    conditioned; the depth-only render gives the same depths."""
    from paper_2312_08715_gb300 import b3d
    rng = np.random.default_rng(2)
    cells = np.array(np.unravel_index(rng.permutation(125)[:60], (5, 5, 5))).T
    kinds = [(synth.voxel_mesh(cells, 0.02, origin=(-0.05, -0.05, -0.05)), True), (synth.box_mesh((0.1, 0.06, 0.08)), True),
             (synth.table_mesh(0.1), False)]
    meshes, closed = zip(*(kinds[k % 3] for k in range(n_obj)))
    world = np.stack([synth.rigid(synth.random_rotation(rng), [0.16 * (k % 6 - 2.5), 0.16 * (k // 6 - 2.5), 0.03 * (k % 4)])
                      for k in range(n_obj)]).astype(np.float32)
    H = np.stack([synth.rigid(synth.yaw(0.2 * k), [0.02 * k, -0.01, 1.3]) for k in range(3)]).astype(np.float32)
    cam = synth.Camera(93, 71, 80.0, 82.0, 46.3, 35.2, 0.01, 4.0)
    ctx = b3d.Context(0)
    ctx.set_scene(cam, [ctx.load_mesh(m, closed=c) for m, c in zip(meshes, closed)], world, np.zeros((71, 93), np.float32))
    d, t = ctx.render_camera(H)
    only, _ = ctx.render_camera(H, want_tid=False)
    ctx.sync()
    assert torch.equal(only, d)
    d, t = d.cpu().numpy(), t.cpu().numpy()
    first = np.concatenate([[0], np.cumsum([len(m.faces) for m in meshes])])
    seen = {int(np.searchsorted(first, i, side="right")) for i in np.unique(t) if i >= 0}
    assert len(seen) == n_obj
    for k in range(len(H)):
        poses = np.stack([H[k].astype(np.float64) @ P for P in world.astype(np.float64)])
        od, ot, of = orc.render(synth.Scene(cam, list(meshes), poses), edge_tol=1e-4, z_tol=1e-5, want_flags=True)
        mis = ot != t[k]
        assert not (mis & ((of & 1) == 0)).any()
        ok = ~mis & ((of & 4) == 0)
        assert (np.abs(d[k][ok] - od[ok]) <= 1e-5 * od[ok]).all()
    ctx.close()
