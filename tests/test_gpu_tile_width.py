"""A tile may be as wide as the tuning says where the scorer strides over its pixels (half windows
0 and from 3 on); only the column scorers (1 and 2) need a thread for each column."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half_window,tiles", [(0, 1), (1, 2), (2, 2), (3, 1)])
def test_rectangles_are_set_up_once_per_tile(half_window, tiles):
    """A bar of 160 x 1 x 1 cells, 150 pixels wide: one tile of 256 pixels, two of 128, which is
    what the counting build's CTA has threads."""
    from paper_2312_08715_gb300 import b3d
    cam = synth.Camera(200, 80, 300.0, 300.0, 100.0, 40.0, 0.01, 5.0)
    cells = np.argwhere(np.ones((160, 1, 1), bool))
    ctx = b3d.Context(0)
    ctx.set_scene(cam, [ctx.load_mesh(synth.voxel_mesh(cells, 0.002, origin=(-0.16, -0.001, -0.001)), closed=True)],
                  synth.rigid(np.eye(3), [0, 0, 0.64]).astype(np.float32)[None], np.full((80, 200), 0.64, np.float32))
    b3d.b3d_set_instrumentation(ctx.h, 2)
    P = torch.as_tensor(np.repeat(synth.rigid(np.eye(3), [0, 0, 0.64]).astype(np.float32)[None], 64, 0), device="cuda")
    lik = dict(kind=0, radius=0.004, p_outlier=0.02, half_window=half_window)
    rects = []
    for tile in (256, 128):
        b3d.b3d_set_tuning(ctx.h, tile, 128, 0, 0)
        ctx.score(0, P, lik)
        ctx.sync()
        rects.append(int(b3d.b3d_work_counters(ctx.h)[2]))
    assert rects[1] == 2 * rects[0] // tiles, rects
    ctx.close()
