"""The launch shape that an untuned call picks follows the depth its grid is searched at, not the
scene's pose where the two differ, and stays the general one where no depth is known. The work
counters show the tile width: a rectangle is set up once for every tile its hypothesis has."""
import math

import numpy as np
import pytest

from paper_2312_08715_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _context(pose, fill=1.0):
    """A cube of 10^3 cells, a fraction of them filled, alone before a 160x120 camera."""
    from paper_2312_08715_gb300 import b3d
    cells = np.argwhere(np.random.default_rng(3).permutation(1000).reshape(10, 10, 10) < 1000 * fill)
    cam = synth.Camera(160, 120, 300.0, 300.0, 80.0, 60.0, 0.01, 5.0)
    ctx = b3d.Context(0)
    ctx.set_scene(cam, [ctx.load_mesh(synth.voxel_mesh(cells, 0.005, origin=(-0.025, -0.025, -0.025)), closed=True)],
                  np.asarray(pose, np.float32)[None], np.full((120, 160), 0.4, np.float32))
    b3d.b3d_set_instrumentation(ctx.h, 2)
    return ctx


LIK = dict(kind=0, radius=0.004, p_outlier=0.02, half_window=1)
STAGES = [synth.StageSpec(5, 0.002, 1, 30, math.radians(5))]  # 3,750 hypotheses
NEAR, FAR = synth.rigid(np.eye(3), [0, 0, 0.25]), synth.rigid(np.eye(3), [0, 0, 4.0])


def _searched(ctx):
    """Work counters of an enumeration around NEAR."""
    from paper_2312_08715_gb300 import b3d
    ctx.enumerate_c2f(0, NEAR.astype(np.float32), STAGES, LIK, 4, 1, np.eye(3))
    ctx.sync()
    return b3d.b3d_work_counters(ctx.h)


def _listed(ctx):
    from paper_2312_08715_gb300 import b3d
    P = torch.as_tensor(np.repeat(NEAR.astype(np.float32)[None], 3750, 0), device="cuda")
    ctx.score(0, P, LIK)
    ctx.sync()
    return b3d.b3d_work_counters(ctx.h)


def test_search_near_a_far_scene_pose():
    near, far = _context(NEAR), _context(FAR)
    np.testing.assert_array_equal(_searched(far), _searched(near))
    for c in (near, far):
        c.close()


@pytest.mark.parametrize("how", ["device pose", "placeholder", "behind"])
def test_unknown_depth_keeps_the_general_shape(how):
    from paper_2312_08715_gb300 import b3d
    start = {"device pose": FAR, "placeholder": np.eye(4), "behind": synth.rigid(np.eye(3), [0, 0, -4.0])}[how]
    ctx, general = _context(start), _context(start)
    b3d.b3d_set_tuning(general.h, 64, 256, 0, 0)
    for c in (ctx, general):
        if how == "device pose":
            b3d.b3d_set_object_pose_dev(c.h, 0, torch.as_tensor(NEAR.astype(np.float32), device="cuda"), c.stream)
    np.testing.assert_array_equal(_listed(ctx), _listed(general))
    for c in (ctx, general):
        c.close()


def test_time_near_a_far_scene_pose():
    """Untuned, the search is no more than 10% slower than under the general shape."""
    from paper_2312_08715_gb300 import b3d
    ms = []
    for tuned in (False, True):
        ctx = _context(FAR, fill=0.6)
        if tuned:
            b3d.b3d_set_tuning(ctx.h, 64, 256, 0, 0)
        b3d.b3d_set_instrumentation(ctx.h, 1)
        best = float("inf")
        for _ in range(8):
            b3d.b3d_kernel_time(ctx.h, 0)
            ctx.enumerate_c2f(0, NEAR.astype(np.float32), STAGES, LIK, 4, 1, np.eye(3))
            ctx.sync()
            best = min(best, b3d.b3d_kernel_time(ctx.h, 0)[0])
        ms.append(best)
        ctx.close()
    print(ms)
    assert ms[0] <= 1.10 * ms[1], ms
