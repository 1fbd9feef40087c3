"""The batched autotuner on an owner that was never tuned times the shapes it names, so what it
keeps is as fast as the shape such an owner's launches choose for themselves."""
import numpy as np
import pytest

from paper_2312_08715_gb300 import synth
from _scenes import gpu_context, observed

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _score_ms(b3d, owner, items, lik):
    """Device time of the fastest of eight batched enumerations' score launches."""
    best = float("inf")
    b3d.b3d_set_instrumentation(owner.h, 1)
    for _ in range(8):
        b3d.b3d_kernel_time(owner.h, 0)
        b3d.b3d_enumerate_multi(owner.h, items, lik, owner.stream)
        owner.sync()
        best = min(best, b3d.b3d_kernel_time(owner.h, 0)[0])
    b3d.b3d_set_instrumentation(owner.h, 0)
    return best


def test_small_objects_keep_a_small_shape(orc):
    """Four scenes of one object of 500 cells at 64x48, 24,000 hypotheses each: CTAs of 32 threads
    take 1.40 ms, the 256 threads that a search among unset shapes had kept 2.04. The kept tuning's
    time may exceed the untuned call's by 10% (the candidates are timed once)."""
    from paper_2312_08715_gb300 import b3d
    stages = [synth.StageSpec(8, 0.004, 1, 47, 0.2)]
    ctxs, items, keep = [], [], []
    for k in range(4):
        wl = synth.single_object_workload(k)
        ctx = gpu_context(wl.scene, observed(orc, wl))
        out = (torch.empty((4, 4, 4), device="cuda"), torch.empty(4, device="cuda"), torch.empty(4, device="cuda"))
        items.append(b3d.c2f_item(ctx.h, 0, wl.hidden.astype(np.float32), b3d.schedule(stages, 4, 7 + k, np.eye(3)), *out))
        ctxs.append(ctx)
        keep.append(out)
    lik = b3d.lik_params(**wl.lik)
    untuned, owner = b3d.Context(0), b3d.Context(0)
    t_untuned = _score_ms(b3d, untuned, items, lik)
    best = b3d.b3d_autotune_multi(owner.h, items, lik, owner.stream)
    assert b3d.b3d_get_tuning(owner.h) == best
    t_kept = _score_ms(b3d, owner, items, lik)
    assert t_kept <= 1.10 * t_untuned, (best, t_kept, t_untuned)
    # the reported tuning is the one in use
    same = b3d.Context(0)
    b3d.b3d_set_tuning(same.h, **best)
    t_same = _score_ms(b3d, same, items, lik)
    assert abs(t_kept - t_same) <= 0.10 * t_same, (t_kept, t_same)
    for c in ctxs + [untuned, owner, same]:
        c.close()
