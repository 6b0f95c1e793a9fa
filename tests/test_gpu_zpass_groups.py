"""The z pass's rotations per block and the launch size change no bit of a peak:
groups that divide a launch and that leave a remainder, launches of one rotation
and of a few, plain and label-aware, two objects in one pass."""
import numpy as np
import pytest

from paper_2605_21398_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_21398_gb300 import build, dock
    build.build()
    c = dock.Context(0)
    yield c
    c.close()


@pytest.mark.parametrize("labels", [False, True])
@pytest.mark.parametrize("N", [32, 64, 96, 128])
def test_groups_and_batches_change_nothing(ctx, workload, N, labels):
    w = workload("tiny32", N=N, h=16.0 / N, poses=90)
    contact = (np.arange(len(w.poses_world)) % 3 > 0).astype(np.uint8)
    ob = ctx.object_grid(w.obj.verts, w.obj.tris, w.h, N)
    sw = ctx.sweep_grid(w.poses_world, w.radius, w.length, w.h, N, contact=contact)
    sw.set_label_aware(labels)
    q = synth.random_unit_quats(23, 4)
    default = ctx.get_tuning(N)
    ref = None
    try:
        for batch, group in ((23, 0), (23, 1), (23, 5), (23, 23), (7, 3), (1, 1)):
            ctx.set_tuning(N=N, batch=batch, group=group)
            _, p = ctx.search_so3(ob, sw, len(q), 1, sampler=3, quats=q, want_peaks=True)
            if ref is None:
                ref = p
            assert np.array_equal(p["score"], ref["score"]) and np.array_equal(p["idx"], ref["idx"]), (batch, group)
    finally:
        ctx.set_tuning(**default)
