"""The distance kernel deals 8, 32 or 128 poses to a block, by the number of
poses in the launch: the same pose gets the same distance, witness and normal in
each form (bit for bit), the oracle's distance, and the edges of the forms (one
pose, a partly filled block, a trajectory that is no multiple of 32) work."""
import numpy as np
import pytest

import oracle as O
from paper_2605_21398_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_21398_gb300 import build, dock
    build.build()
    c = dock.Context(0)
    yield c
    c.close()


def _poses(w, n):
    rng = np.random.default_rng(3)
    base = [(w.gt_q, w.gt_t)]
    for _ in range(4):
        q = synth.quat_mul(synth.axis_angle_quat(np.radians(rng.normal(size=3))), w.gt_q)
        base.append((q / np.linalg.norm(q), w.gt_t + rng.normal(size=3) * 0.04))
    return [base[i % 5] for i in range(n)]


@pytest.mark.parametrize("P", [1, 31, 33, 129, 200])
def test_same_distances_in_every_block_form(ctx, workload, P):
    w = workload("tiny32")
    poses = w.poses_world[:P]
    ob = ctx.object_grid(w.obj.verts, w.obj.tris, w.h, w.N)
    sw = ctx.sweep_grid(poses, w.radius, w.length, w.h, w.N)
    padded = (P + 127) // 128 * 128
    ref = None
    # at most 20000, 200000 and more (padded) poses per launch: 8, 32, 128 per block
    for B in (5, 20000 // padded + 5, 200000 // padded + 5):
        B -= B % 5
        T = _poses(w, B)
        d, wit, nrm = ctx.distances(ob, sw, np.array([np.concatenate(p) for p in T]))
        if ref is None:
            ref = (d[:5].copy(), wit[:5].copy(), nrm[:5].copy())
            for b in range(5):
                do = O.distances(w.obj.verts, w.obj.tris, poses, O.quat_to_mat(T[b][0]), T[b][1], w.radius, w.length)[0]
                sel = do < O.TAU_OUT2
                # FP32 coordinates of up to 15 mm through about ten roundings
                assert np.all(np.abs(ref[0][b][sel] - do[sel]) < 2e-5)
        near = np.tile(ref[0] < O.TAU_OUT2, (B // 5, 1))   # beyond the cutoff any triangle passed over may be reported
        for got, want in zip((d, wit, nrm), ref):
            reps = np.tile(want, (B // 5,) + (1,) * (want.ndim - 1))
            assert np.array_equal(got[near], reps[near])


@pytest.mark.parametrize("K", [1, 5, 160])
def test_refined_candidates_do_not_depend_on_the_batch(ctx, workload, K):
    w = workload("tiny32")
    ob = ctx.object_grid(w.obj.verts, w.obj.tris, w.h, w.N)
    sw = ctx.sweep_grid(w.poses_world, w.radius, w.length, w.h, w.N)
    starts = _poses(w, 5)
    alone = [ctx.refine_se3(ob, sw, [dict(q=q, t=t)])[0] for q, t in starts]
    for i, o in enumerate(ctx.refine_se3(ob, sw, [dict(q=q, t=t) for q, t in _poses(w, K)])):
        for key in ("q", "t", "xi", "J"):
            assert np.array_equal(o[key], alone[i % 5][key])
