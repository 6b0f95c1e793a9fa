"""Distances of poses beyond the cutoff (Eq. (21)): 32 consecutive poses share one
walk of the tree, and a pose farther than tau_out2 from the mesh is given the
nearest of the triangles that the walk met and whose sphere passes its own test.
Poses within the cutoff get the same bits whether or not the walk is shared with
such a pose."""
import numpy as np
import pytest

import oracle as O
from paper_2605_21398_gb300 import synth

pytestmark = pytest.mark.gpu

I = np.array([[1.0, 0, 0, 0, 0, 0, 0]])


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_21398_gb300 import build, dock
    build.build()
    c = dock.Context(0)
    yield c
    c.close()


def _along_x(sign, tip):
    e1, e2, a = synth._frame_from_axis(np.array([sign, 0.0, 0.0]))
    return np.concatenate([synth.mat_to_quat(np.stack([e1, e2, a], axis=1)), tip])


@pytest.mark.parametrize("N", [32])
def test_the_nearest_triangle_of_a_shared_walk(ctx, N):
    # a leaf of three triangles; the sphere of the first (radius 3.0 about x = 3.95)
    # reaches past the leaf's (5.4 about x = -0.5)
    V = np.array([[4, -3, 0], [4, 3, 0], [3.9, 0, 0.5], [-5, 0, 0], [-4.8, 0.3, 0], [-4.8, 0, 0.3], [-4.6, 0, 0], [-4.6, 0.2, 0], [-4.6, 0, 0.2]])
    T = np.arange(9, dtype=np.int32).reshape(3, 3)
    ob = ctx.object_grid(V, T, 0.6, N)
    near, far = _along_x(-1.0, [-5.05, 0.0, 0.0]), _along_x(1.0, [5.6, 0.0, 0.0])
    poses = np.array([far] * 32 + [far] * 31 + [near])
    d, w, n = ctx.distances(ob, ctx.sweep_grid(poses, 0.8, 2.0, 0.6, N), I)
    assert np.all(np.isinf(d[0, :32]))   # no pose of this walk passes the leaf's test
    # FP32 coordinates of up to 6 mm through about ten roundings
    assert np.all(np.abs(d[0, 32:63] - 1.6) < 1e-5) and abs(d[0, 63] - 0.05) < 1e-5
    assert np.all(np.abs(w[0, 32:63, 0] - 4.0) < 1e-5) and np.all(np.abs(n[0, 32:63] - [-1, 0, 0]) < 1e-6)


def _tilts(w, n):
    rng = np.random.default_rng(5)
    out = []
    for _ in range(n):
        q = synth.quat_mul(synth.axis_angle_quat(np.radians(rng.normal(size=3))), w.gt_q)
        out.append(np.concatenate([q / np.linalg.norm(q), w.gt_t + rng.normal(size=3) * 0.04]))
    return np.array(out)


@pytest.mark.parametrize("B", [3, 200])
def test_sharing_a_walk_does_not_change_poses_within_the_cutoff(ctx, workload, B):
    w = workload("tiny32")
    poses, obj = w.poses_world, _tilts(w, B)
    ob = ctx.object_grid(w.obj.verts, w.obj.tris, w.h, w.N)
    d0, w0, n0 = ctx.distances(ob, ctx.sweep_grid(poses, w.radius, w.length, w.h, w.N), obj)
    # every eighth pose pulled back along its axis by 0.05 to 1.5 mm
    back = poses.copy()
    k = np.arange(0, len(back), 8)
    axis = np.array([O.quat_to_mat(p[:4])[:, 2] for p in back[k]])
    back[k, 4:] += axis * np.linspace(0.05, 1.5, len(k))[:, None]
    d1, w1, n1 = ctx.distances(ob, ctx.sweep_grid(back, w.radius, w.length, w.h, w.N), obj)
    kept = np.ones(len(poses), dtype=bool)
    kept[k] = False
    same = kept[None, :] & (d0 < O.TAU_OUT2)
    assert np.array_equal(d0[same], d1[same]) and np.array_equal(w0[same], w1[same]) and np.array_equal(n0[same], n1[same])
    for b in range(3):
        R, t = O.quat_to_mat(obj[b][:4]), obj[b][4:]
        do = O.distances(w.obj.verts, w.obj.tris, back, R, t, w.radius, w.length, eps=1e9)[0]
        in_ = do < O.TAU_OUT2
        assert np.all(np.abs(d1[b][in_] - do[in_]) < 2e-5)   # FP32 coordinates of up to 15 mm
        assert np.all(d1[b][~in_] >= do[~in_] - 2e-5)
        assert np.any(np.isfinite(d1[b][~in_]))
