"""Voxels at the boundary of a probe: the radius (or length) is set so that one
lattice point lies just inside or just outside the cylinder's side (or far cap),
by 1e-12 to 1e-5 of it, for probes along each axis, skewed, and nearly along the
rows.  The bits equal the oracle's."""
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


def _axis_pose(axis, tip):
    axis = np.asarray(axis, dtype=np.float64)
    axis = axis / np.linalg.norm(axis)
    e1, e2, a = synth._frame_from_axis(axis)
    return np.concatenate([synth.mat_to_quat(np.stack([e1, e2, a], axis=1)), tip])


@pytest.mark.parametrize("N", [32, 64, 96, 128])
@pytest.mark.parametrize("axis", [(0, 0, 1), (0, 1, 0), (1, 0, 0), (1, 2, 3), (1, 0.02, -0.03), (1, 0.2, 0.1)])
def test_tangent_voxels(ctx, N, axis):
    h, r0, L0 = 16.0 / N, 0.8, 9.0
    rng = np.random.default_rng(N)
    for trial in range(6):
        pose = _axis_pose(axis, rng.uniform(-1, 1, size=3))
        poses = np.stack([pose] + [pose + np.r_[0, 0, 0, 0, rng.normal(size=3) * 0.3] for _ in range(rng.integers(0, 3))])
        q = np.array([1.0, 0, 0, 0]) if trial == 0 else synth.random_quat(rng)
        o = O.sweep_origin(poses, q, h, N)
        R, Rp = O.quat_to_mat(q), O.quat_to_mat(pose[:4])
        k = np.arange(N)
        z, y, x = np.meshgrid(k, k, k, indexing="ij")
        p = np.stack([x, y, z], axis=-1) * h + o
        l = (p @ R.T - pose[4:]) @ Rp
        rad = np.hypot(l[..., 0], l[..., 1])
        eps = 10.0 ** rng.uniform(-12, -5) * rng.choice([-1.0, 1.0])
        if trial % 2 == 0:
            d = np.abs(rad - r0) + 10.0 * ((l[..., 2] < 0.2 * L0) | (l[..., 2] > 0.8 * L0))
            r, L = rad.flat[np.argmin(d)] * (1 + eps), L0
        else:
            d = np.abs(l[..., 2] - L0) + 10.0 * (rad > 0.7 * r0)
            r, L = r0, l[..., 2].flat[np.argmin(d)] * (1 + eps)
        sw = ctx.sweep_grid(poses, r, L, h, N)
        S, _ = O.sweep_grid(poses, q, h, N, r, L)
        bits, _ = sw.voxelise(q)
        assert np.array_equal(bits[0], np.asarray(S).astype(np.uint8)), (trial, np.argwhere(bits[0] != S)[:5])
