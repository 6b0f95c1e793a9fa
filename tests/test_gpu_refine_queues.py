"""The distance kernel's queues when they are full: a flat tip over a finely
tessellated plate meets hundreds of triangles at the same distance, so no bound
rules any out.  128 poses in a block then put more nodes on its stack than it
holds without going depth first (704), and more candidates in its queue (2048)
than it settles at once.  The distance is the gap, in every block form, and the
same bits in each."""
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


def _plate(n, side, thick):
    """n x n quads on top of a slab, two triangles for each of the other faces."""
    g = np.linspace(-side / 2, side / 2, n + 1)
    x, y = np.meshgrid(g, g, indexing="ij")
    V = np.stack([x.ravel(), y.ravel(), np.zeros(x.size)], axis=1)
    i, j = np.meshgrid(np.arange(n), np.arange(n), indexing="ij")
    a = (i * (n + 1) + j).ravel()
    b, c, d = a + n + 1, a + n + 2, a + 1
    T = np.concatenate([np.stack([a, b, c], axis=1), np.stack([a, c, d], axis=1)])
    s, k = side / 2, len(V)
    V = np.concatenate([V, [[-s, -s, 0], [s, -s, 0], [s, s, 0], [-s, s, 0], [-s, -s, -thick], [s, -s, -thick], [s, s, -thick], [-s, s, -thick]]])
    q = np.array([(0, 4, 5, 1), (1, 5, 6, 2), (2, 6, 7, 3), (3, 7, 4, 0), (4, 7, 6, 5)]) + k
    return V, np.concatenate([T, q[:, :3], q[:, [0, 2, 3]]]).astype(np.int32)


@pytest.mark.parametrize("gap", [0.05, -0.02])
@pytest.mark.parametrize("P", [128, 96])
def test_full_queues(ctx, gap, P):
    V, T = _plate(48, 8.0, 1.0)
    rng = np.random.default_rng(P)
    poses = np.tile([1.0, 0, 0, 0, 0, 0, 0], (P, 1))   # body upwards
    poses[:, 4:6] = rng.uniform(-2.4, 2.4, size=(P, 2))
    poses[:, 6] = gap
    h, N = 0.3, 64
    ob, sw = ctx.object_grid(V, T, h, N), ctx.sweep_grid(poses, 1.0, 4.0, h, N)
    lift = np.array([0.0, 0.003, -0.003, 0.01, -0.01])
    ref = None
    for B in (5, 170, 1700):   # 8, 32 and 128 poses a block
        obj = np.tile([1.0, 0, 0, 0, 0, 0, 0], (B, 1))
        obj[:, 6] = lift[np.arange(B) % 5]
        d, w, n = ctx.distances(ob, sw, obj)
        # FP32 coordinates of a few millimetres through about ten roundings
        assert np.all(np.abs(d - (gap - obj[:, 6:7])) < 5e-6)
        assert np.all(np.abs(w[..., 2] - obj[:, None, 6]) < 5e-6)
        if ref is None:
            ref = d[:5], w[:5], n[:5]
        for got, want in zip((d, w, n), ref):
            assert np.array_equal(got, np.tile(want, (B // 5,) + (1,) * (want.ndim - 1)))
