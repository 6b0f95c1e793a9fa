"""The object grid (Eq. (1)-(4)) of meshes with long thin triangles, bit for bit
the oracle's: finely tessellated capped cylinders (every side quad two needles,
with the sharp corner at each of the three vertices in turn) along the axes and
turned, and needles of all angles and lengths strewn over the lattice."""
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


def _cylinder(n, radius, height, R, corner):
    a = 2 * np.pi * np.arange(n) / n
    low = np.stack([radius * np.cos(a), radius * np.sin(a), np.full(n, -height / 2)], axis=1)
    V = np.concatenate([low, low + [0, 0, height], [[0, 0, -height / 2], [0, 0, height / 2]]])
    i = np.arange(n)
    j = (i + 1) % n
    T = np.concatenate([np.stack(t, axis=1) for t in
                        ((i, j, n + j), (i, n + j, n + i), (np.full(n, 2 * n), j, i), (np.full(n, 2 * n + 1), n + i, n + j))])
    return V @ R.T, np.ascontiguousarray(np.roll(T, corner, axis=1), dtype=np.int32)


def _same_grid(ctx, V, T, h, N):
    ob = ctx.object_grid(V, T, h, N)
    G, o = ob.export_grid()
    Go, oo, _, fits = O.object_grid(V, T, h, N)
    assert fits and np.array_equal(o, oo)
    assert np.array_equal(G, Go.astype(np.float32)), np.argwhere(G != Go.astype(np.float32))[:5]


@pytest.mark.parametrize("corner", [0, 1, 2])
@pytest.mark.parametrize("sides, turned, N", [(360, False, 128), (720, False, 128), (1440, False, 128),
                                              (360, True, 64), (720, True, 64), (1440, True, 64)])
def test_finely_tessellated_cylinder(ctx, sides, turned, N, corner):
    R = synth.quat_to_mat(synth.random_quat(np.random.default_rng(sides))) if turned else np.eye(3)
    _same_grid(ctx, *_cylinder(sides, 3.0, 12.0, R, corner), 19.2 / N, N)


@pytest.mark.parametrize("corner", [0, 1, 2])
@pytest.mark.parametrize("edge", [0.5, 2.0, 8.0])
def test_strewn_needles(ctx, edge, corner):
    rng = np.random.default_rng([int(10 * edge), corner])
    n = 300
    s = 10.0 ** rng.uniform(-4, -1, size=(n, 1))
    d = rng.normal(size=(n, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    e = np.cross(d, rng.normal(size=(n, 3)))
    e /= np.linalg.norm(e, axis=1, keepdims=True)
    apex = rng.uniform(-4, 4, size=(n, 3)) - 0.5 * edge * d
    tri = np.stack([apex, apex + edge * d, apex + edge * rng.uniform(0.3, 1, size=(n, 1)) * (d * np.cos(s) + e * np.sin(s))], axis=1)
    V = np.concatenate([np.roll(tri, corner, axis=1).reshape(-1, 3), [[-8.2] * 3, [8.2] * 3, [8.2, 8.2, 8.1]]])
    T = np.arange(len(V), dtype=np.int32).reshape(-1, 3)
    _same_grid(ctx, V, T, 0.3, 64)
