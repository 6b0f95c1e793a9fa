"""The object grid's cells (Eq. (1)-(4)) against the oracle where the kernel's
sizes change: a voxel as large as a cell, cells of several voxel rounds, sides
that are no power of two, thin and degenerate triangles (whose FP32 distance is
not usable), a touchable sub-mesh; and the spectrum through a field."""
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


def _mesh(scale, n_theta, seed, spikes):
    obj = synth.star_mesh(4, 0.05, n_theta, 2 * n_theta, seed)
    V, T = obj.verts * scale, obj.tris
    if spikes:
        # every tenth triangle split at a point 1e-9 to 1e-3 of an edge away from a vertex: slivers
        rng = np.random.default_rng(seed)
        V, T = list(V), [tuple(t) for t in T]
        for i in range(0, len(T), 10):
            a, b, c = T[i]
            s = 10.0 ** rng.uniform(-9, -3)
            V.append(V[a] * (1 - s) + V[b] * s)
            m = len(V) - 1
            T[i] = (a, m, c)
            T.append((m, b, c))
            T.append((a, b, m))   # a triangle without area closes the gap
        V, T = np.array(V), np.array(T, dtype=np.int32)
    return V, T


@pytest.mark.parametrize("N, h, scale, n_theta, spikes, touchable", [
    (32, 0.6, 1.0, 16, False, False),     # h > cut: one voxel per cell
    (32, 0.5, 1.0, 24, True, True),
    (64, 0.1, 0.35, 16, False, True),     # 125 voxels per cell: two rounds of 64
    (64, 0.06, 0.15, 12, True, False),    # 500 voxels per cell
    (96, 0.17, 1.0, 40, True, True),
    (128, 0.15, 1.0, 64, False, False)])
def test_object_cells_match_the_oracle(ctx, N, h, scale, n_theta, spikes, touchable):
    V, T = _mesh(scale, n_theta, 5, spikes)
    touch = (np.arange(len(T)) % 3 != 0).astype(np.uint8) if touchable else None
    ob = ctx.object_grid(V, T, h, N, touchable=touch)
    G, o = ob.export_grid()
    Go, oo, _, fits = O.object_grid(V, T, h, N, touch=touch)
    assert fits and np.array_equal(o, oo)
    # the same FP64 expressions in the same order, rounded to FP32 once
    assert np.array_equal(G, Go.astype(np.float32))


@pytest.mark.parametrize("N", [32, 64, 96, 128])
def test_spectrum_through_a_field(ctx, N):
    V, T = _mesh(1.0, 24, 7, False)
    h = 16.0 / N
    ob = ctx.object_grid(V, T, h, N)
    q = np.array([1.0, 0.0, 0.0, 0.0])
    poses = np.concatenate([q, [0.0, 0.0, 0.0]])[None]
    sw = ctx.sweep_grid(poses, 0.8, 4.0, h, N)
    C = ctx.search_scores(ob, sw, q)
    M = 2 * N
    G, _ = ob.export_grid()
    S, _ = sw.voxelise(q)
    want = np.fft.irfftn(np.conj(np.fft.rfftn(G.astype(np.float64), s=(M, M, M))) *
                         np.fft.rfftn(S[0].astype(np.float64), s=(M, M, M)), s=(M, M, M))
    # FP32 transforms of length M per axis: a few units of the last place of the largest value
    assert np.max(np.abs(C - want)) <= 2e-6 * np.max(np.abs(want))
