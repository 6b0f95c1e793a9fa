"""The bins of the object grid where one triangle meets many of their cells: a
mesh whose entries exceed 32 bits is refused before they are counted, and the
same shape with fewer triangles gives the oracle's grid."""
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


def _rod(n, half, width):
    """2 n triangles along the lattice's diagonal: every box spans the lattice."""
    a = 2 * np.pi * np.arange(n) / n
    d = np.ones(3) / np.sqrt(3)
    e1, e2, _ = synth._frame_from_axis(d)
    ring = width * (np.cos(a)[:, None] * e1 + np.sin(a)[:, None] * e2)
    V = np.concatenate([ring - half, ring + half])
    i = np.arange(n)
    j = (i + 1) % n
    T = np.concatenate([np.stack([i, j, n + j], axis=1), np.stack([i, n + j, n + i], axis=1)])
    return V, T.astype(np.int32)


def test_more_entries_than_32_bits_are_refused(ctx):
    from paper_2605_21398_gb300 import dock
    # one voxel per cell at h = 0.6; 1200 boxes of about 125^3 cells
    V, T = _rod(600, 37.0, 0.2)
    ctx.object_grid(*_rod(12, 35.0, 2.0), 0.6, 128).close()
    held = ctx.memory_stats()[0]
    with pytest.raises(dock.DockError) as e:
        ctx.object_grid(V, T, 0.6, 128)
    assert e.value.status == dock.E_TOO_LARGE and "cells" in str(e.value)
    assert ctx.memory_stats()[0] == held   # everything released


def test_boxes_that_span_the_lattice(ctx):
    V, T = _rod(12, 35.0, 2.0)
    ob = ctx.object_grid(V, T, 0.6, 128)
    G, _ = ob.export_grid()
    Go, _, _, fits = O.object_grid(V, T, 0.6, 128)
    assert fits and np.array_equal(G, Go.astype(np.float32))


@pytest.mark.parametrize("N, h", [(32, 0.6), (64, 0.3), (96, 0.5), (128, 0.15)])
@pytest.mark.parametrize("n", [2, 15, 16, 70])
def test_boxes_shared_by_a_warp_and_its_parts(ctx, N, h, n):
    # 4 to 140 triangles: a part of a warp, whole warps and a part, more than a block
    half = 0.5 * (N - 1) * h - 1.6
    V, T = _rod(max(n, 3), half, 0.7)
    V, T = V @ synth.quat_to_mat(synth.random_quat(np.random.default_rng(n))).T * 0.55, T[:2 * n]
    ob = ctx.object_grid(V, T, h, N)
    G, _ = ob.export_grid()
    Go, _, _, fits = O.object_grid(V, T, h, N)
    assert fits and np.array_equal(G, Go.astype(np.float32))
