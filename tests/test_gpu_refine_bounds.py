"""A query's distance where a search ends above the bound that ruled other
triangles out: on triangles of many millimetres the search of one triangle may
end 1e-5 above the lowest point it was given, and a neighbour whose value lies in
between must not be lost.  Poses that touch the edge between two side triangles
of a cylinder get the smallest of the triangles' own distances, bit for bit."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# (object pose, probe pose): found by comparing two million queries with an exhaustive evaluation
CASES = [
    ([0.9999961801314508, -0.001471433359351109, -0.002079939817663428, 0.0010716607349748795, 0.014562667540067433,
      -0.027956277037871277, -0.021714491295159975],
     [0.70613384533396, 0.7061338453339601, -0.03708089095309093, -0.03708089095309093, -0.3158283464784411,
      -2.998877511066707, 4.181410985357446]),
    ([0.9999939380804052, 0.0031503907466906363, 0.0013796538581074662, -0.0005435032822383734, 0.03397873326321046,
      0.031775900260125736, 0.0033482706631186177],
     [0.5608916540324332, -0.5608916540324332, -0.4305816443332916, 0.4305816443332916, -2.8801015912655026,
      0.77037489472242, -1.1869759146068573])]


@pytest.fixture(scope="module")
def ctx():
    from paper_2605_21398_gb300 import build, dock
    build.build()
    c = dock.Context(0)
    yield c
    c.close()


def _cylinder(n, radius, height):
    a = 2 * np.pi * np.arange(n) / n
    low = np.stack([radius * np.cos(a), radius * np.sin(a), 0 * a - height / 2], 1)
    V = np.concatenate([low, low + [0, 0, height], [[0, 0, -height / 2], [0, 0, height / 2]]])
    T = []
    for i in range(n):
        j = (i + 1) % n
        T += [(i, j, n + j), (i, n + j, n + i), (2 * n, j, i), (2 * n + 1, n + i, n + j)]
    return V, np.array(T, dtype=np.int32)


@pytest.mark.parametrize("case", [0, 1])
def test_no_neighbour_is_lost_to_a_bound(ctx, case):
    obj, probe = CASES[case]
    V, T = _cylinder(100, 3.0, 12.0)
    h, N = 0.3, 64
    # the probe alone
    sw = ctx.sweep_grid(np.array([probe]), 0.8, 3.0, h, N)
    full = ctx.distances(ctx.object_grid(V, T, h, N), sw, np.array([obj]))[0][0, 0]
    # every side triangle alone, with specks at the mesh's corners that keep its anchor
    lo, hi = V.min(axis=0), V.max(axis=0)
    specks = np.concatenate([lo + 1e-3 * np.eye(3) * [1, 1, 1], hi - 1e-3 * np.eye(3)])
    specks[0], specks[3] = lo, hi
    own = []
    for t in T[np.argsort(np.linalg.norm(V[T].mean(axis=1)[:, :2] - np.array(probe[4:6]), axis=1))][:24]:
        Vt = np.concatenate([V[t], specks])
        ob = ctx.object_grid(Vt, np.arange(9, dtype=np.int32).reshape(3, 3), h, N)
        own.append(ctx.distances(ob, sw, np.array([obj]))[0][0, 0])
        ob.close()
    assert np.isfinite(min(own)) and full == min(own), (full, min(own))
