"""The tree over an object's triangles (csrc/bvh.h, compiled here for the host):
the threads that build it are limited, and the tree is the same for any number."""
import ctypes
import os
import subprocess
import threading

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_21398_gb300", "csrc")

SHIM = r"""
#include "bvh.h"
#include <cstring>
extern "C" long long tree(const double *V, const int *T, long long nt, int threads, int *order, int *nodes)
{
    dock::BvhBuilder B;
    dock::build_bvh(V, T, nt, B, threads);
    memcpy(order, B.order.data(), sizeof(int) * nt);
    for (size_t i = 0; i < B.nodes.size(); ++i) {
        nodes[3 * i] = B.nodes[i].left;
        nodes[3 * i + 1] = B.nodes[i].first;
        nodes[3 * i + 2] = B.nodes[i].count;
    }
    return (long long)B.nodes.size();
}
"""


@pytest.fixture(scope="module")
def tree(tmp_path_factory):
    from paper_2605_21398_gb300 import build
    d = tmp_path_factory.mktemp("bvh")
    src, so = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    cuda = os.path.join(os.path.dirname(os.path.dirname(build._nvcc())), "include")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I", CSRC, "-I", cuda, "-o", so, src, "-lpthread"],
                   check=True)
    fn = ctypes.CDLL(so).tree
    dp, ip = ctypes.POINTER(ctypes.c_double), ctypes.POINTER(ctypes.c_int)
    fn.restype = ctypes.c_longlong
    fn.argtypes = [dp, ip, ctypes.c_longlong, ctypes.c_int, ip, ip]

    def run(V, T, threads):
        order, nodes = np.empty(len(T), np.int32), np.full((len(T) + 2, 3), -7, np.int32)
        n = fn(V.ctypes.data_as(dp), T.ctypes.data_as(ip), len(T), threads, order.ctypes.data_as(ip), nodes.ctypes.data_as(ip))
        return order, nodes[:n]
    return run


def _mesh(n):
    rng = np.random.default_rng(n)
    V = np.repeat(rng.normal(size=(n, 1, 3)), 3, axis=1) + 0.01 * rng.normal(size=(n, 3, 3))
    return np.ascontiguousarray(V.reshape(-1, 3)), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


@pytest.mark.parametrize("n", [1, 4, 5, 8191, 8192, 20001])
@pytest.mark.parametrize("threads", [2, 3, 16])
def test_tree_does_not_depend_on_the_threads(tree, n, threads):
    V, T = _mesh(n)
    order, nodes = tree(V, T, threads)
    one, nodes1 = tree(V, T, 1)
    assert np.array_equal(order, one) and np.array_equal(nodes, nodes1)
    assert np.array_equal(np.sort(order), np.arange(n))
    leaves = nodes[nodes[:, 0] < 0]
    assert leaves[:, 2].sum() == n and leaves[:, 2].max() <= 4


def _threads():
    return len(os.listdir("/proc/self/task"))


@pytest.mark.parametrize("limit", [1, 5, 16])
def test_threads_are_limited(tree, limit):
    V, T = _mesh(600000)   # a thread at every node of 8192 triangles would be 127
    before, seen, done = _threads(), [0], threading.Event()

    def watch():
        while not done.is_set():
            seen[0] = max(seen[0], _threads())

    w = threading.Thread(target=watch)
    w.start()
    tree(V, T, limit)
    done.set()
    w.join()
    # the caller is one of them, the watcher beside
    assert seen[0] - before - 1 <= limit - 1
