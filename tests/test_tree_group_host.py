"""The group query of the tree neighbour list on the CPU: the periodic distance between
intervals against every pair of their points, and the leaves that a group's query visits
against the particles within reach of any of the group's (tests/host/tree_group.cpp over
csrc/tree_core.cuh)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
LEAF, STACK = 4, 1088   # TREE_LEAF and TREE_STACK of csrc


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("tree") / "libtree_group.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC",
                    os.path.join(HERE, "host", "tree_group.cpp"), "-o", out], check=True)
    lib = C.CDLL(out)
    lib.box_gap.restype = C.c_uint32
    lib.box_gap.argtypes = [C.c_uint32] * 4
    lib.group_leaves.argtypes = [C.c_int, C.c_void_p, C.c_void_p, C.c_void_p, C.c_float, C.c_int,
                                 C.c_int, C.c_void_p, C.c_void_p]
    return lib


@pytest.mark.parametrize("offset", [0, 1, 2 ** 28 - 1])
def test_interval_distance_equals_every_pair_of_points(lib, offset):
    """Circle of 16 points; `offset` moves all of them (the last to the end of the range)."""
    m, unit = 16, 2 ** 28
    d = np.abs(np.arange(m)[:, None] - np.arange(m)[None])
    d = np.minimum(d, m - d)
    for a in range(m):
        for b in range(a, m):
            for lo in range(m):
                for hi in range(lo, m):
                    want = int(d[a:b + 1, lo:hi + 1].min()) * unit
                    got = lib.box_gap(*(x * unit + offset for x in (a, b, lo, hi)))
                    assert got == want, (a, b, lo, hi)


def test_interval_distance_at_the_ends_of_the_range(lib):
    top = 2 ** 32 - 1
    assert lib.box_gap(0, top, 5, 5) == 0
    assert lib.box_gap(5, 5, 0, top) == 0
    assert lib.box_gap(0, top, 0, top) == 0
    assert lib.box_gap(0, 0, top, top) == 1          # neighbours through the face
    assert lib.box_gap(top, top, 0, 0) == 1
    assert lib.box_gap(0, 10, top - 4, top) == 1
    assert lib.box_gap(0, 0, 2 ** 31, 2 ** 31) == 2 ** 31
    assert lib.box_gap(1, 2, 4, top) == 2


def morton(u):
    """Morton code of the top 10 bits (the order of the cell sort)"""
    c = np.zeros(len(u), np.int64)
    for b in range(10):
        for a in range(3):
            c |= ((u[:, a].astype(np.int64) >> (22 + b)) & 1) << (3 * b + a)
    return c


@pytest.mark.parametrize("n,box,r", [(1, (6, 6, 6), 2.9), (5, (6, 6, 6), 2.9), (127, (9, 6, 12), 2.0),
                                     (700, (10, 10, 10), 2.0), (3000, (30, 8, 8), 1.5),
                                     (900, (5.9, 5.9, 5.9), 2.9)])
@pytest.mark.parametrize("per", [1, 8])
@pytest.mark.parametrize("how", ["morton", "random"])
def test_group_query_visits_every_leaf_within_reach(lib, n, box, r, per, how):
    box = np.array(box, float)
    rng = np.random.default_rng(n + per)
    pos = rng.uniform(-0.5, 0.5, (n, 3)) * box
    k = n // 2   # half of them at the faces x = +-L/2
    pos[:k, 0] = np.where(rng.random(k) < 0.5, -0.5, 0.5) * box[0] + rng.uniform(-0.3, 0.3, k)
    pos -= box * np.floor(pos / box + 0.5)
    q = np.rint(pos / box * 2.0 ** 32).astype(np.int64)
    u = np.ascontiguousarray(((q & 0xFFFFFFFF) ^ 0x80000000).astype(np.uint32))
    order = np.argsort(morton(u), kind="stable") if how == "morton" else rng.permutation(n)
    order = np.ascontiguousarray(order, np.int32)
    x = (u[order].astype(np.int64) - 2 ** 31) / 2.0 ** 32 * box
    leaves = np.zeros(n + 64, np.int32)
    deepest = C.c_int()
    for first in range(0, n, per):
        count = min(per, n - first)
        got = lib.group_leaves(n, u.ctypes.data, order.ctypes.data, box.ctypes.data,
                               r * r * (1.0 + 1e-5), first, count, leaves.ctypes.data,
                               C.addressof(deepest))
        assert got >= 0 and deepest.value <= STACK
        visited = leaves[:got]
        assert np.all(np.diff(visited) > 0)          # ascending: the order of the rows
        d = x[first:first + count, None] - x[None]
        d -= box * np.rint(d / box)
        near = ((d * d).sum(-1) < r * r).any(0)
        assert set(np.flatnonzero(near) // LEAF) <= set(visited.tolist())


def test_the_stack_holds_a_query_that_reaches_everything(lib):
    """2^20 particles of one place: every node is within reach, the deepest stack there is."""
    n = 2 ** 20
    u = np.full((n, 3), 7, np.uint32)
    order = np.arange(n, dtype=np.int32)
    box = np.full(3, 10.0)
    leaves = np.zeros(n // LEAF, np.int32)
    deepest = C.c_int()
    got = lib.group_leaves(n, u.ctypes.data, order.ctypes.data, box.ctypes.data, 1.0, 0, 8,
                           leaves.ctypes.data, C.addressof(deepest))
    assert got == n // LEAF and np.array_equal(leaves, np.arange(n // LEAF))
    assert deepest.value <= 32 * 18 + 64   # 32 a level at most, 64 on top
