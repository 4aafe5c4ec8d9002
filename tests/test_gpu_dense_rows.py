"""Neighbour rows where a lane's buffer of waiting hits fills to its last slot.

The builder of one warp a cell (csrc/nlist_warp.cuh) tests candidates 32 at a time and
empties the buffer when some lane holds more than SLOTS - 32 hits; a lane that holds
exactly SLOTS - 32 and finds a chunk full of hits ends with SLOTS.  The cell here holds
two tight clumps of 48, all within reach of each other, and the cell before it in the
stencil's order `before` particles that are within reach of the clumps' bounding box (they
pass the cull) but of no particle: the second pass over the cell's members then tests the
chunk (before, 32 - before members) and the chunk of the next 32 members.
"""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu

CLUMP = 48


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


def dense_cell(before):
    pairs = wl.gauss_single()
    r = float(pairs.rcut[0, 0]) + 0.4          # r_list
    edge = 12 * 1.02 * r                       # 12 cells an axis, more than the split builder takes
    corner = np.full(3, -0.5 * edge + 5 * edge / 12)
    rng = np.random.default_rng(51)
    at = lambda x, z, m: corner + r * np.array([x, 0.5, z]) + 1e-3 * rng.standard_normal((m, 3))
    low, high = at(0.5, 0.05, CLUMP), at(0.1, 0.5, CLUMP)
    far = at(0.1 - 0.68, 0.05 - 0.68, before)
    runner = corner + r * np.array([[4.3, 4.4, 4.1]])   # moves enough for a rebuild at each step
    pos = np.concatenate([low, high, far, runner])
    # the geometry that the docstring states
    box_lo, box_hi = pos[:2 * CLUMP].min(0), pos[:2 * CLUMP].max(0)
    gap = np.maximum(np.maximum(box_lo - far, far - box_hi), 0.0)
    assert np.linalg.norm(gap, axis=1).max() < 0.99 * r
    d = np.linalg.norm(pos[:2 * CLUMP, None] - far[None], axis=-1)
    assert d.min() > 1.05 * r
    inner = np.linalg.norm(pos[:2 * CLUMP, None] - pos[None, :2 * CLUMP], axis=-1)
    assert inner.max() < 0.95 * r
    vel = np.zeros_like(pos)
    vel[-1] = [60.0, 30.0, 0.0]                # 0.33 a step: more than half of r_buff
    return pos, vel, edge, pairs, r


def waiting(before, slots):
    """The most hits that wait in a lane's buffer during the second pass: its members 32 .. 63
    against the stream (before, members 0 .. 2 CLUMP - 1), 32 candidates at a time."""
    stream = [-1] * before + list(range(2 * CLUMP))
    lanes, most = np.zeros(32, int), 0
    for c in range(0, len(stream), 32):
        for lane in range(32):
            lanes[lane] += sum(m >= 0 and m != 32 + lane for m in stream[c:c + 32])
        most = max(most, int(lanes.max()))
        if lanes.max() > slots - 32:
            lanes %= 4
    return most


@pytest.mark.parametrize("before,slots", [(8, 56), (24, 40)])
@pytest.mark.parametrize("route", ["resident", "separate"])
def test_rows_of_a_full_buffer(before, slots, route, monkeypatch):
    assert waiting(before, slots) == slots
    if route == "separate":
        monkeypatch.setenv("GBMD_NO_GRAPHS", "1")
    pos, vel, edge, pairs, r = dense_cell(before)
    w = wl.Workload(pos, vel, np.zeros(len(pos), np.int32), np.full(3, edge), pairs, r_buff=0.4)
    s = gbmd.System.from_workload(w, nlist_capacity=160)
    for step in range(3):
        x = s.state()[0]
        d = x[:, None] - x[None]
        d -= edge * np.rint(d / edge)
        near = (d * d).sum(-1)
        assert np.abs(np.sqrt(near) - r).min() > 1e-6   # none within the rounding of the list's test
        want = near < r * r
        np.fill_diagonal(want, False)
        counts, idx = s.neighbors(cap=160)
        assert np.array_equal(counts, want.sum(1))
        for i in range(len(x)):
            assert np.array_equal(idx[i, :counts[i]], np.flatnonzero(want[i]))
        s.step(1)
    s.close()
