"""Which kernels run a call: seen by the launches that the library counts."""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_event_records_leave_calls_of_many_steps_as_they_are(prec):
    """The records are for single steps; 64 steps are one launch with them as without."""
    import torch
    stream = torch.cuda.Stream()
    s = gbmd.System.from_workload(wl.lj_fluid(3000, 0.84, 1.2, seed=750), precision=prec,
                                  stream=stream.cuda_stream)
    ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
    for e in ev:
        e.record(stream)   # makes the CUDA event
    stream.synchronize()

    def launches(steps):
        s.sync()
        before = s.info()["kernel_launches"]
        s.step(steps)
        s.sync()
        return s.info()["kernel_launches"] - before

    assert launches(64) == 1
    s.set_force_events(*ev)
    assert launches(64) == 1
    assert launches(1) >= 1
    assert ev[0].elapsed_time(ev[1]) > 0.0   # the single step's force kernel was bracketed
    assert launches(64) == 1
    s.set_force_events(None, None)
    assert launches(1) == 1
    s.close()


def test_noalloc_thermo_of_a_tree_list_whose_wide_types_take_many_tiles():
    """2,197,000 particles, fewer than the 4,194,304 of the header, whose 66,575 far-reaching
    ones take four to an energy tile: 33,288 tiles."""
    m = 130
    g = np.arange(m) - 0.5 * (m - 1)
    rng = np.random.default_rng(760)
    pos = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    pos += rng.uniform(-0.05, 0.05, pos.shape)
    types = np.zeros(len(pos), np.int32)
    types[rng.permutation(len(pos))[:len(pos) // 33]] = 1
    rcut = np.array([[0.9, 2.4], [2.4, 2.4]])   # one type without neighbours, one with ~90
    pairs = wl.PairTable(np.full((2, 2), 0.1), np.full((2, 2), 0.9), rcut)
    w = wl.Workload(pos, np.zeros_like(pos), types, np.full(3, float(m)), pairs, r_buff=0.4)
    s = gbmd.System.from_workload(w, precision="fp64", nlist="tree", threads_per_particle=1)
    t = gbmd.gbmd_get_thermo_noalloc(s.handle)
    ref = gbmd.gbmd_get_thermo(s.handle)
    assert t["pe"] == ref["pe"] < 0.0 and t["virial"] == ref["virial"]
    s.close()


def test_a_batch_counts_the_launches_of_every_member():
    """A member that the team takes and one too large for it: 16 steps are one launch of
    the first and at least 16 of the second."""
    b = gbmd.Batch("mixed")
    ss = [gbmd.System.from_workload(wl.lj_fluid(n, 0.84, 1.2, seed=770)) for n in (2000, 60000)]
    for s in ss:
        b.add(s)
    b.step(16)
    b.sync()
    first = b.info()["kernel_launches"]
    assert first >= 16
    b.step(16)
    b.sync()
    assert b.info()["kernel_launches"] - first >= 16
    b.close()
    for s in ss:
        s.close()


@pytest.mark.parametrize("n,resident", [(20000, True), (100_000, False)])
def test_a_system_beside_work_on_another_stream_takes_no_launch_of_the_whole_chip(n, resident):
    """While another stream's steps have not been waited for, a system's steps are single
    launches, which the others' can run beside; the results are the same."""
    import torch
    streams = [torch.cuda.Stream() for _ in range(2)]
    w = wl.lj_fluid(n, 0.84, 1.2, seed=771)
    a, b = (gbmd.System.from_workload(w, stream=x.cuda_stream) for x in streams)
    a.sync()
    b.sync()

    def launches(s):
        return s.info()["kernel_launches"]   # waits for the system's stream alone

    start = launches(a)
    assert launches(b) == start
    a.step(64)                    # alone
    b.step(64)                    # beside a
    alone, beside = launches(a) - start, launches(b) - start
    if resident:
        assert alone == 1 and beside >= 64
    else:                         # the rebuild by one kernel, and by seven
        assert beside > alone >= 64
    for x, y in zip(a.state(), b.state()):
        assert np.array_equal(x, y)
    start = launches(b)
    b.step(64)                    # nothing pending elsewhere any more
    if resident:
        assert launches(b) - start == 1
    a.step(64)
    for x, y in zip((*a.state(), a.forces()), (*b.state(), b.forces())):
        assert np.array_equal(x, y)
    a.close()
    b.close()


def test_a_call_of_no_steps_leaves_its_stream_idle():
    import torch
    streams = [torch.cuda.Stream() for _ in range(2)]
    w = wl.lj_fluid(20000, 0.84, 1.2, seed=772)
    a, b = (gbmd.System.from_workload(w, stream=x.cuda_stream) for x in streams)
    for s in (a, b):
        s.sync()
    a.step(0)
    start = b.info()["kernel_launches"]
    b.step(64)
    assert b.info()["kernel_launches"] - start == 1
    a.close()
    b.close()
