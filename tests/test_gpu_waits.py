"""Kernels whose blocks wait for each other: systems on different streams and threads at the
same time; and launches of many waves in which an early block ends the run, so that warps
of later blocks find the system frozen; and waits that run out.  GBMD_TEAM_POLLS = 0 at a
new layout lets every wait in memory run out at once: the blocks that are not the last to
arrive give up, the kernel returns by itself and the system stops with TIMEOUT."""
import threading

import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


def rounds(w, stream, out, **kw):
    """New states, single steps and readouts over and over: rebuilds inside and outside
    of the steps, each a launch whose blocks wait for each other."""
    s = gbmd.System.from_workload(w, stream=stream, **kw)
    for k in range(12):
        s.set_state(w.pos, w.vel * (1.0 + 0.01 * k))
        s.step(7)
        out.append((*s.state(), s.forces()))
    s.close()


@pytest.mark.parametrize("n", [3000, 30011, 90001])
def test_systems_on_streams_of_their_own_equal_one_after_another(n):
    import torch
    ws = [wl.lj_fluid(n, 0.84, 1.2, seed=700 + k) for k in range(3)]
    opt = [{"precision": "mixed"}, {"precision": "fp64"}, {"precision": "mixed", "sort_period": 5}]
    want = [[] for _ in ws]
    for w, kw, o in zip(ws, opt, want):
        rounds(w, None, o, **kw)
    got = [[] for _ in ws]
    streams = [torch.cuda.Stream() for _ in ws]
    ts = [threading.Thread(target=rounds, args=(w, st.cuda_stream, o), kwargs=kw)
          for w, st, o, kw in zip(ws, streams, got, opt)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    for g, e in zip(got, want):
        assert len(g) == len(e) == 12
        for a, b in zip(g, e):
            for x, y in zip(a, b):
                assert np.array_equal(x, y)


def overlapping_at_the_corner(w):
    """Two particles of one type at one place, at the start of the sort order: blocks of the
    first wave find the non-finite force."""
    a = int(np.argmin((w.pos + 0.5 * w.box).sum(1)))
    d = w.pos - w.pos[a]
    d -= w.box * np.rint(d / w.box)
    r2 = np.where(w.types == w.types[a], (d * d).sum(1), np.inf)
    r2[a] = np.inf
    pos = w.pos.copy()
    pos[int(np.argmin(r2))] = pos[a]
    return pos


@pytest.mark.parametrize("name,kw", [
    ("lj", {"threads_per_particle": 2}), ("lj", {"threads_per_particle": 4}),
    ("lj", {"threads_per_particle": 1}), ("lj", {"precision": "fp64"}),
    ("lj", {"integrator": "nvt", "kT": 1.2, "tau": 0.5}), ("lj", {"force_path": "staged"}),
    ("colloid", {"nlist": "tree"})])
def test_a_launch_of_many_waves_ends_when_an_early_block_finds_a_non_finite_force(name, kw):
    """Step kernels (no team at these sizes), hundreds to thousands of blocks."""
    w = wl.lj_fluid(120_000, 0.84, 1.2, seed=710) if name == "lj" else \
        wl.colloid_mixture(100_000, ratio=10.0, seed=711)
    s = gbmd.System.from_workload(w, **kw)
    s.step(2)
    s.sync()
    s.set_state(overlapping_at_the_corner(w), w.vel)
    for _ in range(2):
        s.step(3)
        with pytest.raises(gbmd.GbmdError) as e:
            s.sync()
        assert e.value.status == "NONFINITE"
    s.close()


def dead(call):
    with pytest.raises(gbmd.GbmdError) as e:
        call()
    assert e.value.status == "TIMEOUT", e.value


def test_create_reports_a_wait_that_ran_out(monkeypatch):
    w = wl.lj_fluid(5000, 0.84, 1.2, seed=720)
    want = gbmd.System.from_workload(w).forces()
    for kw in ({}, {"precision": "fp64"}):
        monkeypatch.setenv("GBMD_TEAM_POLLS", "0")
        dead(lambda: gbmd.System.from_workload(w, **kw))
        monkeypatch.delenv("GBMD_TEAM_POLLS")
    c = wl.colloid_mixture(3000, ratio=5.0, seed=721)
    monkeypatch.setenv("GBMD_TEAM_POLLS", "0")
    dead(lambda: gbmd.System.from_workload(c, nlist="tree"))
    monkeypatch.delenv("GBMD_TEAM_POLLS")
    s = gbmd.System.from_workload(w)
    assert np.array_equal(s.forces(), want)
    s.close()


@pytest.mark.parametrize("n,kw", [(8000, {}), (8000, {"precision": "fp64"}),
                                  (8000, {"integrator": "nvt", "kT": 1.2, "tau": 0.5}),
                                  (100_000, {})])   # the last: by k_rebuild
def test_steps_report_a_wait_that_ran_out_and_the_system_stays_stopped(n, kw, monkeypatch):
    w = wl.lj_fluid(n, 0.84, 1.2, seed=722)
    s = gbmd.System.from_workload(w, **kw)
    s.step(2)
    s.sync()
    monkeypatch.setenv("GBMD_TEAM_POLLS", "0")
    t = s.info()
    s.set_tuning(t["threads_per_particle"], 256)   # a new layout
    s.step(60)
    dead(s.sync)
    monkeypatch.delenv("GBMD_TEAM_POLLS")
    s.step(5)
    for call in (s.sync, s.forces, s.thermo, s.state, lambda: s.set_state(w.pos, w.vel),
                 lambda: s.set_cell_scale(1.2)):
        dead(call)
    s.close()


def test_a_batch_goes_on_with_new_members_after_waits_that_ran_out(monkeypatch):
    """Shares of one grid, whose barrier words the next members' teams take over, and a lone
    tree member, which the graph of the rest rebuilds by its own resident grid."""
    sizes = [2000, 300, 1000, 2300, 2600, 3100, 3700, 4100, 4800, 5500, 6300, 7200, 8300, 9000]
    ws = [wl.lj_fluid(n, 0.84, 1.2, seed=730 + n, pairs=wl.wca_single()) for n in sizes]
    ws.append(wl.colloid_mixture(3000, ratio=4.0, seed=731))
    make = lambda: [gbmd.System.from_workload(w, nlist="tree" if k == len(sizes) else "cell")
                    for k, w in enumerate(ws)]
    want = []
    for s in make():
        s.set_tuning(2, 128)
        s.step(70)
        want.append((*s.state(), s.forces()))
        s.close()
    b = gbmd.Batch("mixed")
    b.set_tuning(2, 128)
    ss = make()
    for s in ss:
        b.add(s)
    monkeypatch.setenv("GBMD_TEAM_POLLS", "0")
    b.step(70)
    monkeypatch.delenv("GBMD_TEAM_POLLS")
    for s in ss:
        s.close()
    ss = make()
    for s in ss:
        b.add(s)
    b.step(70)
    for s, e in zip(ss, want):
        for x, y in zip((*s.state(), s.forces()), e):
            assert np.array_equal(x, y)
    b.step(70)
    b.sync()
    b.close()
    for s in ss:
        s.close()
