"""The autotuner times the steps as they are run and puts the system back as it was."""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


def close_velocities(a, b, prec):
    # half a kick of the force, whose sums take another order after another choice of lanes
    # or cells: 0.0025 times a relative 1e-5 (FP32) or 1e-12 of forces of a few hundred
    assert np.abs(a - b).max() <= 0.0025 * (1e-5 if prec == "mixed" else 1e-12) * 1e3


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("kw", [{}, {"integrator": "nvt", "kT": 1.2, "tau": 0.5}, {"nlist": "tree"}])
def test_the_state_is_as_before(prec, kw):
    w = wl.lj_fluid(3001, 0.84, 1.2, seed=740)
    s = gbmd.System.from_workload(w, precision=prec, sort_period=10, **kw)
    s.step(23)
    s.set_step_limit(25)   # the tuner's steps count neither against it nor into the state
    pos, vel, image, step = s.state()
    th, n_rebuilds = s.thermo(), s.info()["n_rebuilds"]
    s.autotune(None)
    pos2, vel2, image2, step2 = s.state()
    assert step2 == step == 23 and s.info()["n_rebuilds"] - n_rebuilds == 0
    assert np.array_equal(pos, pos2) and np.array_equal(image, image2)
    close_velocities(vel, vel2, prec)
    th2 = s.thermo()
    if "kT" in kw:
        assert abs(th2["eta"] - th["eta"]) <= 1e-6 * abs(th["eta"]) and th["eta"] != 0.0
    s.step(10)
    s.sync()
    assert s.info()["step"] == 25
    s.close()


def test_a_batch_is_as_before():
    """Small members, which the team steps, one beyond it and one on the tree list."""
    ws = [wl.lj_fluid(n, 0.84, 1.2, seed=741, pairs=wl.wca_single()) for n in (600, 2500, 9000, 40000)]
    ws.append(wl.colloid_mixture(2000, ratio=4.0, seed=742))
    b = gbmd.Batch("mixed")
    ss = [gbmd.System.from_workload(w, nlist="tree" if k == 4 else "cell") for k, w in enumerate(ws)]
    for s in ss:
        b.add(s)
    b.step(21)
    before = [s.state() for s in ss]
    b.autotune(None)
    for s, (pos, vel, image, step) in zip(ss, before):
        pos2, vel2, image2, step2 = s.state()
        assert step2 == step == 21
        assert np.array_equal(pos, pos2) and np.array_equal(image, image2)
        close_velocities(vel, vel2, "mixed")
    b.step(20)
    b.sync()
    b.close()
    for s in ss:
        s.close()


def us_per_step(s, stream, steps=128):
    import torch
    s.step(64)
    s.sync()
    t = []
    for _ in range(5):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        a.record(stream)
        s.step(steps)
        b.record(stream)
        s.sync()
        t.append(a.elapsed_time(b) * 1e3 / steps)
    return sorted(t)[2]


@pytest.mark.parametrize("prec,n", [("mixed", 20000), ("fp64", 40000)])
def test_the_choice_is_no_slower_than_the_default(prec, n):
    """By the step kernel's times of its candidates the choice stepped 26% and 19% slower
    than the default here.  Three tries, for a GPU that others load."""
    import torch
    stream = torch.cuda.Stream()
    ratios = []
    for _ in range(3):
        s = gbmd.System.from_workload(wl.lj_fluid(n, 0.84, 1.2, seed=5), precision=prec,
                                      stream=stream.cuda_stream)
        default = us_per_step(s, stream)
        s.autotune(None)
        ratios.append(us_per_step(s, stream) / default)
        s.close()
        if ratios[-1] <= 1.1:
            return
    raise AssertionError(ratios)
