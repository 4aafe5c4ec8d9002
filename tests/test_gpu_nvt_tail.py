"""The thermostat between the halves of a step by the separate kernels: each system's last
block takes the sum of the squares, its threads up to four slots side by side."""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


SIZES = [2, 15, 16, 17, 500, 8191, 8193, 33000]   # chunks from one to several turns of the slots


def members(prec):
    few = np.array([[-0.6, 0.1, 0.0], [0.6, 0.0, 0.2]])
    for n in SIZES:
        w = wl.Workload(few, 0.5 * few[::-1], np.zeros(2, np.int32), np.full(3, 9.0), wl.lj_single()) \
            if n == 2 else wl.lj_fluid(n, 0.84 if n >= 200 else 0.02, 1.2, seed=780 + n)
        yield gbmd.System.from_workload(w, precision=prec, integrator="nvt", kT=1.2, tau=0.5)


def result(s):
    return [*s.state(), *sorted(s.thermo().items())]


def same(a, b):
    return all(np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y for x, y in zip(a, b))


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("block", [32, 96, 128, 512])
def test_members_by_the_separate_kernels_equal_each_alone(prec, block, monkeypatch):
    """Members that stop at different steps, in one batch stepped by the separate kernels,
    against each by itself on its default route (resident blocks): bitwise."""
    want = []
    for k, s in enumerate(members(prec)):
        s.set_tuning(2, 128)
        s.step(5 + 3 * k)
        want.append(result(s))
        s.close()
    monkeypatch.setenv("GBMD_NO_GRAPHS", "1")
    b = gbmd.Batch(prec)
    ss = list(members(prec))
    for k, s in enumerate(ss):
        s.set_step_limit(5 + 3 * k)
        b.add(s)
    b.set_tuning(2, block)
    for _ in range(2):
        b.step(20)
    for s, w in zip(ss, want):
        assert same(result(s), w)
    b.close()
    for s in ss:
        s.close()
