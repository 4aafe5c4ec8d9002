"""How a batch's members are stepped, over the plans that its rule chooses from: clusters that
all run at once, shares of one grid, more members than SMs, the shared graph, and a graph for
the members that the resident blocks do not take.  Each against its members alone: bitwise."""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu

STEPS = 67


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


# sizes, and whether some member's steps are single launches of many steps (the team's)
PLANS = {
    "one_member_by_the_grid": ([20000], True),
    "clusters_of_16": ([500] * 4, True),
    "clusters_of_4": ([500] * 16, True),
    "clusters_of_1": ([500] * 64, True),
    "eight_clusters_of_16_do_not_run_at_once": ([4000] * 8, True),
    "shares_of_two": ([30000, 20001], True),
    "shares_small_beside_large": ([32768] + [700] * 9, True),
    "a_share_each": ([1000] * 150, True),
    "more_members_than_sms": ([300] * 155, True),
    "uneven_by_the_graph": ([20000] + [1500] * 151, False),
    "rest_beside_the_team": ([2000] * 9 + [40000], True),
    "few_beside_the_rest_by_the_graph": ([2000, 40000], False),
}


@pytest.mark.parametrize("name", list(PLANS))
@pytest.mark.parametrize("prec,kw", [("mixed", {}), ("fp64", {}),
                                     ("mixed", {"integrator": "nvt", "kT": 1.2, "tau": 0.5})],
                         ids=["mixed", "fp64", "nvt"])
def test_members_equal_each_alone(name, prec, kw):
    sizes, team = PLANS[name]
    # a few configurations of each size serve all of its members
    ws = {(n, q): wl.lj_fluid(n, 0.84, 1.2, seed=790 + q) for n in set(sizes) for q in range(2)}
    b = gbmd.Batch(prec)
    ss = [gbmd.System.from_workload(ws[n, k % 2], precision=prec, **kw) for k, n in enumerate(sizes)]
    for s in ss:
        b.add(s)
    b.set_tuning(2, 128)
    b.step(STEPS)
    b.sync()
    small = min(range(len(sizes)), key=lambda k: sizes[k])
    # the team: two launches beside those of create; the graph: one a step and more
    assert (ss[small].info()["kernel_launches"] < STEPS) == team
    got = [(*s.state(), *sorted(s.thermo().items())) for s in ss]
    b.close()
    want = {}
    for k, n in enumerate(sizes):
        if (n, k % 2) not in want:
            a = gbmd.System.from_workload(ws[n, k % 2], precision=prec, **kw)
            a.set_tuning(2, 128)
            a.step(STEPS)
            want[n, k % 2] = (*a.state(), *sorted(a.thermo().items()))
            a.close()
        for x, y in zip(got[k], want[n, k % 2]):
            assert np.array_equal(x, y) if isinstance(x, np.ndarray) else x == y
    for s in ss:
        s.close()
