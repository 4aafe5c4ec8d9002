"""The resident team kernel and the cooperative rebuild against the separate kernels.

A system's steps run by a cluster, by the grid of a cooperative launch or by the step
kernel with the rebuild as one cooperative kernel; GBMD_NO_GRAPHS=1 at create launches
the separate kernels one by one.  The rows, the order of every sum and so the
trajectories are the same: every comparison here is bitwise.
"""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu

STEPS = 67   # more than one launch of the team kernel (64 steps), the last one ragged


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


def four_types(n, seed):
    base = wl.lj_fluid(n, 0.9, 1.2, seed=seed)
    types = np.random.default_rng(seed).integers(0, 4, base.n).astype(np.int32)
    a = np.arange(4)
    sigma = 0.85 + 0.05 * np.abs(a[:, None] - a[None, :])
    pairs = wl.PairTable(0.6 + 0.2 * (a[:, None] + a[None, :]), sigma, 2.5 * sigma)
    return wl.Workload(base.pos, base.vel, types, base.box, pairs, r_buff=0.4)


def few(n):
    """One or two particles, which the lattice generator does not spread."""
    pos = np.array([[-0.6, 0.1, 0.0], [0.6, 0.0, 0.2]])[:n]
    return wl.Workload(pos, 0.5 * pos[::-1], np.zeros(n, np.int32), np.full(3, 9.0),
                       wl.lj_single(), r_buff=0.4)


def fluid(n, **kw):
    rho = 0.84 if n >= 200 else 0.1   # the box holds two list radii on each axis
    return lambda: wl.lj_fluid(n, rho, 1.2, seed=300 + n, **kw)


def clump(n_side=12):
    """Soft particles crowded at the centre: some cells hold many times the mean."""
    u = (np.arange(n_side) - 0.5 * (n_side - 1)) / (0.5 * n_side)
    pos = np.stack(np.meshgrid(u, u, u, indexing="ij"), -1).reshape(-1, 3)
    pos = 9.0 * pos * np.abs(pos)
    return wl.Workload(pos, -0.3 * pos, np.zeros(len(pos), np.int32), np.full(3, 18.0),
                       wl.gauss_single(), r_buff=0.4)


# name: (workload, precision, create options).  Sizes at the edges of the rules: a cluster
# of one block, of 16, the whole grid, the largest team, the cooperative rebuild alone;
# two cells an axis (raw fixed point), four warps a cell and one; every pair-table mode.
CASES = {
    "n1": (lambda: few(1), "mixed", {}),
    "n2_fp64_nvt": (lambda: few(2), "fp64", {"nvt": 1.0}),
    "n33": (fluid(33), "mixed", {"sort_period": 1}),
    "n500_two_cells": (fluid(500), "mixed", {}),
    "n500_fp64_nvt": (fluid(500), "fp64", {"nvt": 1.2}),
    "n2049_cluster_16": (fluid(2049), "mixed", {"sort_period": 10}),
    "n4097_grid_nvt": (fluid(4097), "mixed", {"nvt": 1.2, "sort_period": 10}),
    "n4097_fp64_grid": (fluid(4097), "fp64", {"sort_period": 10}),
    "ka_3001": (lambda: wl.lj_fluid(3001, 1.2, 1.0, seed=31, binary=True, r_buff=0.3), "mixed", {}),
    "ka_3001_fp64": (lambda: wl.lj_fluid(3001, 1.2, 1.0, seed=32, binary=True, r_buff=0.3),
                     "fp64", {}),
    "four_types_2500": (lambda: four_types(2500, 33), "mixed", {"sort_period": 5}),
    "mie_4500": (fluid(4500, pairs=wl.mie_single()), "mixed", {}),
    "yukawa_20011_nvt": (fluid(20011, pairs=wl.yukawa_single()), "mixed",
                         {"nvt": 1.2, "sort_period": 20}),
    "gauss_700_fp64": (fluid(700, pairs=wl.gauss_single()), "fp64", {}),
    "n49152_team": (fluid(49152), "mixed", {"sort_period": 30}),
    "n49153_two_in_one": (fluid(49153), "mixed", {"sort_period": 30}),
    "n77824_team_two_in_one": (fluid(77824), "mixed", {"sort_period": 30}),
    "n40001_two_in_one_nvt": (fluid(40001), "mixed", {"nvt": 1.2}),
    "ka_39001_two_in_one": (lambda: wl.lj_fluid(39001, 1.2, 1.0, seed=39, binary=True, r_buff=0.3),
                            "mixed", {}),
    "n77825_coop_rebuild": (fluid(77825), "mixed", {}),
    "n60001_fp64_team": (fluid(60001), "fp64", {"sort_period": 30}),
    "clump_1728_buckets_run_over": (clump, "mixed", {"sort_period": 3}),
    "dilute_1500_no_buckets": (lambda: wl.lj_fluid(1500, 0.02, 1.2, seed=38), "mixed",
                               {"sort_period": 2}),
    "n33001_fp64_one_lane": (fluid(33001), "fp64", {}),
    "tree_3000": (lambda: wl.colloid_mixture(3000, ratio=5.0, seed=34), "mixed",
                  {"nlist": "tree", "sort_period": 10}),
    "tree_20000_r10_fp64": (lambda: wl.colloid_mixture(20000, ratio=10.0, seed=35), "fp64",
                            {"nlist": "tree"}),
}


def create(name):
    make, prec, opt = CASES[name]
    w, opt = make(), dict(opt)
    kT = opt.pop("nvt", None)
    if kT:
        opt.update(integrator="nvt", kT=kT, tau=0.5)
    return gbmd.System.from_workload(w, precision=prec, **opt)


def result(s):
    info = s.info()
    counts, idx = s.neighbors(cap=int(info["nlist_capacity"]))
    u, vir = s.per_particle()
    th = s.thermo()
    return [*s.state(), s.forces(), counts, idx, u, vir, *sorted(th.items()),
            info["n_rebuilds"], info["n_sorts"]]


def assert_same(a, b):
    assert len(a) == len(b)
    for k, (x, y) in enumerate(zip(a, b)):
        if isinstance(x, np.ndarray):
            assert np.array_equal(x, y), k
        else:
            assert x == y, (k, x, y)


@pytest.mark.parametrize("name", list(CASES))
def test_resident_steps_equal_the_separate_kernels(name, monkeypatch):
    s = create(name)
    s.step(STEPS)
    got = result(s)
    monkeypatch.setenv("GBMD_NO_GRAPHS", "1")
    plain = create(name)
    plain.step(STEPS)
    want = result(plain)
    assert_same(got, want)
    # and in single steps, with a readout between: one launch each
    monkeypatch.delenv("GBMD_NO_GRAPHS")
    one = create(name)
    for _ in range(5):
        one.step(1)
        one.forces()
    one.step(STEPS - 5)
    assert_same(result(one), want)
    for x in (s, plain, one):
        x.close()


def test_batch_of_every_cluster_size_and_the_rest_equals_alone():
    """Members from two particles to more than a batch's team takes (stepped by the
    graph of the rest), and one on the tree list, in one batch."""
    ws = [few(2), *(fluid(n, pairs=wl.wca_single())()
                    for n in (130, 700, 2500, 9000, 32768, 32769)),
          wl.colloid_mixture(2000, ratio=4.0, seed=36)]
    ws[0].pairs = wl.wca_single()
    kinds = ["cell"] * 7 + ["tree"]
    want = []
    for w, nl in zip(ws, kinds):
        s = gbmd.System.from_workload(w, precision="mixed", nlist=nl, sort_period=20)
        s.set_tuning(2, 128)
        s.step(STEPS)
        want.append((s.state(), s.forces(), s.thermo()))
        s.close()
    b = gbmd.Batch("mixed")
    b.set_tuning(2, 128)
    ss = [gbmd.System.from_workload(w, precision="mixed", nlist=nl, sort_period=20)
          for w, nl in zip(ws, kinds)]
    for s in ss:
        b.add(s)
    b.step(STEPS)
    for s, (st, F, th) in zip(ss, want):
        for x, y in zip(s.state(), st):
            assert np.array_equal(x, y)
        assert np.array_equal(s.forces(), F)
        assert s.thermo() == th
    b.close()
    for s in ss:
        s.close()


@pytest.mark.parametrize("sizes", [
    [2, 300, 1000, 2300, 2600, 3100, 3700, 4100, 4800, 5500, 6300, 7200, 8300, 9000],
    [240 + k for k in range(160)]], ids=["shares_of_one_grid", "more_teams_than_SMs"])
def test_batch_of_many_members_equals_alone(sizes):
    ws = [few(n) if n == 2 else fluid(n)() for n in sizes]
    b = gbmd.Batch("mixed")
    b.set_tuning(2, 128)
    ss = [gbmd.System.from_workload(w, precision="mixed") for w in ws]
    for s in ss:
        b.add(s)
    b.step(STEPS)
    got = [(s.state(), s.thermo()) for s in ss]
    b.close()
    for w, s, (st, th) in list(zip(ws, ss, got))[::max(1, len(ws) // 16)]:
        a = gbmd.System.from_workload(w, precision="mixed")
        a.set_tuning(2, 128)
        a.step(STEPS)
        for x, y in zip(a.state(), st):
            assert np.array_equal(x, y)
        assert a.thermo() == th
        a.close()
    for s in ss:
        s.close()


@pytest.mark.parametrize("name", ["n33", "n500_fp64_nvt", "n4097_grid_nvt", "tree_3000",
                                  "n33001_fp64_one_lane"])
def test_readouts_of_parts_equal_the_whole(name):
    """Each array of a readout alone (positions without the force kernel) and in pairs, small
    (one copy) and large, against the whole state."""
    import ctypes
    s = create(name)
    s.step(7)
    n = s.info()["n"]
    pos, vel, image, step = s.state()
    whole = {"pos": pos, "vel": vel, "image": image}
    F = s.forces()
    for parts in (["pos"], ["vel"], ["image"], ["pos", "image"], ["vel", "image"], ["pos", "vel"]):
        got = {k: np.full_like(whole[k], -7) for k in parts}
        at = ctypes.c_int64()
        args = [got[k].ctypes.data_as(ctypes.c_void_p) if k in got else None
                for k in ("pos", "vel", "image")]
        assert gbmd.load().gbmd_get_state(s.handle, *args, ctypes.byref(at)) == 0
        assert at.value == step and len(pos) == n
        for k in parts:
            assert np.array_equal(got[k], whole[k]), (parts, k)
        assert np.array_equal(s.forces(), F)
    s.close()


@pytest.mark.parametrize("n", [2, 31, 33, 4095, 131072, 131073])
@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_thermo_sums_at_the_edges_of_its_tiles(prec, n):
    """The reduced sums against the per-particle values, added up in extended precision:
    both add the same FP64 numbers, up to n of them one after another at worst, so the
    difference is below n 2^-53 of the sum of magnitudes (the blocks add far fewer)."""
    s = gbmd.System.from_workload(few(2) if n == 2 else fluid(n)(),
                                  precision=prec)
    s.step(3)
    u, vir = s.per_particle()
    vel = s.state()[1]
    th = s.thermo()
    terms = [(th["pe"], u), (th["ke"], 0.5 * vel.ravel() ** 2)]
    terms += [(th["virial"][c], vir[:, c]) for c in range(6)]
    for got, x in terms:
        # + 4 ulp a term: v.v is formed with fused multiply-adds
        bound = (n + 4) * 2.0 ** -53 * float(np.abs(x).sum()) + 1e-300
        assert abs(got - float(np.sum(x.astype(np.longdouble)))) <= bound
    s.close()


def test_fp64_rows_from_empty_to_longer_than_the_queue():
    """FP64 forces where neighbouring lanes hold rows of very different lengths: a dense
    droplet in a dilute gas (queues that stay empty, fill up and wrap round)."""
    import oracle
    oracle.build()
    rng = np.random.default_rng(37)
    g = (np.arange(7) - 3.0) * 0.9
    drop = np.stack(np.meshgrid(g, g, g, indexing="ij"), -1).reshape(-1, 3)
    gas = rng.uniform(-14.0, 14.0, (900, 3))
    gas = gas[np.abs(gas).max(1) > 4.0]
    d = gas[:, None] - gas[None]
    d -= 28.0 * np.rint(d / 28.0)
    close = (d ** 2).sum(-1) < 0.81
    gas = gas[~np.triu(close, 1).any(0)]
    pos = np.concatenate([drop + 0.02 * rng.standard_normal(drop.shape), gas])
    pos = pos[rng.permutation(len(pos))]
    for kw in ({}, {"threads_per_particle": 1}):
        s = gbmd.System(pos, np.zeros_like(pos), np.full(3, 28.0), precision="fp64", **kw)
        counts = s.neighbors(cap=int(s.info()["nlist_capacity"]))[0]
        assert counts.min() <= 3 and counts.max() > 64
        F = s.forces()
        Fo, *_ = oracle.forces(s.state()[0], np.full(3, 28.0), np.zeros(len(pos), np.int32),
                               wl.lj_single().as_dict())
        assert np.linalg.norm(F - Fo) <= 1e-12 * np.linalg.norm(Fo)
        s.close()
