"""FP64 pair forces over the range of the pair arithmetic: separations from far below any
the fluid reaches to the cut, along axes (components exactly zero) and across box
faces, in cubic and in very unequal boxes, for every potential.

The reference takes the same FP64 positions in extended precision.  Bound: f is a
difference of two terms t1 - t2.  d and r^2 carry at most 4 roundings (u = 2^-53), the
powers up to r^-14 multiply r^2's by 7, exp and pow add up to 16 ulp and the argument's
error times the argument (below 5 here): under 100 u of |t1| + |t2|, plus the fixed
point's units, below 2^-60 of the edge in d, times the force's slope, at most
15 (|t1| + |t2|) / r.
"""
import numpy as np
import pytest

from paper_1308_5587_gb300 import gbmd, workloads as wl

pytestmark = pytest.mark.gpu
U = 2.0 ** -53
POTS = {"lj": wl.lj_single, "mie": wl.mie_single, "wca": wl.wca_single,
        "yukawa": wl.yukawa_single, "gauss": wl.gauss_single}


@pytest.fixture(scope="module", autouse=True)
def _setup():
    from paper_1308_5587_gb300 import _build
    _build.build()


def pairs_in(box, rc, rng, lo):
    """Isolated pairs on a grid of sites farther apart than two cuts."""
    m = np.maximum((box / (2.6 * rc + 1.0)).astype(int), 1)
    m = np.minimum(m, 7)
    g = np.stack(np.meshgrid(*[(np.arange(k) / k - 0.5) for k in m], indexing="ij"), -1)
    a = g.reshape(-1, 3) * box + 1e-3 * rng.standard_normal((int(np.prod(m)), 3))
    d = rng.standard_normal(a.shape)
    d[::4, 0] = 0.0
    d[::8, 1] = 0.0
    a[::4] = np.round(a[::4] * 1024) / 1024   # so that equal coordinates stay equal
    d *= (np.exp(rng.uniform(np.log(lo), np.log(0.999 * rc), len(a))) /
          np.linalg.norm(d, axis=1))[:, None]
    return np.concatenate([a, a - d])


def terms(t, r):
    """The two terms of the pair force's magnitude."""
    e, s = float(t.eps[0, 0]), float(t.sigma[0, 0])
    if t.potential in ("lj", "wca"):
        return 48 * e * (s / r) ** 12 / r, 24 * e * (s / r) ** 6 / r
    if t.potential == "mie":
        n, m = float(t.mie_n[0, 0]), float(t.mie_m[0, 0])
        c = n / (n - m) * (n / m) ** (m / (n - m)) * e
        return c * n * (s / r) ** n / r, c * m * (s / r) ** m / r
    if t.potential == "yukawa":
        k = float(t.kappa[0, 0])
        return e * np.exp(-k * r) / r ** 2, -e * np.exp(-k * r) * k / r
    return e / s ** 2 * r * np.exp(-r * r / (2 * s * s)), 0 * r


@pytest.mark.parametrize("pot", list(POTS))
@pytest.mark.parametrize("box", [(9.0, 9.0, 9.0), (70.0, 40.0, 1900.0), (64.0, 64.0, 64.0)])
@pytest.mark.parametrize("tpp", [1, 4])
def test_fp64_forces_of_isolated_pairs(pot, box, tpp):
    t = POTS[pot]()
    box = np.array(box)
    rc = 2.0 ** (1.0 / 6.0) if pot == "wca" else float(np.asarray(t.rcut)[0, 0])
    pos = pairs_in(box, rc, np.random.default_rng(41), lo=1e-3)
    w = wl.Workload(pos, np.zeros_like(pos), np.zeros(len(pos), np.int32), box, t, r_buff=0.4)
    s = gbmd.System.from_workload(w, precision="fp64", threads_per_particle=tpp)
    x = s.state()[0]
    F = s.forces()
    n = len(pos) // 2
    L = box.astype(np.longdouble)
    d = x[:n].astype(np.longdouble) - x[n:]
    d -= L * np.rint(d / L)
    r = np.sqrt((d * d).sum(1))
    t1, t2 = terms(t, r)
    want = ((t1 - t2) / r)[:, None] * d
    bound = (np.abs(t1) + np.abs(t2)) * (100 * U + 15 * 2.0 ** -60 * box.max() / r)
    assert np.all(r < rc)
    for got in (F[:n], -F[n:]):
        assert np.all(np.sqrt(((got - want) ** 2).sum(1)) <= bound)
    s.close()
