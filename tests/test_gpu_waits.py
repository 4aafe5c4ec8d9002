"""Kernels whose blocks wait for each other: systems on different streams and threads at the
same time."""
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
