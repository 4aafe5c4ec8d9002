"""Which kernels run a call: seen by the launches that the library counts."""
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
