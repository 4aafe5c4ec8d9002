"""A kernel whose blocks wait for each other is launched so that all of them are resident:
gbmd::launch, which create, set_state, a new cell grid and the recoveries go through, passes
the cooperative attribute on.  The launch calls of the runtime are replaced on the host
(tests/host/launch_attr.cu); no GPU is used."""
import ctypes as C
import os
import subprocess

import pytest

from paper_1308_5587_gb300 import _build

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("launch") / "liblaunch_attr.so")
    # -Bsymbolic: the library's own two launch calls, not the runtime's
    subprocess.run(["nvcc", *_build.FLAGS, "-shared", "-cudart", "shared", "-Xlinker", "-Bsymbolic",
                    os.path.join(HERE, "host", "launch_attr.cu"),
                    os.path.join(_build.CSRC, "k_step.cu"), "-o", out], check=True)
    return C.CDLL(out)


@pytest.mark.parametrize("cooperative", [0, 1])
@pytest.mark.parametrize("grid,block,smem", [(1, 32, 0), (152, 768, 225280)])
def test_launch_keeps_the_cooperative_attribute(lib, cooperative, grid, block, smem):
    seen = (C.c_int * 6)()
    assert lib.launch_seen(cooperative, grid, block, smem, seen) == 0
    assert seen[0] + seen[1] == 1
    assert seen[2] == cooperative
    assert list(seen[3:]) == [grid, block, smem]
