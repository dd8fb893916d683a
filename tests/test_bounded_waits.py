"""Device waits of the tensor-core kernels, by reading their source: a wait that gives up cannot be made
to happen on a GPU without holding it up."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1510_04686_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as fh:
        return re.sub(r"//[^\n]*", lambda m: m.group(0) if "----" in m.group(0) else "", fh.read())


@pytest.mark.parametrize("name", ["crt_gemm.cu", "tc_gemm.cu"])
def test_a_warp_gives_up_as_a_whole(name):
    """The epilogue warps run instructions of the whole warp after each wait, so all lanes of one take
    the same answer; the single elected threads of the other roles wait for themselves."""
    roles, epilogue = _code(name).split("// ---------------- epilogue", 1)
    epilogue = epilogue.split("tcgen05.dealloc", 1)[0]
    assert len(re.findall(r"\bmbar_wait_warp\(", epilogue)) >= 1
    assert not re.search(r"\bmbar_wait\(", epilogue)
    assert not re.search(r"=\s*!\*abort_flag", epilogue)
    waits = [m.start() for m in re.finditer(r"\bmbar_wait\(", roles)]
    assert waits and min(waits) > roles.index("elect_one()")
    assert re.search(r"mbar_wait_warp\([^{]*\{\s*return __all_sync\(0xffffffffu, mbar_wait\(",
                     _code("tc_common.cuh"))


@pytest.mark.parametrize("name", ["crt_gemm.cu", "tc_gemm.cu"])
def test_copies_in_flight_land_before_memory_is_released(name):
    """After the last wait of any role and a barrier, all threads give loads and MMAs in flight time to
    land when a wait gave up; only then the CTA (or the pair) frees tensor memory and leaves."""
    tail = _code(name).split("// ---------------- epilogue", 1)[1]
    tail = tail[:tail.index("tcgen05.dealloc")]
    last = tail[tail.rindex("mbar_wait"):]
    assert re.search(r"__syncthreads\(\);\s*land_in_flight\(abort_flag\);", last)
    assert "cluster_sync();" not in last.split("land_in_flight", 1)[0]
