"""Waits of the tensor-core kernels, read from their sources.  A thread that gives up a bounded wait
leaves its role's loop for the end of the kernel, so a barrier without a bound may only join warps
that reach it on every path: the whole of the epilogue, after its loop."""
import re

import pytest

from paper_2305_06668_gb300 import build as gpu_build

EPILOGUE = {"gram64.cu": 256, "umma.cu": 128, "update64.cu": 256}  # threads


@pytest.mark.parametrize("name", EPILOGUE)
def test_named_barriers_join_the_whole_epilogue(name):
    text = (gpu_build.CSRC / name).read_text()
    found = re.findall(r"bar(?:rier)?\.sync\s+([^,;]+),\s*([^;]+);", text)
    assert found and all((i.strip(), c.strip()) == ("3", str(EPILOGUE[name])) for i, c in found), found


@pytest.mark.parametrize("name", [*EPILOGUE, "umma.cuh"])
def test_polls_stand_in_bounded_loops(name):
    text = (gpu_build.CSRC / name).read_text()
    polls = [m.start() for m in re.finditer(r"if \(mbar_try\(", text)]
    assert polls
    for at in polls:
        assert re.search(r"clock64\(\) - t0 > (kWaitCycles|max_cycles)", text[at:at + 400]), text[at:at + 400]
