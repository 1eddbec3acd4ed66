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


SOURCES = sorted(p.name for p in gpu_build.CSRC.glob("*.cu*"))


def test_polls_stand_in_bounded_loops():
    polls = 0
    for name in SOURCES:
        text = (gpu_build.CSRC / name).read_text()
        for m in re.finditer(r"if \(mbar_try\(", text):
            polls += 1
            assert re.search(r"clock64\(\) - t0 > (kWaitCycles|max_cycles)", text[m.start():m.start() + 400]), name
    assert polls


@pytest.mark.parametrize("name", SOURCES)
def test_error_words_belong_to_the_call(name):
    """No kernel writes, and no host code reads or clears, a word that calls on other streams and threads
    share: a process-wide error flag is cleared by whichever call looks first."""
    text = (gpu_build.CSRC / name).read_text()
    word = r"^(?:static\s+)?__device__\s+(?:volatile\s+)?(?:int|unsigned|uint32_t)\s+\w+\s*(?:=[^;(]*)?;"
    assert not re.findall(word, text, re.M) and "cudaMemcpyFromSymbol" not in text
