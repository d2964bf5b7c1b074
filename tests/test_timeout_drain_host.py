"""Kernels that feed shared memory by bulk copies leave after a timed-out wait
only once the copies in flight have been waited for again: the shared memory
of a block that has left may belong to another one.  Checked in the sources
(a wait that runs out is not provoked on a GPU)."""
import pathlib
import re

import pytest

CSRC = pathlib.Path(__file__).resolve().parent.parent / "paper_2310_16214_gb300" / "csrc"


def _block(text, start):
    """The braced block that opens at or after `start`, or the single statement there."""
    i = start
    while text[i] in " \n":
        i += 1
    if text[i] != "{":
        return text[i:text.index(";", i) + 1]
    depth, j = 0, i
    while True:
        depth += {"{": 1, "}": -1}.get(text[j], 0)
        j += 1
        if depth == 0:
            return text[i:j]


def _bulk_copy_files():
    return sorted(p.name for p in CSRC.glob("*.cu") if "tma_load_1d(" in p.read_text())


def test_files_found():
    assert {"fft.cu", "tridiag.cu", "tridiag_wm.cu"} <= set(_bulk_copy_files())


@pytest.mark.parametrize("name", _bulk_copy_files())
def test_block_drains_its_copies_before_leaving(name):
    text = re.sub(r"//[^\n]*", "", (CSRC / name).read_text())
    # every test of a block-wide vote on a bounded wait
    tests = list(re.finditer(r"if \(!(?:ok|__syncthreads_and\((?:[^()]|\([^()]*\))*\))\)", text))
    assert tests, "no vote on a bounded wait found"
    for m in tests:
        body = _block(text, m.end())
        if "return" in body:
            # either it waits again before it leaves, or the wait voted on is the one
            # whose leader waits twice as long
            again = "mbar_wait_bounded" in body[:body.index("return")]
            waits = re.findall(r"mbar_wait_(?:bounded|block)\(", text[:m.start()] + m.group())
            assert again or waits[-1] == "mbar_wait_block(", "%s: %s" % (name, body)


def test_the_leader_waits_longer():
    text = (CSRC / "tma.cuh").read_text()
    assert re.search(r"bool mbar_wait_block\([^)]*bool leader\) \{\s*return mbar_wait_bounded\(bar, parity, "
                     r"leader \? 2 \* kWaitLimitCycles : kWaitLimitCycles\);", text)
