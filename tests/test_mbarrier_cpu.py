"""The order that a tile's mbarrier needs, read from the kernels' source: lane 0 initialises it, and the
whole warp passes a barrier before any lane polls it.  Without that barrier the other lanes may poll a
word that is not initialised, or one that an earlier block left behind as complete, and nothing orders
what they then read after the copy.  (Which lanes run first is the hardware's choice, so that a run on
a device shows nothing either way.)"""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1211_7275_gb300", "csrc")


def _code(path):
    with open(path) as fh:
        return re.sub(r"//[^\n]*", "", fh.read())


def _block_end(code, at):
    """End of the innermost braces around position `at`."""
    depth = 0
    for k in range(at, len(code)):
        if code[k] == "{":
            depth += 1
        elif code[k] == "}":
            depth -= 1
            if depth < 0:
                return k
    raise AssertionError("unbalanced braces")


def _inits():
    out = []
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        code = _code(path)
        out += [pytest.param(code, m.start(), id=f"{os.path.basename(path)}-{n}")
                for n, m in enumerate(re.finditer(r"\bmbar_init\(", code))]
    return out


def test_the_kernels_use_mbarriers():
    assert len(_inits()) >= 2


@pytest.mark.parametrize("code,at", _inits())
def test_warp_barrier_between_initialisation_and_first_wait(code, at):
    end = _block_end(code, at)   # of the one lane's block
    wait = re.search(r"\bmbar_wait\(", code[end:])
    assert wait, "an initialised barrier that nothing waits for"
    assert "mbar_wait(" not in code[at:end], "the initialising lane waits before the others may"
    assert "__syncwarp()" in code[end:end + wait.start()]
