"""The kernels' 32-bit indices over a level's pair lists never wrap (CPU): a loop that steps past the end of a list of
2^32 - 1 pairs would come back to its start and never end."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1909_05600_gb300", "csrc")
CONST = {"P2P_T": 128}


def _read(name):
    with open(os.path.join(CSRC, name)) as f:
        return f.read()


MAX_LISTED = int(re.search(r"MAX_LISTED = (0x[0-9a-f]+)ll;", _read("ffm_internal.cuh")).group(1), 16)


def _loops():
    """(file, variable, step) of every 32-bit loop over a pair list."""
    out = []
    for name in ("tree.cu", "transfer.cu", "nearfield.cu", "farfield.cu"):
        for v, step in re.findall(r"for \(uint32_t (e[bg]?) = [^;]*; e[bg]? < [^;]*; (?:e[bg]? \+= (\w+)|\+\+e)\)", _read(name)):
            out.append((name, v, 1 if not step else CONST[step] if step in CONST else int(step)))
    return sorted(set(out))


def test_loops_are_found():
    steps = {(f, s) for f, _, s in _loops()}
    assert {("tree.cu", 32), ("tree.cu", 256), ("nearfield.cu", 128), ("transfer.cu", 32)} <= steps


@pytest.mark.parametrize("name,var,step", _loops())
def test_index_stays_past_the_end(name, var, step):
    # lane + step past the last index, as the kernels add them in 32 bits
    for end in (MAX_LISTED, MAX_LISTED - 1, MAX_LISTED - step + 1):
        last = end - 1
        assert (last + step) % 2 ** 32 >= end, "the index wraps to the start of the list"
        assert (last + step + 31) % 2 ** 32 >= end


def test_tiles_stay_past_the_end():
    # tiles of up to 256 pairs start inside the list and compare their pairs' indices with its end
    assert MAX_LISTED - 1 + 256 < 2 ** 32
