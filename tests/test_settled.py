"""The rule by which a dual of the scaling form counts as settled (csrc/settled.h), compiled for the host: a cycle of rounding
ends the loop, steps that all lead one way do not, however small."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_00392_b200", "csrc")


@pytest.fixture(scope="module")
def settles_at(tmp_path_factory):
    """Iteration at which a sequence of values (steps in units in the last place, from `start`) settles, or None."""
    d = tmp_path_factory.mktemp("settled")
    src = d / "settled.cpp"
    src.write_text('#include "%s"\nextern "C" int settled(int a, int b, int c) { return rtp::dual_settled(a, b, c); }\n'
                   % os.path.join(CSRC, "settled.h"))
    lib = str(d / "settled.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-o", lib, str(src)], check=True)
    fn = ctypes.CDLL(lib).settled

    def run(steps, start):
        v = int(np.float32(start).view(np.int32)) + np.cumsum([0] + list(steps))
        for t in range(1, len(v)):
            if fn(int(v[t]), int(v[t - 1]), int(v[t - 2]) if t > 1 else 0):
                return t
        return None
    return run


@pytest.mark.parametrize("start", [1.0, 0.99999988, 3.7e-20, 6.0e17])
def test_a_cycle_settles_and_a_drift_does_not(settles_at, start):
    for step in (2, 3, 4, -2, -3, -4, 5, 100):
        assert settles_at([step] * 60, start) is None                   # always the same way
    for swing in (2, 3, 4):
        assert settles_at([90, 40, 9] + [swing, -swing] * 4, start) == 5          # a cycle of two values
        assert settles_at([90, 40, 9] + [swing, 1 - swing] * 4, start) == 5       # that moves by a unit in two
    assert settles_at([5, -5] * 30, start) is None                     # wider than rounding goes
    assert settles_at([7, 1], start) == 2 and settles_at([7, 0], start) == 2 and settles_at([-9, -1], start) == 2
