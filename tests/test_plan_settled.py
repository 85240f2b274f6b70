"""The rule by which an iteration of the scaling form counts as settled up to a common factor (csrc/settled.h), compiled for
the host: a factor that all columns share ends the loop, a column that moves against the others by more than 2^-22 of its value
(two or three units in the last place, by its mantissa) does not."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_00392_b200", "csrc")


@pytest.fixture(scope="module")
def settled(tmp_path_factory):
    d = tmp_path_factory.mktemp("plan_settled")
    src = d / "plan_settled.cpp"
    src.write_text('#include "%s"\nextern "C" int settled(float lo, float hi) { return rtp::plan_settled(lo, hi); }\n'
                   % os.path.join(CSRC, "settled.h"))
    lib = str(d / "plan_settled.so")
    subprocess.run(["g++", "-shared", "-fPIC", "-o", lib, str(src)], check=True)
    fn = ctypes.CDLL(lib).settled
    fn.argtypes = [ctypes.c_float, ctypes.c_float]

    def run(now, last):
        rel = (now - last) / last                     # float32, as the kernels take it
        return bool(fn(float(rel.min()), float(rel.max())))
    run.rule = lambda lo, hi: bool(fn(lo, hi))
    return run


def test_columns_that_are_not_a_number_leave_it_to_the_rule_for_single_duals(settled):
    assert not settled.rule(float("nan"), float("nan"))
    assert settled.rule(0.0, 0.0) and settled.rule(-1e-7, 1e-7) and not settled.rule(-1e-6, 1e-6)


@pytest.mark.parametrize("columns", [2, 17, 640])
def test_a_common_factor_settles_and_a_column_that_drifts_does_not(settled, columns):
    rng = np.random.default_rng(columns)
    last = np.exp(rng.uniform(-20, 20, columns)).astype(np.float32)
    unit = np.float32(2.0 ** -23)
    assert settled(last, last)
    for c in (1, 3, 50, -50):                         # rounding a common factor moves a column by half a unit at most
        now = (last.astype(np.float64) * (1.0 + c * 2.0 ** -23)).astype(np.float32)
        assert settled(now, last), c
    for sign in (1, -1):
        one = last.copy()
        one[-1] = np.nextafter(last[-1], np.float32(np.inf * sign))
        assert settled(one, last)                     # a unit in the last place
        for steps in (3, 4, 20):                      # more than two units of 2^-23 against the others
            far = last.copy()
            far[0] = last[0] * (1 + sign * steps * unit)
            assert not settled(far, last), (sign, steps)


@pytest.mark.parametrize("mantissa,most", [(1.0, 2), (1.25, 2), (1.5, 3), (1.99999, 3)])
def test_how_far_one_column_may_move_alone(settled, mantissa, most):
    for scale in (2.0 ** -30, 1.0, 2.0 ** 40):
        last = np.array([1.0, mantissa * scale, 3.0], np.float32)
        for ulps in range(1, 6):
            now = last.copy()
            now.view(np.int32)[1] += ulps
            assert settled(now, last) == (ulps <= most), (scale, ulps)
