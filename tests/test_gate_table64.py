"""Host logic: the FP64 gate table (csrc/mm_gate_table64.h), evaluated as the
kernel evaluates it, against the same exponential-Euler step in long double and
against the step with the rates evaluated directly in double."""
import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2005_06332_gb300", "csrc")


@pytest.fixture(scope="module")
def checker(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("gtab64") / "gate_table64_check")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-I" + CSRC,
                    os.path.join(ROOT, "tests", "gate_table64_check.cpp"), "-o", out], check=True)
    return out


@pytest.mark.parametrize("dt", [0.001, 0.025, 0.1])
def test_gate_step_is_no_less_accurate_than_the_rates(checker, dt):
    """Interval centres and both ends of every interval, the ends of the
    table, the removable singularities and random voltages; gates anywhere in
    [0, 1] and close to their steady state.  The table's error is at most the
    direct evaluation's, at the worst point and in the root mean square."""
    r = np.random.default_rng(3)
    c = -120.0 + 0.25 * np.arange(961)
    V = np.concatenate([c, np.clip(c - 0.125, -120, 120), np.clip(np.nextafter(c + 0.125, -200), -120, 120),
                        [-40.0, -55.0, np.nextafter(-40.0, 0), np.nextafter(-55.0, -60), 120.0, -120.0, 0.0, -0.0, 5e-324],
                        r.uniform(-120, 120, 4000), r.normal(-65, 5, 4000)])
    V = np.clip(V, -120.0, 120.0)
    x = r.random((len(V), 3))
    text = "\n".join("%r %r %r %r" % (float(v), *map(float, g)) for v, g in zip(V, x))
    out = subprocess.run([checker, repr(dt)], input=text, capture_output=True, text=True, check=True).stdout
    rows = np.array([l.split() for l in out.strip().splitlines()], dtype=np.longdouble)
    assert len(rows) == len(V)
    table, exact, direct = rows[:, :3], rows[:, 3:6], rows[:, 6:]
    et, ed = np.abs(table - exact), np.abs(direct - exact)
    assert np.all(et.max(axis=0) <= ed.max(axis=0)), (et.max(axis=0), ed.max(axis=0))
    assert np.all(np.sqrt((et ** 2).mean(axis=0)) <= np.sqrt((ed ** 2).mean(axis=0)))
    # one rounding of X, one of x - X, one of the result, all below 2^-53 for gates in [0, 1], and D's relative error
    assert et.max() < 4 * 2.0 ** -53
