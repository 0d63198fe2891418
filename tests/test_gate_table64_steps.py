"""Host logic: the FP64 gate table (csrc/mm_gate_table64.h) at time steps from
far below a gate's time constant to far above it, where a step's factors E or
D leave the range that the table's FP32 terms hold: the gates stepped with the
table against the same step in long double."""
import subprocess

import numpy as np
import pytest

from test_gate_table64 import checker  # noqa: F401  (fixture)


@pytest.mark.parametrize("dt", [1e-300, 1e-40, 1e-34, 1e-28, 1e-12, 1.0, 3.0, 6.0, 8.0, 10.0, 20.0, 1000.0, 1e300])
def test_gate_step_at_any_time_step(checker, dt):  # noqa: F811
    """The bound of the ordinary time steps, 4 2^-53 for the roundings of X,
    x - X, the result and D, and 2 2^-53 for the interpolation of D, whose
    error of seven points is at most e^y (|y| h / tau)^7 / (2^6 7!) with h =
    0.125 mV and rates that change over tau = 10 mV or more: 2^-53 at its
    largest, y = -7, and as much again for the rates' curvature."""
    r = np.random.default_rng(4)
    c = -120.0 + 0.25 * np.arange(961)
    V = np.concatenate([np.clip(c + d, -120, 120) for d in (-0.125, -0.1, -0.03, 0.0, 0.06, 0.124)] +
                       [r.uniform(-120, 120, 3000)])
    x = r.random((len(V), 3))
    text = "\n".join("%r %r %r %r" % (float(v), *map(float, g)) for v, g in zip(V, x))
    out = subprocess.run([checker, repr(dt)], input=text, capture_output=True, text=True, check=True).stdout
    rows = np.array([l.split() for l in out.strip().splitlines()], dtype=np.longdouble)
    assert len(rows) == len(V)
    assert np.abs(rows[:, :3] - rows[:, 3:6]).max() <= 6 * 2.0 ** -53
