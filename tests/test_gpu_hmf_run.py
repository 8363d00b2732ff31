"""Small HMF systems take all stages of md_step in one cluster launch: states equal those of the
launched stages (step_graphs = 0) bit for bit, over sizes from one particle to past the
largest cluster (16 CTAs), odd ones among them, and step counts that end inside and after
blocks of eight (needs a GB300)."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("N", [1, 2, 3, 511, 1025, 4097, 10_007, 16_379, 16_380, 16_381, 16_385, 20_000])
@pytest.mark.parametrize("n", [1, 2, 9, 27])
def test_one_launch_equals_launched_stages(N, prec, n):
    q, p = inputs.default_state(0, N, 5)
    out, launches = [], []
    for graphs in (1, 0):
        with System(0, N, 0.0, 0.1, 1, precision=prec) as s:
            s.set_tuning("step_graphs", graphs)
            s.set_state(q, p)
            s.step(n)
            launches.append(s.launch_count)
            out.append(s.get_state() + (s.force(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    if N <= 16_379 and n > 1:
        assert launches[0] < launches[1]


def test_more_steps_than_one_launch_holds():
    q, p = inputs.default_state(0, 700, 5)
    out = []
    for graphs in (1, 0):
        with System(0, 700, 0.0, 0.01, 1, precision="mixed") as s:
            s.set_tuning("step_graphs", graphs)
            s.set_state(q, p)
            s.step(601)
            out.append(s.get_state())
    for a, b in zip(*out):
        assert np.array_equal(a, b)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("N", [2, 1025, 10_007])
@pytest.mark.parametrize("speed", [1e7, 1e12, 1e36, 1.7e308, np.inf, np.nan])
def test_angles_beyond_any_range(N, prec, speed):
    """One particle's speed drives its angle out of the FP32 reduction's range, or to infinity:
    the other particles feel what they feel in the launched stages."""
    q, p = inputs.default_state(0, N, 5)
    p[N // 2] = speed
    out = []
    for graphs in (1, 0):
        with System(0, N, 0.0, 10.0, 1, precision=prec) as s:
            s.set_tuning("step_graphs", graphs)
            s.set_state(q, p)
            s.step(1)
            out.append(s.get_state())
    for a, b in zip(*out):
        assert np.array_equal(a, b, equal_nan=True)
    if prec == "fp64" and not abs(speed) < 1e308:  # a sum with a non-finite angle is NaN
        assert np.all(np.isnan(out[0][1]))
