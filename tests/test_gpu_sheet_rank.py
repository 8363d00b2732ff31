"""Unsoftened sheets by rank counts against the pair kernel that compares every ordered pair
(symmetric = 0; needs a GB300): the counts are whole numbers, so forces and states are equal
bit for bit, over the sorted tiles' edges (8192 FP32 keys, 4096 FP64 keys), runs of equal
positions, signed zeros, infinities and NaN."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu


def _both(q, p, prec, steps=0):
    out = []
    for symmetric in (1, 0):
        with System(4, q.size, 0.0, 0.01, 1, precision=prec) as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, p)
            s.step(steps)
            out.append((s.force(),) + s.get_state())
    return out


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("N", [1, 2, 4095, 4096, 4097, 8191, 8192, 8193, 20_001, 100_003])
def test_ranks_equal_pair_counts(N, prec):
    q, p = inputs.sheet_state(N, N)
    for a, b in zip(*_both(q, p, prec)):
        assert a.tobytes() == b.tobytes()


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_steps_equal(prec):
    q, p = inputs.sheet_state(9001, 3)
    for a, b in zip(*_both(q, p, prec, steps=12)):
        assert a.tobytes() == b.tobytes()


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("N", [700, 9001])
def test_ties_zeros_and_non_finite_positions(N, prec):
    q, p = inputs.sheet_state(N, 4)
    q = np.round(q * 50) / 50  # about 100 values: long runs of equal positions
    q[5::97], q[6::97] = 0.0, -0.0
    q[11], q[200], q[N - 3] = np.inf, -np.inf, np.inf
    q[50], q[N - 1] = np.nan, -np.nan
    q[70], q[71] = 1e300, 1.1e300  # both infinite in FP32
    for a, b in zip(*_both(q, p, prec)):
        assert np.array_equal(a, b, equal_nan=True)


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
def test_all_particles_at_one_place(prec):
    f = _both(np.full(9001, 0.25), np.zeros(9001), prec)[0][0]
    assert not f.any()
