"""Unsoftened sheets by rank counts over every tile shape (needs a GB300): 2,048 keys up to
N = 32,768, 4,096 above, 8,192 for FP32 above 131,072, and one, two and four particles per
thread (152 SMs: up to 155,648 and 311,296).  Forces equal those of the pair kernel that
compares every ordered pair (symmetric = 0) bit for bit, with runs of equal positions,
signed zeros, infinities and NaN as well."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu


def _forces(q, prec):
    out = []
    for symmetric in (1, 0):
        with System(4, q.size, 0.0, 0.01, 1, precision=prec) as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.force())
    return out


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("N", [2047, 2048, 2049, 32_768, 32_769, 131_072, 131_073, 160_001, 320_001])
def test_ranks_equal_pair_counts(N, prec):
    a, b = _forces(inputs.sheet_state(N, N)[0], prec)
    assert a.tobytes() == b.tobytes()


@pytest.mark.parametrize("prec", ["mixed", "fp64"])
@pytest.mark.parametrize("N", [40_001, 140_001, 320_001])
def test_ties_zeros_and_non_finite_positions(N, prec):
    q = inputs.sheet_state(N, 4)[0]
    q = np.round(q * 50) / 50
    q[5::97], q[6::97] = 0.0, -0.0
    q[11], q[200], q[N - 3] = np.inf, -np.inf, np.inf
    q[50], q[N - 1] = np.nan, -np.nan
    q[8191], q[8192] = 1e300, 1.1e300
    a, b = _forces(q, prec)
    assert np.array_equal(a, b, equal_nan=True)
