"""The FP64 pair stages on the integer pipe against the oracle (needs a GB300): softenings on
both sides of the integer form's range, systems far larger and smaller than their softening
length, outliers that make single units take the FP64 tile, ragged sizes at the tile edges.

Tolerance as for every FP64 force: 1e-12 of sum_j |f_ij| per particle and component.  A
particle at a non-finite position makes every force NaN, as in the FP64 kernels."""
import numpy as np
import pytest

import oracle as ora
from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu

MODELS = {"grav2d": 2}


def _force(model, q, eps):
    N = q.size // {1: 1, 2: 2, 3: 3}[model]
    with System(model, N, eps, 0.01, 1, precision="fp64") as s:
        assert s.force_kernel == 6
        s.set_state(q, np.zeros_like(q))
        return s.force()


@pytest.mark.parametrize("eps", [1.0, 1e-3, 2.0**-28, 0.99 * 2.0**-28, 1e-12])
@pytest.mark.parametrize("N", [2, 127, 129, 513, 1025])
@pytest.mark.parametrize("model", MODELS.values())
def test_force_over_softenings(model, N, eps):
    q, _ = inputs.default_state(model, N, 50 + N)
    err = np.abs(_force(model, q, eps) - ora.force(model, q, eps))
    assert np.all(err <= 1e-12 * ora.force_abs(model, q, eps))


@pytest.mark.parametrize("scale", [1e-9, 1e-3, 30.0, 1e4, 1e7])
@pytest.mark.parametrize("model", [m for m in MODELS.values() if m > 1])
def test_force_over_scales(model, scale):
    q, _ = inputs.default_state(model, 700, 3)
    q = q * scale
    err = np.abs(_force(model, q, 1e-4) - ora.force(model, q, 1e-4))
    assert np.all(err <= 1e-12 * ora.force_abs(model, q, 1e-4))


@pytest.mark.parametrize("at", [0, 300, 1024, 1299])
@pytest.mark.parametrize("model", [m for m in MODELS.values() if m > 1])
def test_outliers_and_coincident_particles(model, at):
    N = 1300
    q, _ = inputs.default_state(model, N, 9)
    q[at] = 1e9  # beyond 2^26 sqrt(eps): its units run in FP64
    q[N + (at + 7) % N] = -1e5
    q[(at + 11) % N], q[N + (at + 11) % N] = q[(at + 12) % N], q[N + (at + 12) % N]
    err = np.abs(_force(model, q, 1e-4) - ora.force(model, q, 1e-4))
    assert np.all(err <= 1e-12 * ora.force_abs(model, q, 1e-4))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("model", [m for m in MODELS.values() if m > 1])
def test_a_non_finite_position_reaches_every_force(model, bad):
    q, _ = inputs.default_state(model, 1100, 9)
    q[600] = bad
    assert np.isnan(_force(model, q, 1e-3)).all()
