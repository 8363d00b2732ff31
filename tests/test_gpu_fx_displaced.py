"""FP64 2D and 3D systems far from the origin, whole or in two groups (needs a GB300): the range of
the fixed-point units is taken from each unit's first row, so displaced systems keep them, and
groups far apart meet in FP64 units.  Per particle against the one-sided FP64 kernel, which
reads the same coordinates: 2 x 76 x 2^-53 of the particle's own sum of the terms' magnitudes
(12 roundings of a term and fewer than 64 additions on either side)."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu

TOL = 2 * 76 * 2.0**-53
EPS = 1e-3


def _state(dim, N, at, groups):
    x = inputs.default_state(dim, N, 3)[0].reshape(dim, N) + at
    if groups == 2:
        x[:, ::2] *= -1.0
    return x.reshape(-1)


def _sums(q, dim, v, i):
    x = q.reshape(dim, -1)
    d = x[:, i, None] - x[:, None, :]
    s = (d * d).sum(0) + EPS
    if v is None:
        return (2 if dim == 2 else 1) / x.shape[1] * (np.abs(d) / (s if dim == 2 else s**1.5)).sum(2)
    u = v.reshape(dim, -1)
    w = u[:, i, None] - u[:, None, :]
    return 2.0 / x.shape[1] * (np.sqrt((w * w).sum(0)) / s).sum(1)


@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("at", [10.0, 1e3, 1e7, 1e12])
@pytest.mark.parametrize("dim,N", [(2, 700), (2, 11_001), (3, 700), (3, 11_001)])
def test_every_particles_force(dim, N, at, groups):
    q, out = _state(dim, N, at, groups), []
    for symmetric in (1, 0):
        with System(dim, N, EPS, 0.01, 1, precision="fp64") as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.force().reshape(dim, N))
    i = np.arange(0, N, max(1, N // 400))
    assert np.all(np.abs(out[0] - out[1])[:, i] <= TOL * _sums(q, dim, None, i))


@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("at", [10.0, 1e3, 1e7])
@pytest.mark.parametrize("N", [700, 11_001])
def test_every_particles_jacobian_product(N, at, groups):
    h = 1e-40  # steps so short that every kick sees the same state
    q = _state(2, N, at, groups)
    v, out = np.random.default_rng(N).standard_normal(2 * N), []
    for symmetric in (1, 0):
        with System(2, N, EPS, h, 1, precision="fp64") as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.tangent_step(1, v, np.zeros_like(v))[1].reshape(2, N))
    i = np.arange(0, N, max(1, N // 400))
    assert np.all(np.abs(out[0] - out[1])[:, i] <= TOL * 2.4 * h * _sums(q, 2, v, i))
