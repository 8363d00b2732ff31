"""FP64 Ring forces of clusters near theta = 0 and pi, where sines are held to more than the
fixed-point units' 2^-62 (needs a GB300): per particle against the one-sided FP64 kernel,
which reads the same records.  A term of either is within 12 roundings, a sum passes through
fewer than 64 additions of comparable partial sums: 2 x 76 x 2^-53 of the particle's own sum of
the terms' magnitudes."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System

pytestmark = pytest.mark.gpu

N = 1500


def _cluster(g, extent, at=0.0):
    return at + extent * (2 * g.random(N) - 1)


STATES = {
    "1e-6": lambda g: _cluster(g, 1e-6),
    "1e-3": lambda g: _cluster(g, 1e-3),
    "0.03": lambda g: _cluster(g, 0.03),
    "at pi": lambda g: _cluster(g, 1e-6, np.pi),
    "whole turns apart": lambda g: _cluster(g, 1e-6) + 2 * np.pi * (np.arange(N) % 3),
    "a third elsewhere": lambda g: np.where(np.arange(N) % 3 == 0, 3 * g.random(N) - 1.5, _cluster(g, 1e-6)),
    "one elsewhere": lambda g: np.where(np.arange(N) == 700, 1.0, _cluster(g, 1e-6)),
    "spread": lambda g: np.pi * (2 * g.random(N) - 1),
}


@pytest.mark.parametrize("n", [N, 12_000])
@pytest.mark.parametrize("eps", [2.0**-17, 1e-3, 1.0])
@pytest.mark.parametrize("kind", STATES)
def test_every_particles_force(kind, eps, n):
    q = np.resize(STATES[kind](np.random.default_rng(7)), n) * (1 + np.arange(n) // N * 2.0**-20)
    out = []
    for symmetric in (1, 0):
        with System(1, n, eps, 0.01, 1, precision="fp64") as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.force())
    # sin theta as the records hold it, rounded at 2^-53 of itself: S_ij and its rounding
    s, c, a, b = np.sin(q), np.cos(q), np.sin(0.5 * q), np.cos(0.5 * q)
    i = np.arange(0, n, max(1, n // 500))
    S = np.abs(s[i, None]) * np.abs(c) + np.abs(c[i, None]) * np.abs(s)
    h = a[i, None] * b - b[i, None] * a
    H = np.abs(a[i, None] * b) + np.abs(b[i, None] * a)
    dd = h * h + 0.5 * eps
    tol = (S * dd**-1.5 * (1 + 3 * H * np.abs(h) / dd)).sum(1)
    assert np.all(np.abs(out[0] - out[1])[i] <= 2 * 76 * 2.0**-53 * tol / (8 * n))
