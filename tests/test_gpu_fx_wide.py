"""FP64 2D and 3D forces on the integer pipe in systems that are wide against their softening
length, up to the largest coordinates that the fixed-point units take (needs a GB300).
Against a long-double sum of the definition: a term is within 8 roundings (its coordinate
differences, their squares, the power, the product, the unit), and a sum passes through fewer
than 30 FP64 additions (segments and column partials of 1,024 particles), 38 x 2^-53 of the
sum of the terms' magnitudes per particle and component."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu


def _force(dim, q, eps):
    """(f, sum of |terms|) in long double."""
    x = q.reshape(dim, -1).astype(np.longdouble)
    N = x.shape[1]
    f, a = np.zeros_like(x), np.zeros_like(x)
    for i in range(N):
        d = x[:, i : i + 1] - x
        s = (d * d).sum(0) + np.longdouble(eps)
        t = d / s if dim == 2 else d / (s * np.sqrt(s))
        f[:, i], a[:, i] = -t.sum(1), np.abs(t).sum(1)
    scale = np.longdouble(2 if dim == 2 else 1) / N
    return f * scale, (a * scale).astype(np.float64)


@pytest.mark.parametrize("dim,R,eps", [(2, 1.0, 1e-3), (2, 1000.0, 1e-8), (2, 4000.0, 1e-8), (3, 1.0, 1e-4), (3, 1.0, 1e-8), (3, 30.0, 1e-6)])
def test_forces_of_wide_systems(dim, R, eps):
    N = 1024
    q = (inputs.default_state(2, N, 3)[0] if dim == 2 else inputs.ball_state(N, 3)[0]) * R
    with System(dim, N, eps, 0.01, 1, precision="fp64") as s:
        s.set_state(q, np.zeros_like(q))
        f = s.force().reshape(dim, N)
    want, scale = _force(dim, q, eps)
    assert np.all(np.abs(f - want) <= 38 * 2.0**-53 * scale)
