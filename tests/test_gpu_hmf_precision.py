"""Precision of the FP64 HMF forces where the magnetization is small (needs a GB300)."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kick", [0, 1])
@pytest.mark.parametrize("size", [1.0, 1e-3, 1e-6, 1e-9, 1e-12])
def test_forces_keep_their_bits_with_a_small_magnetization(size, kick):
    """f_i = cos(t_i) My - sin(t_i) Mx with one (Mx, My), whatever its size: the residual of the
    best such pair is within the roundings of the sine, the cosine, a product, the FMA and M,
    5 x 2^-53 |M| (the angles' sines and cosines in long double).  After a step (kick = 1), the
    same of the forces at the new angles."""
    N = 2000
    q = 2 * np.pi * np.arange(N) / N
    q = q - size * np.sin(q)  # |M| about size / 2
    with System(0, N, 0.0, 0.1, 1, precision="fp64") as s:
        s.set_state(q, np.zeros(N))
        s.step(kick)
        q = s.get_state()[0]
        f = s.force().astype(np.longdouble)
    t = q.astype(np.longdouble)
    A = np.stack([-np.sin(t), np.cos(t)], 1)
    # normal equations in long double: sines and cosines of spread angles, nearly orthogonal
    g, r = A.T @ A, A.T @ f
    det = g[0, 0] * g[1, 1] - g[0, 1] * g[1, 0]
    m = np.array([(g[1, 1] * r[0] - g[0, 1] * r[1]) / det, (g[0, 0] * r[1] - g[1, 0] * r[0]) / det])
    size = float(np.hypot(*m.astype(float)))
    assert size > 0
    assert float(np.abs(A @ m - f).max()) <= 5 * 2.0**-53 * size
