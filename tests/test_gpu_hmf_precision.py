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


@pytest.mark.parametrize("steps", [0, 1, 9])
@pytest.mark.parametrize("extent", [1e-12, 1e-6, 1e-3, 0.02])
@pytest.mark.parametrize("N", [2, 3, 1000, 50_000])
def test_forces_of_cold_systems(N, extent, steps):
    """All angles near 0, where doubles have more bits than fixed-point numbers: forces at the
    given state and after steps (in one launch for the smaller N) against long double, within 76
    roundings (12 of a term, 64 of the sums) of |cos t_i| mean|sin| + |sin t_i| mean|cos|.  The
    stages' table-driven sine rounds its term r^3 / 6 to FP32, |r| the smaller of the angle and half
    a table step: 2^-23 of it for the particle's sine and for the mean's.  Systems that are not so
    cold (|M| below 1 - 2^-24) stay in fixed point, whose sums round each sine to 2^-55."""
    g = np.random.default_rng(N)
    with System(0, N, 0.0, 0.1, 1, precision="fp64") as s:
        s.set_state(extent * (2 * g.random(N) - 1), np.zeros(N))
        s.step(steps)
        q = s.get_state()[0]
        f = s.force()
    t = q.astype(np.longdouble)
    sn, cs = np.sin(t), np.cos(t)
    want = cs * sn.mean() - sn * cs.mean()
    scale = (np.abs(cs) * np.abs(sn).mean() + np.abs(sn) * np.abs(cs).mean()).astype(np.float64)
    r = min(float(np.abs(t).max()), np.pi / 4096)
    scale += (cs.mean() < 1 - 2.0**-24) * 2.0**-55 / (76 * 2.0**-53)
    assert np.all(np.abs((f - want).astype(np.float64)) <= 76 * 2.0**-53 * scale + (steps > 0) * 2 * 2.0**-23 * r**3 / 6)


def test_a_system_that_becomes_cold_and_warm_again():
    """Angles within 1e-3 swing through 0 in a quarter period of 15.7 steps: the stages change from
    fixed point to doubles and back, launched and in one launch alike (the same bits), and the
    forces stay within 2^-54 + 76 x 2^-53 x 1e-3 of long double (fixed point: sums to 2^-55,
    products to 2^-59; doubles: the sine's term r^3 / 6 to 2^-23, twice)."""
    N = 3000
    q = 1e-3 * (2 * np.random.default_rng(1).random(N) - 1)
    cold = []
    for n in range(0, 33, 4):
        out = []
        for graphs in (1, 0):
            with System(0, N, 0.0, 0.1, 1, precision="fp64") as s:
                s.set_tuning("step_graphs", graphs)
                s.set_state(q, np.zeros(N))
                s.step(n)
                out.append((s.get_state()[0], s.force()))
        assert all(np.array_equal(a, b) for a, b in zip(*out))
        t = out[0][0].astype(np.longdouble)
        sn, cs = np.sin(t), np.cos(t)
        cold.append(cs.mean() > 1 - 2.0**-24)
        assert np.all(np.abs(out[0][1] - (cs * sn.mean() - sn * cs.mean())) <= 2.0**-54 + 76 * 2.0**-53 * 1e-3)
    assert not cold[0] and any(cold) and not cold[-1]
