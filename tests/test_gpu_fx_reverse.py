"""Precision of the FP64 2D reverse and tangent stages on the integer pipe, particle by particle,
in systems wide against their softening length and for tangents of uneven sizes (needs a
GB300).  Both sides are FP64 forms: the one-sided kernel (symmetric = 0) and the default.  A
term of either is within 12 roundings of |w| / s (J v) or |d| / s^2 (df/deps), a particle's sum
passes through fewer than 64 additions of comparable partial sums: 2 x 76 x 2^-53 of the
particle's own sum of the terms' magnitudes.  Steps are so short that every kick of a step
sees the same state; the kicks' coefficients sum to less than 2.4."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu

H, KICKS, TOL = 1e-6, 2.4, 2 * 76 * 2.0**-53

# (N, R, eps): extents of 2^5 to 2^25 softening lengths; coordinates on both sides of 2^9
SYSTEMS = [(1024, 1.0, 1e-3), (1024, 1.0, 1e-6), (1024, 1.0, 1e-8), (1024, 10.0, 1e-8), (1024, 1000.0, 1e-4), (700, 3000.0, 1e-8),
           (12_001, 1.0, 1e-3), (12_001, 0.6, 1e-6)]

TANGENTS = {
    "random": lambda g, n: g.standard_normal(n),
    "one outlier": lambda g, n: np.where(np.arange(n) == 5, 1.0, 1e-10 * g.standard_normal(n)),
    "a translation": lambda g, n: 1.0 + 1e-10 * g.standard_normal(n),
    "wide range": lambda g, n: np.exp(10 * g.standard_normal(n)),
    "equal": lambda g, n: np.full(n, 0.3),
    "equal and huge": lambda g, n: np.full(n, 2.0**1000),
}


def _sums(q, v, eps):
    """Per particle: sum_j |v_i - v_j| / s_ij."""
    x, u = q.reshape(2, -1), v.reshape(2, -1)
    out = np.zeros(x.shape[1])
    for i in range(0, out.size, 250):
        d, w = x[:, i : i + 250, None] - x[:, None, :], u[:, i : i + 250, None] - u[:, None, :]
        out[i : i + 250] = (np.sqrt((w * w).sum(0)) / ((d * d).sum(0) + eps)).sum(1)
    return out


@pytest.mark.parametrize("kind", TANGENTS)
@pytest.mark.parametrize("N,R,eps", SYSTEMS)
def test_every_particles_jacobian_product(N, R, eps, kind):
    q = R * inputs.default_state(2, N, 3)[0]
    v, out = TANGENTS[kind](np.random.default_rng(N), 2 * N), []
    for symmetric in (1, 0):
        with System(2, N, eps, H, 1, precision="fp64") as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.tangent_step(1, v, np.zeros_like(v))[1].reshape(2, N))
    if kind.startswith("equal"):  # zero; NaN where d.w overflows in padding, in both forms
        assert np.array_equal(out[0], out[1], equal_nan=True)
        return
    tol = TOL * KICKS * H * 2.0 / N * _sums(q, v, eps)
    assert np.all(np.abs(out[0] - out[1]) <= tol)


@pytest.mark.parametrize("N,R,eps", [s for s in SYSTEMS if s[0] < 10_000])
def test_every_particles_derivative_by_eps(N, R, eps):
    """With one particle k moving in one direction c, d(kinetic energy)/d eps is its own
    (df/deps)_c times the kicks."""
    q = R * inputs.default_state(2, N, 3)[0]
    x = q.reshape(2, N)
    for n, k in enumerate([0, 63, 64, 128, 600, N - 1]):
        c, p, out = n % 2, np.zeros_like(q), []
        p[c * N + k] = 1.0
        for symmetric in (1, 0):
            with System(2, N, eps, H, 1, precision="fp64") as s:
                s.set_tuning("symmetric", symmetric)
                s.set_state(q, p)
                out.append(s.grad(1, 0)[3])
        d = x[:, k : k + 1] - x
        s2 = ((d * d).sum(0) + eps) ** 2
        # the moving particle's own terms, and its displacement's effect on the others' lambda
        assert abs(out[0] - out[1]) <= TOL * KICKS * H * 2.0 / N * (np.abs(d) / s2).sum()
