"""The FP64 pair stages and potentials on the integer pipe (needs a GB300): softenings on both
sides of the integer form's range, systems far larger and smaller than their softening
length, outliers that make single units take the FP64 tile, ragged sizes at the tile edges.

2D and 3D forces against the oracle, 1e-12 of sum_j |f_ij| per particle and component.

Ring forces against the one-sided FP64 kernel, which reads the same records (the rounding
of their sines and cosines, common to both, is what limits the FP64 Ring force against the
oracle where particles come closer than sqrt(eps)): that kernel rounds S and sin(d/2) to
2^-53 each (product and FMA), which moves a pair's term S dd^(-3/2) by at most
2^-52 (dd^(-3/2) + 3 |S sin(d/2)| dd^(-5/2)), and its sums and products by 1e-14 of their
magnitude.

Potentials against a long-double sum of the definition, 1e-13 of the sum of the terms'
magnitudes (the oracle adds the pairs one by one in FP64, which costs more than that where
all terms are nearly equal)."""
import numpy as np
import pytest

import oracle as ora
from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu

PLANAR = [2, 3]


def _force(model, q, eps, symmetric=1):
    D = model if model > 1 else 1
    with System(model, q.size // D, eps, 0.01, 1, precision="fp64") as s:
        s.set_tuning("symmetric", symmetric)
        assert s.force_kernel == (6 if symmetric else 1)
        s.set_state(q, np.zeros_like(q))
        return s.force()


def _bound(model, q, eps):
    return 1e-12 * ora.force_abs(model, q, eps)


@pytest.mark.parametrize("eps", [1.0, 1e-3, 2.0**-28, 0.99 * 2.0**-28, 1e-12])
@pytest.mark.parametrize("N", [2, 63, 65, 127, 129, 513, 1025])
@pytest.mark.parametrize("model", PLANAR)
def test_force_over_softenings(model, N, eps):
    q, _ = inputs.default_state(model, N, 50 + N)
    assert np.all(np.abs(_force(model, q, eps) - ora.force(model, q, eps)) <= _bound(model, q, eps))


@pytest.mark.parametrize("eps", [4.1, 4.0, 1e-3, 2.0**-17, 0.99 * 2.0**-17])
@pytest.mark.parametrize("N", [1, 2, 127, 129, 513, 1025])
def test_ring_force_over_softenings(N, eps):
    q, _ = inputs.default_state(1, N, 50 + N)
    if N > 500:
        q[7] = q[400]  # coincident particles
    d = q[:, None] - q
    S, sh = np.abs(np.sin(d)), np.abs(np.sin(0.5 * d))
    dd = sh * sh + 0.5 * eps
    tol = (2.0**-52 * (dd**-1.5 + 3 * S * sh * dd**-2.5) + 1e-14 * S * dd**-1.5).sum(1) / (8 * N)
    assert np.all(np.abs(_force(1, q, eps) - _force(1, q, eps, 0)) <= tol)


@pytest.mark.parametrize("N", [9_999, 10_000, 10_001, 262_144, 262_145])
@pytest.mark.parametrize("model", [1] + PLANAR)
def test_force_at_the_kernel_shapes_edges(model, N):
    """Sampled rows on both sides of the sizes where the tile shape changes."""
    q, _ = inputs.default_state(model, N, 50)
    f = _force(model, q, 1e-3).reshape(-1, N)
    rows = np.unique(np.concatenate([[0, 63, 64, 127, 128, N - 1], np.linspace(0, N - 1, 20).astype(np.int64)]))
    fo, scale = ora.force_rows(model, q, rows, 1e-3, True)
    assert np.all(np.abs(f[:, rows] - fo) <= 1e-12 * scale)


@pytest.mark.parametrize("scale", [1e-9, 1e-3, 30.0, 1e4, 1e7])
@pytest.mark.parametrize("model", PLANAR)
def test_force_over_scales(model, scale):
    q, _ = inputs.default_state(model, 700, 3)
    q = q * scale
    assert np.all(np.abs(_force(model, q, 1e-4) - ora.force(model, q, 1e-4)) <= _bound(model, q, 1e-4))


@pytest.mark.parametrize("at", [0, 300, 1024, 1299])
@pytest.mark.parametrize("model", PLANAR)
def test_outliers_and_coincident_particles(model, at):
    N = 1300
    q, _ = inputs.default_state(model, N, 9)
    q[at] = 1e9  # beyond 2^26 sqrt(eps): its units run in FP64
    q[N + (at + 7) % N] = -1e5
    q[(at + 11) % N], q[N + (at + 11) % N] = q[(at + 12) % N], q[N + (at + 12) % N]
    assert np.all(np.abs(_force(model, q, 1e-4) - ora.force(model, q, 1e-4)) <= _bound(model, q, 1e-4))


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("model", [1] + PLANAR)
def test_a_non_finite_position_reaches_every_force(model, bad):
    q, _ = inputs.default_state(model, 1100, 9)
    q[600] = bad
    assert np.isnan(_force(model, q, 1e-3)).all()


def _potential(model, q, eps):
    """(V, the sum of its terms' magnitudes) in long double."""
    D = model if model > 1 else 1
    x = q.reshape(D, -1).astype(np.longdouble)
    N, v, a = x.shape[1], np.longdouble(0), np.longdouble(0)
    for i in range(N - 1):
        d = x[:, i : i + 1] - x[:, i + 1 :]
        if model == 1:
            t = -1 / np.sqrt(2 * np.sin(d[0] / 2) ** 2 + np.longdouble(eps)) / np.sqrt(np.longdouble(2))
        else:
            s = (d * d).sum(0) + np.longdouble(eps)
            t = np.log(s) if model == 2 else -1 / np.sqrt(s)
        v, a = v + t.sum(), a + np.abs(t).sum()
    return v / N, float(a / N)


def _check_potential(model, q, eps):
    v, scale = _potential(model, q, eps)
    with System(model, q.size // (model if model > 1 else 1), eps, 0.01, 1) as s:
        s.set_state(q, np.zeros_like(q))
        assert abs(float(s.energy()[1] - v)) <= 1e-13 * scale


@pytest.mark.parametrize("model,eps", [(m, e) for m in (1, 2, 3) for e in (4.1, 1.0, 1e-3, 2.0**-17, 0.99 * 2.0**-17)]
                         + [(m, e) for m in (2, 3) for e in (2.0**-28, 0.99 * 2.0**-28, 1e-12)])
@pytest.mark.parametrize("N", [2, 255, 257, 513])
def test_potential_over_softenings(model, N, eps):
    _check_potential(model, inputs.default_state(model, N, 50 + N)[0], eps)


@pytest.mark.parametrize("scale", [1e-9, 1e-3, 30.0, 1e6, 1e9])
@pytest.mark.parametrize("model", [2, 3])
def test_potential_over_scales(model, scale):
    q = inputs.default_state(model, 400, 3)[0] * scale
    q[5] *= 1e4
    _check_potential(model, q, 1e-4)


def _tangent(q, v, eps, symmetric, dt=0.01):
    with System(2, q.size // 2, eps, dt, 1, precision="fp64") as s:
        s.set_tuning("symmetric", symmetric)
        s.set_state(q, np.zeros_like(q))
        return s.tangent_step(1, v, np.zeros_like(v))


TANGENTS = {
    "random": lambda g, n: g.standard_normal(n),
    "one particle": lambda g, n: np.eye(1, n, 5)[0],
    "wide range": lambda g, n: np.exp(30 * g.standard_normal(n)),
    "zero": lambda g, n: np.zeros(n),
    "tiny": lambda g, n: 1e-290 * g.standard_normal(n),
    "huge": lambda g, n: 1e150 * g.standard_normal(n),
}


@pytest.mark.parametrize("kind", TANGENTS)
@pytest.mark.parametrize("N,eps", [(1, 1e-3), (2, 1e-3), (65, 1.0), (129, 1e-4), (700, 2.0**-28), (10_001, 1e-3)])
def test_tangent_stages_equal_the_one_sided_kernel(N, eps, kind):
    """One step of the tangent dynamics against the one-sided FP64 kernel: per kick each
    side's J v is within 1e-13 of sum_j |J_ij| (|v_i| + |v_j|), |J_ij| <= 3 / s_ij <= 3 / eps,
    of which the largest row bounds the difference of dp (and, drifted, of dq); the state's own
    difference (1e-13 of the forces) enters the next kicks' J the same way.  Four kicks,
    |b| summing to 2.4, and a factor 4 for the growth within the step."""
    g = np.random.default_rng(N)
    q, _ = inputs.default_state(2, N, 3)
    if N > 600:
        q[7], q[N + 9] = 1e9, -3e4  # outliers: units in FP64
    v = TANGENTS[kind](g, 2 * N)
    x, a = q.reshape(2, N), np.abs(v).reshape(2, N).sum(0)
    S = 0.0
    for i in range(0, N, 500):
        d = x[:, i : i + 500, None] - x[:, None, :]
        s = (d * d).sum(0) + eps
        S = max(S, ((a[i : i + 500, None] + a) / s).sum(1).max() * 6.0 / N)
    tol = 1e-13 * 4 * 2.4 * 0.01 * S + 1e-15 * np.abs(v).max()
    for got, want in zip(_tangent(q, v, eps, 1), _tangent(q, v, eps, 0)):
        assert np.abs(got - want).max() <= tol


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_tangent_reaches_every_particle(bad):
    q, _ = inputs.default_state(2, 300, 3)
    v = np.ones(600)
    v[40] = bad
    dq, dp = _tangent(q, v, 1e-3, 1)
    assert not np.isfinite(dp[:300]).any()


@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_non_finite_hmf_angle(bad):
    """The magnetization of the given state, and with it every force, is NaN."""
    q, p = inputs.default_state(0, 1001, 3)
    q[500] = bad
    with System(0, 1001, 0.0, 0.1, 1, precision="fp64") as s:
        s.set_state(q, p)
        assert np.isnan(s.force()).all()
