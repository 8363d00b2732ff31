"""FP64 2D and 3D systems whose extent is nothing against their softening length, by themselves,
displaced, with a few particles elsewhere, or as groups of a wider system (needs a GB300): forces
and tangents per particle against the one-sided FP64 kernel.  A term of either is within 12
roundings, a sum passes through fewer than 64 additions of comparable partial sums:
2 x 76 x 2^-53 of the particle's own sum of the terms' magnitudes."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu

TOL = 2 * 76 * 2.0**-53
# extent in softening lengths, displacement, particles elsewhere
STATES = {
    "2^-20": (2.0**-20, 0.0, None),
    "2^-30": (2.0**-30, 0.0, None),
    "2^-45": (2.0**-45, 0.0, None),
    "2^-45 displaced": (2.0**-45, 0.7, None),
    "2^-45 and one elsewhere": (2.0**-45, 0.0, [77]),
    "2^-45 and a tenth elsewhere": (2.0**-45, 0.0, slice(0, None, 10)),
    "2^-45, the first elsewhere": (2.0**-45, 0.0, [0]),
}


def _state(dim, N, eps, kind):
    extent, at, other = STATES[kind]
    q = inputs.default_state(dim, N, 3)[0].reshape(dim, N)
    x = np.sqrt(eps) * (extent * q + at)
    if other is not None:
        x[:, other] = np.sqrt(eps) * q[:, other]
    return x.reshape(-1)


def _pair(q, dim, eps, i):
    x = q.reshape(dim, -1)
    d = x[:, i, None] - x[:, None, :]
    return d, (d * d).sum(0) + eps


@pytest.mark.parametrize("dim,N", [(2, 300), (2, 11_000), (3, 300), (3, 11_000), (2, 1), (3, 2)])
@pytest.mark.parametrize("eps", [1.0, 1e-4])
@pytest.mark.parametrize("kind", [k for k in STATES])
def test_every_particles_force(dim, N, eps, kind):
    if N < 100 and STATES[kind][2] is not None:
        pytest.skip("no particles elsewhere")
    q, out = _state(dim, N, eps, kind), []
    for symmetric in (1, 0):
        with System(dim, N, eps, 0.01, 1, precision="fp64") as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.force().reshape(dim, N))
    i = np.arange(0, N, max(1, N // 400))
    d, s = _pair(q, dim, eps, i)
    scale = (2 if dim == 2 else 1) / N * (np.abs(d) / (s if dim == 2 else s**1.5)).sum(2)
    assert np.all(np.abs(out[0] - out[1])[:, i] <= TOL * scale)


@pytest.mark.parametrize("N", [300, 11_000])
@pytest.mark.parametrize("kind", [k for k in STATES])
def test_every_particles_jacobian_product(N, kind):
    eps, h = 1e-2, 1e-40  # steps so short that every kick sees the same state
    q = _state(2, N, eps, kind)
    v, out = np.random.default_rng(N).standard_normal(2 * N), []
    for symmetric in (1, 0):
        with System(2, N, eps, h, 1, precision="fp64") as s:
            s.set_tuning("symmetric", symmetric)
            s.set_state(q, np.zeros_like(q))
            out.append(s.tangent_step(1, v, np.zeros_like(v))[1].reshape(2, N))
    i = np.arange(0, N, max(1, N // 400))
    _, s = _pair(q, 2, eps, i)
    w, _ = _pair(v, 2, 0.0, i)
    assert np.all(np.abs(out[0] - out[1])[:, i] <= TOL * 2.4 * h * 2.0 / N * (np.sqrt((w * w).sum(0)) / s).sum(1))


@pytest.mark.parametrize("kind", [k for k in STATES])
def test_every_particles_derivative_by_eps(kind):
    """With one particle k moving in one direction c, d(kinetic energy)/d eps is its own
    (df/deps)_c times the kicks."""
    N, eps, h = 300, 1e-2, 1e-40
    q = _state(2, N, eps, kind)
    for n, k in enumerate([0, 63, 64, 128, 200, N - 1]):
        c, p, out = n % 2, np.zeros_like(q), []
        p[c * N + k] = 1.0
        for symmetric in (1, 0):
            with System(2, N, eps, h, 1, precision="fp64") as s:
                s.set_tuning("symmetric", symmetric)
                s.set_state(q, p)
                out.append(s.grad(1, 0)[3])
        d, s = _pair(q, 2, eps, np.array([k]))
        assert abs(out[0] - out[1]) <= TOL * 2.4 * h * 2.0 / N * (np.abs(d) / s**2).sum(2)[c, 0]
