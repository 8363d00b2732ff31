"""Very large softenings (needs a GB300): where the unit of a fixed-point sum would lie below the
smallest double, or below the terms of padding records, the FP64 kernels run.  Forces and
d/d eps stay finite, and are zero where their terms underflow."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("half", [40, 100, 299, 300, 301, 310, 468, 469, 470, 471, 480])
@pytest.mark.parametrize("dim", [2, 3])
def test_forces(dim, half):
    """A system as wide as the softening length: d / s (2D) and d s^(-3/2) (3D) to 1e-13 of the
    largest, or zero (the FP64 kernels' reciprocals start in FP32, which ends at 2^127)."""
    N, eps = 300, 2.0 ** (2 * half)
    q = inputs.default_state(dim, N, 3)[0]
    x = q.reshape(dim, N)
    d = x[:, :, None] - x[:, None, :]
    s = (d * d).sum(0) + 1.0
    want = -(2 if dim == 2 else 1) / N * (d / (s if dim == 2 else s**1.5)).sum(2)
    unit = 2.0 ** (-half if dim == 2 else max(-2 * half, -1074))  # of the force, lengths in sqrt(eps)
    with System(dim, N, eps, 0.01, 1, precision="fp64") as sy:
        sy.set_state(q * 2.0**half, np.zeros_like(q))
        f = sy.force().reshape(dim, N)
    assert np.isfinite(f).all()
    assert np.all(np.abs(f - want * unit) <= 1e-13 * np.abs(want).max() * unit + 2.0**-1060) or (half >= 64 and not f.any())


@pytest.mark.parametrize("half", [310, 468, 470, 480])
@pytest.mark.parametrize("dim", [2, 3])
def test_forces_that_underflow(dim, half):
    """A system of ordinary size: |f| is at most 4 / eps."""
    q = inputs.default_state(dim, 300, 3)[0]
    with System(dim, 300, 2.0 ** (2 * half), 0.01, 1, precision="fp64") as s:
        s.set_state(q, np.zeros_like(q))
        assert np.abs(s.force()).max() <= 4 * 2.0 ** (-2 * half)


@pytest.mark.parametrize("spread", [1.0, 2.0**-600])
@pytest.mark.parametrize("half", [20, 70, 77, 299, 300, 301, 313, 315, 320])
def test_reverse_stages(half, spread):
    N = 300
    q, p = inputs.default_state(2, N, 3)
    with System(2, N, 2.0 ** (2 * half), 1e-3, 1, precision="fp64") as s:
        s.set_state(q, p)
        g = s.grad(1, 0)[3]
        s.set_state(q, p)
        dq, dp = s.tangent_step(1, spread * p, 0 * p)
    # d/d eps: |p| |df/deps| dt, df/deps at most 4 / eps^2; J v at most 2 |w| / eps
    assert abs(g) <= np.abs(p).sum() * 4 * 2.4e-3 * 2.0 ** max(-4 * half, -1074)
    assert np.abs(dp).max() <= 2.4e-3 * 4 * spread * np.abs(p).max() * 2.0 ** (-2 * half) + 2.0**-1060
