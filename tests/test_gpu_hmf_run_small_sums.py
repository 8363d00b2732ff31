"""Small mixed HMF systems whose sums of sines or cosines are small take the launched stages' FP64
sums in their one launch too (needs a GB300): states equal those of the launched stages bit for
bit where the angles all lie near a multiple of pi / 2, where the magnetization nearly vanishes,
and in ordinary systems."""
import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu


def _angles(kind, N):
    u = 2 * np.random.default_rng(N).random(N) - 1
    if kind == "water bag":
        return inputs.default_state(0, N, 5)[0]
    if kind == "lattice":
        return 2 * np.pi * np.arange(N) / N + 1e-6 * u
    at, extent = kind
    return at + extent * u


@pytest.mark.parametrize("N", [1, 2, 301, 4097, 10_007])
@pytest.mark.parametrize("kind", [(0.0, 1e-12), (0.0, 1e-9), (0.0, 1e-5), (0.0, 1e-3), (np.pi / 2, 1e-9), (np.pi, 1e-5), "lattice", "water bag"])
def test_one_launch_equals_launched_stages(kind, N):
    out = []
    for graphs in (1, 0):
        with System(0, N, 0.0, 0.1, 1, precision="mixed") as s:
            s.set_tuning("step_graphs", graphs)
            s.set_state(_angles(kind, N), np.zeros(N))
            s.step(12)
            out.append(s.get_state() + (s.force(),))
    for a, b in zip(*out):
        assert np.array_equal(a, b)
