"""A context's forward column partials survive a reverse stage that finds no memory for its own
(needs a GB300): md_step after md_grad runs the same kernels, replayed graphs included, with
the same bits, although the allocator would not give the forward partials out again."""
import numpy as np
import pytest
from test_gpu_scratch import Bounded, columns

from paper_1212_0262_gb300 import System, inputs
from paper_1212_0262_gb300.allocator import use_cuda_allocator

pytestmark = pytest.mark.gpu


@pytest.fixture(autouse=True)
def _restore_allocator():
    yield
    use_cuda_allocator()


def test_forward_stages_after_a_refused_reverse_stage():
    N, rows = 60_001, 256  # 115 MB of forward column partials, above the one-sided stages' scratch
    q, p = inputs.default_state(2, N, 3)
    hook, out = Bounded(1 << 62), []
    for bounded in (True, False):
        if bounded:
            hook.install()
        with System(2, N, 1e-2, 0.01, 1) as s:
            s.set_state(q, p)
            s.step(10)  # some of them replayed
            if bounded:
                hook.limit = columns(N, rows, 2) - 1
                s.grad(1, 0)
            s.set_state(q, p)
            s.step(10)
            out.append(s.get_state() + (s.force(),))
        use_cuda_allocator()
    assert hook.refused == 1
    for a, b in zip(*out):
        assert np.array_equal(a, b)
