"""The FP64 pair stages with an allocator that has no room for the column partials of the small
units (md_step, md_force) or of the symmetric reverse stages (md_grad): the calls run with
larger units and one-sided reverse stages instead, within 1e-12 (needs a GB300)."""
import ctypes

import numpy as np
import pytest

from paper_1212_0262_gb300 import System, inputs
from paper_1212_0262_gb300 import binding as B
from paper_1212_0262_gb300.allocator import use_cuda_allocator

pytestmark = pytest.mark.gpu

ALLOC = ctypes.CFUNCTYPE(ctypes.c_void_p, ctypes.c_size_t, ctypes.c_void_p)
FREE = ctypes.CFUNCTYPE(None, ctypes.c_void_p, ctypes.c_void_p)


class Bounded:
    """Blocks of PyTorch's caching allocator, none above `limit` bytes."""

    def __init__(self, limit):
        self.limit, self.refused = limit, 0
        self.cbs = (ALLOC(self._alloc), FREE(self._free))

    def _alloc(self, nbytes, _user):
        import torch

        if nbytes > self.limit:
            self.refused += 1
            return None
        return int(torch.cuda.caching_allocator_alloc(int(nbytes), torch.cuda.current_device()))

    def _free(self, ptr, _user):
        import torch

        torch.cuda.caching_allocator_delete(int(ptr))

    def install(self):
        B.check(B.load().md_set_allocator(ctypes.cast(self.cbs[0], ctypes.c_void_p),
                                          ctypes.cast(self.cbs[1], ctypes.c_void_p), None))


def columns(N, rows, comps, tile=64):
    n_it = -(-N // rows)
    n_jt = rows // tile * n_it
    return (n_it * n_jt - rows // tile * n_it * (n_it - 1) // 2) * tile * comps * 8


@pytest.fixture(autouse=True)
def _restore_allocator():
    yield
    use_cuda_allocator()


@pytest.mark.parametrize("model,N,rows", [(1, 30_001, 256), (2, 30_001, 256), (3, 30_001, 256)])
def test_forward_stages_with_room_for_large_units_only(model, N, rows):
    q, p = inputs.ball_state(N, 3) if model == 3 else inputs.default_state(model, N, 3)
    limit = columns(N, rows, {1: 1, 2: 2, 3: 3}[model]) - 1
    hook, out = Bounded(limit), []
    for bounded in (True, False):
        if bounded:
            hook.install()
        with System(model, N, 1e-2, 0.01, 1) as s:
            s.set_state(q, p)
            s.step(12)  # some of them replayed
            out.append(s.get_state() + (s.force(),))
        use_cuda_allocator()
    assert hook.refused == 1
    for a, b in zip(*out):
        assert np.max(np.abs(a - b)) <= 1e-12 * np.abs(b).max()


def test_gradient_with_room_for_one_sided_stages_only():
    N = 30_001
    q, p = inputs.default_state(2, N, 3)
    limit = columns(N, 256, 6) - 1
    hook, out = Bounded(limit), []
    for bounded in (True, False):
        if bounded:
            hook.install()
        with System(2, N, 1e-2, 0.01, 1) as s:
            s.set_state(q, p)
            out.append(s.grad(1, 0))
        use_cuda_allocator()
    assert hook.refused == 1
    for a, b in zip(*out):  # value, d/dq, d/dp, d/d eps
        assert np.max(np.abs(np.asarray(a) - np.asarray(b))) <= 1e-11 * np.abs(np.asarray(b)).max()
