"""The finish phase of the symmetric pair stages by 128-particle blocks (needs a GB300):
sampled forces against the oracle at ragged last blocks, and where a row of units is cut into
few and into many ranges (pair_vcta), FP32 within 2e-5 and FP64 within 1e-12 of
sum_j |f_ij|."""
import numpy as np
import pytest

import oracle as ora
from paper_1212_0262_gb300 import System, inputs

pytestmark = pytest.mark.gpu

EPS = {1: 0.01, 2: 1e-3, 3: 1e-3, 4: 1e-3}
SIZES = {1: [127, 129, 2999, 3000, 3001, 9000], 2: [129, 1025, 23_999, 24_000, 24_001], 3: [129, 6999, 7000, 7001, 12_345],
         4: [129, 1025, 30_001]}


@pytest.mark.parametrize("vcta", [0, 1, 32])
@pytest.mark.parametrize("prec,tol", [("mixed", 2e-5), ("fp64", 1e-12)])
@pytest.mark.parametrize("model,N", [(m, n) for m, ns in SIZES.items() for n in ns])
def test_sampled_forces(model, N, prec, tol, vcta):
    q, p = inputs.default_state(model, N, N)
    with System(model, N, EPS[model], 0.01, 1, precision=prec) as s:
        s.set_tuning("pair_vcta", vcta)
        s.set_state(q, p)
        f = s.force().reshape(-1, N)
    rows = np.unique(np.concatenate([[0, 126, N - 1, N - 2, max(N // 128 * 128 - 1, 0)], np.linspace(0, N - 1, 24).astype(np.int64)]))
    fo, scale = ora.force_rows(model, q, rows, EPS[model], True)
    assert np.all(np.abs(f[:, rows] - fo) <= tol * scale)
