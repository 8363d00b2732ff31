"""The ensembles' finish phase over what its blocks have to add (needs a GB300): rows cut into many
ranges (few small systems), rows of one range (many systems), two chunks of column-partial rows
(Ring beyond 32,768, 2D beyond 131,072 particles), ragged last blocks, one part only.  Sampled
forces within 2e-5 of sum_j |f_ij| of the oracle, and the same bits in a second pass (tickets)."""
import numpy as np
import pytest

import oracle as ora
from paper_1212_0262_gb300 import Ensemble, inputs

pytestmark = pytest.mark.gpu

ENSEMBLES = {
    "few small": [(1, 255), (2, 1025), (1, 1000)],
    "few": [(1, 9_001), (2, 20_001), (2, 4_097), (1, 4_095)],
    "two column chunks": [(1, 32_768), (1, 33_025), (2, 132_097)],
    "many": [(1 + s % 2, int(300 * 10 ** (s / 39))) for s in range(40)],
    "Ring only": [(1, 5_000), (1, 257)],
    "2D only": [(2, 5_000), (2, 127)],
}


@pytest.mark.parametrize("kind", ENSEMBLES)
def test_sampled_forces(kind):
    members = ENSEMBLES[kind]
    eps = [0.01 if m == 1 else 1e-3 for m, _ in members]
    ens = Ensemble([m for m, _ in members], [n for _, n in members], eps, [0.01] * len(members),
                   list(range(1, len(members) + 1)), precision="mixed")
    states = [inputs.default_state(m, n, n) for m, n in members]
    for s, (q, p) in enumerate(states):
        ens.set_state(s, q, p)
    f, again = ens.force(), ens.force()
    ens.close()
    for s, (m, n) in enumerate(members):
        assert f[s].tobytes() == again[s].tobytes()
        rows = np.unique(np.concatenate([[0, n // 2, n - 1, n - 2, (n - 1) // 256 * 256], np.linspace(0, n - 1, 16).astype(np.int64)]))
        fo, scale = ora.force_rows(m, states[s][0], rows, eps[s], True)
        assert np.all(np.abs(f[s].reshape(-1, n)[:, rows] - fo) <= 2e-5 * scale)
