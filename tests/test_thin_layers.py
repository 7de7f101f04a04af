"""Layers so thin that the wetting potential of FP32 thicknesses overflows,
where no spreading coefficient acts on them."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, B.MLSW_FLAG_NO_PERSISTENT])
@pytest.mark.parametrize("n,thin,S", [
    (1, 0, [[0.0]]),
    (2, 0, [[0.0, 0.0], [-1e-4]]),
    (2, 1, [[-1e-4, 0.0], [0.0]]),
    (3, 1, [[-1e-4, 0.0, 1e-4], [0.0, 0.0], [-1e-4]]),
])
def test_pairs_without_a_coefficient_act_on_no_layer(n, thin, S, flags):
    """D1Q3, exponents (3, 2), one layer of 1e-16: h*/d is 5e14 and its cube
    overflows, but the pair's coefficient is zero. Three steps against the
    oracle, each layer to 4e-6 of its largest height per step (the bound of
    the single-step comparisons)."""
    p = workloads.random_params(40 + n, n, B.MLSW_D1Q3, 64, 1)
    p.update(S=S, nw=3, mw=2, hstar=0.05, beta=[1.0] * n,
             flags=flags | B.MLSW_FLAG_SKIP_STABILITY_CHECK)
    h = workloads.random_heights(41, p, 0.5, 1.0, 1e-3)
    h[thin] *= 1e-16
    h = h.astype(np.float32)
    want = oracle.heights(p, oracle.run(p, oracle.init(p, h.astype(np.float64).ravel()), 3))
    with B.Solver(p, h) as s:
        s.step(3)
        got = s.get_heights().astype(np.float64)
        assert s.status() == B.MLSW_OK
    for i in range(n):
        assert np.abs(got[i] - want[i]).max() <= 3 * 4e-6 * h[i].max(), i
