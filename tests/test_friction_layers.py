"""The tridiagonal friction of the step kernels where it is least benign:
thin precursors under thick films, viscosities decades apart, no slip."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("slip", [0.0, 1.0])
def test_friction_of_uneven_layers_matches_oracle(n, slip):
    """h from 0.05 to 60, mu over two decades, against the dense FP64 solve.
    FP32 inputs and about ten rounded operations per row of a diagonally
    dominant system change a force by at most some 1e2 units of 6e-8 of the
    forces sum_j |K_ij J_j| that the layers' fluxes make one by one (K the
    friction matrix, column by column from the oracle); 1e-5 of the largest
    such sum is the bound."""
    import torch
    rng = np.random.default_rng(500 + n)
    ncell = 64
    p = workloads.random_params(600 + n, n, 2, 1, 1)
    p["mu"] = list(10.0 ** rng.uniform(-2.0, 0.0, n))
    p["beta"] = [slip] * n
    h = np.exp(rng.uniform(np.log(0.05), np.log(60.0), (n, ncell))).astype(np.float32)
    J = rng.normal(0, 1e-3, (2, n, ncell)).astype(np.float32)
    R = B.mlswlbm_friction_eval(p, *(torch.from_numpy(a).cuda() for a in (h, J[0], J[1])))
    R = [r.cpu().numpy().astype(np.float64) for r in R]
    for c in range(ncell):
        hc, Jc = h[:, c].astype(np.float64), J[:, :, c].astype(np.float64)
        want = oracle.friction(p, hc, Jc[0], Jc[1])
        for d in range(2):
            parts = sum(np.abs(oracle.friction(p, hc, np.where(np.arange(n) == j, Jc[d], 0.0),
                                               np.zeros(n))[0]) for j in range(n))
            assert np.abs(R[d][:, c] - want[d]).max() <= 1e-5 * parts.max(), (c, d)
