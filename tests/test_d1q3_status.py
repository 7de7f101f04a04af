"""D1Q3: a height or force that is not usable is reported wherever the cell lies
in the groups of 26 that a warp writes, and a good run reports nothing."""
import numpy as np
import pytest

import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, B.MLSW_FLAG_NO_PERSISTENT])
@pytest.mark.parametrize("nx,cell", [(1, 0), (30, 0), (30, 29), (53, 25), (53, 26), (53, 52), (600, 300),
                                     (600, 599)])
@pytest.mark.parametrize("n,tau", [(1, 1.0), (2, 1.0), (3, 0.8)])
@pytest.mark.parametrize("what", ["negative", "nan", "inf flux"])
def test_unusable_cells_are_reported(nx, cell, n, tau, what, flags):
    p = workloads.random_params(20 + n, n, B.MLSW_D1Q3, nx, 1, tau=tau)
    p["flags"] = flags
    h = workloads.random_heights(21, p)
    with B.Solver(p, h) as s:
        s.step(3)
        assert s.status() == B.MLSW_OK
        f = s.get_state()
        if what == "negative":
            f[n - 1, 0, 0, cell] = -2.0
        elif what == "nan":
            f[0, 0, 0, cell] = np.nan
        else:
            f[n - 1, 1, 0, cell] = np.inf
        s.set_state(f)
        s.step(1)
        assert s.status() == B.MLSW_ERR_NONFINITE
