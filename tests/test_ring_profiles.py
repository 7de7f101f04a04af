"""Ring means on lattices of few rows, few columns and ragged sides."""
import numpy as np
import pytest

import workloads
from paper_2409_16659_gb300 import mlswlbm as B
from tests import droplets

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,nbins", [(1, 1, 3), (700, 1, 40), (5000, 3, 3000), (8, 700, 12),
                                         (9, 33, 20), (255, 7, 9000), (300, 200, 60)])
@pytest.mark.parametrize("tau", [1.0, 0.9])
def test_ring_means_of_flat_and_narrow_lattices(nx, ny, nbins, tau):
    """Equal to the ring means of the read-back interfaces to 1e-12 (FP64
    sums of the same FP32 heights in another order), counts equal; rings in
    shared memory and (nbins 9000) beyond it."""
    p = workloads.random_params(80, 2, B.MLSW_D2Q9, nx, ny, tau=tau)
    h0 = workloads.random_heights(81, p)
    c = (0.3 * nx, 0.7 * ny)
    with B.Solver(p, h0) as s:
        s.step(2)
        prof, cnt = s.radial_profile(c, nbins)
        h = s.get_heights().astype(np.float64)
    z = np.concatenate([np.zeros((1, ny, nx)), np.cumsum(h, axis=0)])
    for m in range(3):
        rad, want, area = droplets.radial_profile(z[m], c, nbins)
        k = len(want)
        assert np.array_equal(cnt[:k], area) and not cnt[k:].any()
        assert np.abs(prof[m][:k] - want).max() <= 1e-12 * max(1.0, z[m].max())
