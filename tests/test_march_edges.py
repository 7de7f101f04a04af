"""The marching D2Q9 step at the sizes where a strip can go wrong: lattices
narrower than its halo, one column more or less than a strip writes or a warp
holds, fewer rows than its warm-up."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu

SIZES = [(1, 1), (2, 3), (3, 2), (4, 1), (5, 4), (6, 5), (7, 3), (55, 3), (56, 2), (57, 5),
         (62, 4), (63, 6), (64, 7), (65, 1), (66, 3), (112, 5), (113, 9), (128, 12)]


@pytest.mark.parametrize("nx,ny", SIZES)
@pytest.mark.parametrize("n,tau", [(1, 1.0), (2, 0.8), (3, 1.0), (5, 1.0)])
def test_populations_and_split_runs_at_edge_sizes(nx, ny, n, tau):
    """Three steps from a non-equilibrium state: every population against
    the oracle (4e-6 of the largest height per step, the bound of the
    single-step comparisons); the same bits when the run is split, resumed
    from a checkpoint, or done in a batch."""
    p = workloads.random_params(900 + n, n, B.MLSW_D2Q9, nx, ny, tau=tau)
    f = np.asarray(workloads.random_populations(901 + nx, p, 0.5, 1.0, 1e-3), np.float32)
    h0 = oracle.heights(p, f.astype(np.float64))
    want = f.astype(np.float64)
    for _ in range(3):
        want = oracle.step(p, want)
    with B.Solver(p, h0) as a, B.Solver(p, h0) as b, B.Solver(p, h0) as c:
        a.set_state(f)
        a.step(3)
        got = a.get_state()
        assert a.status() == B.MLSW_OK
        assert np.abs(got - want).max() <= 3 * 4e-6 * h0.max()
        b.set_state(f)
        for _ in range(3):
            b.step(1)
        assert np.array_equal(b.get_state(), got)
        assert np.array_equal(b.get_heights(), a.get_heights())
        b.set_state(f)
        b.step(2)
        c.load_state(*b.save_state())
        b.step(1)
        c.step(1)
        assert np.array_equal(c.save_state()[1], b.save_state()[1])
        assert np.array_equal(c.get_heights(), a.get_heights())
    q = workloads.random_params(950, 4, B.MLSW_D2Q9, 40, 12)
    with B.Solver(p, h0) as a, B.Batch([q, p], [workloads.random_heights(7, q), h0]) as m:
        a.step(5)
        m.step(2)
        m.step(3)
        assert np.array_equal(m.get_heights(1), a.get_heights())


@pytest.mark.parametrize("nx", [1, 4, 25, 26, 27, 53, 520, 521, 1100])
@pytest.mark.parametrize("n,tau,sub", [(1, 1.0, 0.0), (2, 0.8, 0.0), (3, 1.0, 0.1), (5, 1.0, 0.0)])
def test_d1q3_persistent_cell_groups(nx, n, tau, sub):
    """The one-CTA D1Q3 kernel at the edges of its groups of 26 cells: the
    bits of one launch per step, flat and corrugated substrate."""
    p = workloads.random_params(970 + n, n, B.MLSW_D1Q3, nx, 1, tau=tau)
    p.update(sub_amp=sub, sub_kx=2)
    h0 = workloads.random_heights(971, p)
    q = dict(p, flags=B.MLSW_FLAG_NO_PERSISTENT)
    with B.Solver(p, h0) as a, B.Solver(q, h0) as b:
        a.step(12)
        b.step(12)
        assert np.array_equal(a.get_state(), b.get_state())
        assert a.status() == B.MLSW_OK
