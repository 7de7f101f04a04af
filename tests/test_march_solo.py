"""The march with one column a lane, which lattices of four and five layers and
few columns take: the bits of the march with pairs, which batches run."""
import numpy as np
import pytest

import oracle
import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(1, 4), (3, 3), (4, 9), (7, 5), (8, 33), (25, 70), (26, 11),
                                   (27, 6), (57, 640), (78, 700), (200, 310)])
@pytest.mark.parametrize("n", [4, 5])
@pytest.mark.parametrize("kind", ["fast", "tau1", "substrate", "general"])
def test_single_columns_have_the_bits_of_pairs(nx, ny, n, kind):
    """Six steps in one run, in a resumed run, and beside two alike lattices in a
    batch: heights and populations; lattices on both sides of 26 columns, the
    halves of 57 to 78, and 256^2 or so, where the rule takes single columns."""
    p = workloads.random_params(70 + n, n, B.MLSW_D2Q9, nx, ny,
                                tau=0.8 if kind == "general" else 1.0, multilayer_S=kind != "fast")
    if kind == "substrate":
        p.update(sub_amp=0.05, sub_kx=1, sub_ky=1)
    h = workloads.random_heights(5, p).astype(np.float32)
    with B.Solver(p, h) as a, B.Solver(p, h) as c, B.Batch([p, p], [h, h]) as m:
        a.step(6)
        m.step(6)
        assert np.array_equal(m.get_heights(1), a.get_heights())
        c.step(4)
        c.load_state(*c.save_state())
        c.step(2)
        assert np.array_equal(c.save_state()[1], a.save_state()[1])
        assert np.array_equal(c.get_heights(), a.get_heights())
        assert a.status() == B.MLSW_OK and m.status() == B.MLSW_OK


@pytest.mark.parametrize("nx,ny", [(5, 6), (26, 9), (60, 650)])
@pytest.mark.parametrize("n,tau", [(4, 1.0), (5, 1.3)])
def test_single_columns_against_the_oracle(nx, ny, n, tau):
    """Three steps from a non-equilibrium state, every population to 4e-6 of the
    largest height per step (the bound of the single-step comparisons), and the
    report of a height that is not positive."""
    p = workloads.random_params(900 + n, n, B.MLSW_D2Q9, nx, ny, tau=tau)
    f = np.asarray(workloads.random_populations(901 + nx, p, 0.5, 1.0, 1e-3), np.float32)
    h0 = oracle.heights(p, f.astype(np.float64))
    want = f.astype(np.float64)
    for _ in range(3):
        want = oracle.step(p, want)
    with B.Solver(p, h0) as s:
        s.set_state(f)
        s.step(3)
        assert np.abs(s.get_state() - want).max() <= 3 * 4e-6 * h0.max()
        assert s.status() == B.MLSW_OK
        f[n - 1, 0, ny - 1, nx - 1] = -1.0
        s.set_state(f)
        s.step(1)
        assert s.status() == B.MLSW_ERR_NONFINITE
        assert s.status() == B.MLSW_OK
