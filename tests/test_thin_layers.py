"""Layers at the thin end of the FP32 range: the wetting potential of pairs
without a coefficient, and the FP64 analysis."""
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


@pytest.mark.parametrize("lat", [2, 1])
@pytest.mark.parametrize("n,thin", [(1, 0), (2, 1), (3, 0)])
def test_analysis_of_layers_below_the_normal_fp32_range(n, thin, lat):
    """One layer of 1e-40, at rest: the kinetic energy is zero, the smallest
    height its own, and the free energy (with a coefficient on that layer's
    pair where its thickness is not lost to the interface below) equals the
    sum over the read-back heights to 1e-10, as for thick layers."""
    ny = 1 if lat == 1 else 12
    p = workloads.random_params(60 + n, n, lat, 40, ny)
    S = [[0.0] * (n - i) for i in range(n)]
    S[0][0] = 1e-3 if thin == 0 else 0.0
    p.update(S=S, hstar=0.05, nw=3, mw=2, flags=B.MLSW_FLAG_SKIP_STABILITY_CHECK)
    h = workloads.random_heights(61, p, 0.5, 1.0, 1e-3)
    h[thin] = 1e-40
    h = h.astype(np.float32)
    with B.Solver(p, h) as s:
        mass, ke, hmin = s.get_diagnostics()
        F = s.free_energy()
        got = s.get_heights().astype(np.float64)
    assert ke == 0.0 and hmin == h[thin].min()
    np.testing.assert_allclose(mass, got.sum(axis=(1, 2)), rtol=1e-6)
    z = np.concatenate([np.zeros((1, ny, 40)), np.cumsum(got, axis=0)])
    xp, xm = np.roll(z, -1, axis=2), np.roll(z, 1, axis=2)
    if lat == 1:
        g2 = (0.5 * (xp - xm)) ** 2
    else:
        N, So = (lambda a: np.roll(a, -1, axis=1)), (lambda a: np.roll(a, 1, axis=1))
        gx = (xp - xm) / 3 + ((N(xp) - N(xm)) + (So(xp) - So(xm))) / 12
        gy = (N(z) - So(z)) / 3 + ((N(xp) - So(xp)) + (N(xm) - So(xm))) / 12
        g2 = gx ** 2 + gy ** 2
    r = p["hstar"] / got[thin]
    want = sum(p["gamma"][i] * (1 + 0.5 * g2[i + 1]).sum() for i in range(n)) + \
        (S[0][0] * (3 * r ** 2 - 2 * r ** 3) * (1 + 0.5 * g2[thin])).sum()
    assert np.isfinite(F) and F == pytest.approx(want, rel=1e-10)
