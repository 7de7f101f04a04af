"""Friction of thin layers between thick ones: each layer's own force, also
where it is far smaller than the stresses above and below it."""
from fractions import Fraction

import numpy as np
import pytest

import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


def _forces(p, h, J):
    """Friction forces R_i = h_i G_i in rational arithmetic: J = L G, L by
    integrating the shear stress downward and the velocity upward (the dense
    FP64 oracle loses digits to z_i^3 - z_{i-1}^3 in thin layers, 1e-4 of the
    force at h = 1e-6)."""
    n = p["n"]
    mu, beta = [Fraction(m) for m in p["mu"]], [Fraction(b) for b in p["beta"]]
    h, b = [Fraction(float(v)) for v in h], [Fraction(float(v)) for v in J]
    A = [[Fraction(0)] * n for _ in range(n)]
    for j in range(n):
        u = Fraction(0)
        for i in range(n):
            s, g = (-h[j] if j > i else Fraction(0)), int(i == j)
            u += beta[i] / mu[i] * (s - g * (h[i] + beta[i] / 2))
            A[i][j] = h[i] * u + h[i] ** 2 / mu[i] * (s / 2 - g * h[i] / 3)
            u += h[i] / mu[i] * (s - g * h[i] / 2)
    for c in range(n):
        for r in range(c + 1, n):
            m = A[r][c] / A[c][c]
            A[r] = [A[r][q] - m * A[c][q] for q in range(n)]
            b[r] -= m * b[c]
    G = [None] * n
    for c in reversed(range(n)):
        G[c] = (b[c] - sum(A[c][q] * G[q] for q in range(c + 1, n))) / A[c][c]
    return np.array([float(h[i] * G[i]) for i in range(n)])


@pytest.mark.parametrize("n", [2, 3, 4, 5])
@pytest.mark.parametrize("slip", [0.0, 0.01, 1.0, 30.0])
@pytest.mark.parametrize("thin", [0.05, 1e-2, 1e-4, 1e-6])
def test_friction_of_thin_layers_layer_by_layer(n, slip, thin):
    """One layer of each cell thin, the others 0.3 to 1.5, against the exact
    solve. As for uneven layers (1e2 units of 6e-8), but each layer by
    the forces sum_j |K_ij J_j| that the layers' fluxes make on it one by one:
    every term of its elimination is a sum of those without cancellation."""
    import torch
    rng = np.random.default_rng(700 + n)
    ncell = 32
    p = workloads.random_params(600 + n, n, 2, 1, 1)
    p["mu"] = list(10.0 ** rng.uniform(-2.0, 0.0, n))
    p["beta"] = [slip] * n
    h = rng.uniform(0.3, 1.5, (n, ncell))
    h[rng.integers(0, n, ncell), np.arange(ncell)] = thin * rng.uniform(0.8, 1.2, ncell)
    h = h.astype(np.float32)
    J = (h * rng.normal(0, 1e-3, (2, n, ncell))).astype(np.float32)
    R = B.mlswlbm_friction_eval(p, *(torch.from_numpy(a).cuda() for a in (h, J[0], J[1])))
    R = [r.cpu().numpy().astype(np.float64) for r in R]
    for c in range(ncell):
        for d in range(2):
            Jc = J[d, :, c]
            parts = sum(np.abs(_forces(p, h[:, c], np.where(np.arange(n) == j, Jc, 0.0)))
                        for j in range(n))
            err = np.abs(R[d][:, c] - _forces(p, h[:, c], Jc))
            assert np.all(err <= 1e-5 * parts), (c, d)
