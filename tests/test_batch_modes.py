"""Batches of several modes: units of equal duration, single columns for heavy
kinds, their order, and the nominal heights, against single solvers."""
import numpy as np
import pytest

import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


def _instances(lo, hi, count, layers):
    rng = np.random.default_rng(count)
    out = []
    for j in range(count):
        n, mode = layers[j % len(layers)], j % 4
        nx, ny = (int(v) for v in rng.integers(lo, hi, 2))
        p = workloads.random_params(30 + n, n, B.MLSW_D2Q9, nx, ny, tau=0.8 if mode == 0 else 1.0,
                                    multilayer_S=mode != 1)
        if mode == 2:
            p.update(sub_amp=0.05, sub_kx=1, sub_ky=1)
        out.append((p, workloads.random_heights(j, p).astype(np.float32)))
    return out


@pytest.mark.parametrize("flags", [0, B.MLSW_BATCH_TILE8, B.MLSW_BATCH_AUTOTUNE])
@pytest.mark.parametrize("lo,hi,count,layers", [(3, 70, 10, (5, 4, 2, 3, 1)), (150, 300, 12, (4, 5, 3)),
                                                (20, 120, 8, (1, 2)), (26, 90, 8, (3, 2))])
def test_mixed_modes_match_single_solvers(lo, hi, count, layers, flags):
    """Three steps of all, two of the instances of the first one's kind (pairs
    again where the mixture had single columns), two of the others, one of all:
    the bits of single solvers, in tables of one wave and of several."""
    inst = _instances(lo, hi, count, layers)
    first = [j for j, (p, _) in enumerate(inst) if (p["n"], j % 4) == (inst[0][0]["n"], 0)]
    rest = [j for j in range(count) if j not in first]
    with B.Batch([p for p, _ in inst], [h for _, h in inst], flags=flags) as b:
        b.step(3)
        b.select(first)
        b.step(2)
        b.select(rest)
        b.step(2)
        b.select(list(range(count)))
        b.step(1)
        assert b.status() == B.MLSW_OK
        for j, (p, h) in enumerate(inst):
            with B.Solver(p, h) as s:
                s.step(6)
                assert np.array_equal(b.get_heights(j), s.get_heights()), j
