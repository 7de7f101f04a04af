"""Batches of one kind (layer count and mode), which have a kernel of their
own: the bits of single solvers."""
import numpy as np
import pytest

import workloads
from paper_2409_16659_gb300 import mlswlbm as B

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny", [(5, 4), (57, 9), (64, 33), (130, 70)])
@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
@pytest.mark.parametrize("kind", ["fast", "tau1", "general"])
@pytest.mark.parametrize("vary", ["heights", "parameters", "sizes"])
def test_alike_instances_match_single_solvers(nx, ny, n, kind, vary):
    """Three instances that differ in the heights alone (their parameters come
    as the kernel's), in a tension, or in the size: 3 and 2 steps, then 2 of
    a subset after a step beside an instance of another kind."""
    params, heights = [], []
    for j in range(3):
        size = (nx + j, ny + 2 * j) if vary == "sizes" else (nx, ny)
        p = workloads.random_params(70 + n, n, B.MLSW_D2Q9, *size,
                                    tau=0.9 if kind == "general" else 1.0,
                                    multilayer_S=kind != "fast")
        if vary == "parameters":
            p["gamma"] = [g * (1.0 + 0.01 * j) for g in p["gamma"]]
        params.append(p)
        heights.append(workloads.random_heights(80 + j, p, 0.5 + 0.1 * j, 0.8 + 0.1 * j))
    other = workloads.random_params(91, 2, B.MLSW_D2Q9, 40, 12, tau=0.8)
    solvers = [B.Solver(p, h) for p, h in zip(params, heights)]
    try:
        with B.Batch(params, heights) as a, \
                B.Batch(params + [other], heights + [workloads.random_heights(92, other)]) as m:
            a.step(3)
            a.step(2)
            m.step(3)
            m.select([0, 1, 2])
            m.step(2)
            for j, s in enumerate(solvers):
                s.step(5)
                h = s.get_heights()
                assert np.array_equal(a.get_heights(j), h)
                assert np.array_equal(m.get_heights(j), h)
            assert a.status() == B.MLSW_OK and m.status() == B.MLSW_OK
    finally:
        for s in solvers:
            s.close()
