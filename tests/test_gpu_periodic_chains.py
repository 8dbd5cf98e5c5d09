"""Long chains of periodic sweeps on small grids: the tensor-core kernel of a
step and the boundary kernel after it are launched while the step before still
runs, and each step's boundary terms read what that step wrote.  The weights
shift the field by r points a step and the field holds small whole numbers, so
every precision is exact and one stale value shows."""
import numpy as np
import pytest

from gpuutil import run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,r,kind,prec,shift", [
    ((24, 24, 24), 1, "box", "native", (1, 1, 1)),
    ((24, 24, 24), 1, "box", "native", (-1, 1, -1)),
    ((20, 33, 47), 1, "star", "native", (0, 1, 0)),
    ((24, 30, 28), 2, "star", "native", (0, 0, -2)),
    ((9, 40, 36), 2, "box", "native", (2, -2, 2)),
    ((64, 64), 1, "box", "tf32x3", (1, -1)),
    ((70, 91), 2, "box", "tf32x3", (-2, 2)),
    ((150, 164), 1, "box", "bf16x2", (1, 1)),
    ((40, 60), 4, "star", "tf32", (0, 4)),
])
def test_long_chain_of_small_periodic_sweeps(shape, r, kind, prec, shift):
    a = np.random.default_rng(981).integers(0, 256, shape).astype(np.float64)
    cg = np.zeros((2 * r + 1,) * len(shape))
    cg[tuple(r - s for s in shift)] = 1.0
    for steps in (1, 2, 301):
        got, info = run(a, r, kind, cg, "f32", "periodic", steps, impl="matrixized", prec=prec)
        assert info["kernels_per_sweep"] == 2
        assert np.array_equal(got, np.roll(a, [steps * s for s in shift], range(len(shape)))), (shape, shift, steps)
