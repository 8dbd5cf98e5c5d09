"""Which 2D tensor-core plans compute their faces as boundary strips: short and
narrow grids have more strip points than the strip warps keep up with, and run
single sweeps (the periodic boundary with its own kernel) as their grids' tiles
allow.  Parity with the oracle either way."""
import pytest

import oracle
import stencil_inputs as si
from gpuutil import check, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,r,bc,tb,kernels", [
    ((30000, 96), 2, "dirichlet", 1, 1),
    ((30000, 101), 1, "periodic", 1, 2),
    ((30000, 96), 3, "periodic", 1, 2),
    ((96, 100000), 2, "periodic", 1, 2),
    ((96, 100000), 4, "periodic", 1, 2),
    ((100, 20000), 1, "periodic", 4, 1),
    ((1500, 300), 2, "dirichlet", 2, 1),
    ((1500, 300), 3, "periodic", 1, 1),
])
def test_strips_where_the_warps_keep_up(shape, r, bc, tb, kernels):
    cg = si.coeffs_random(2, r, "box", 960 + r, dtype="f32")
    a = si.round_to(si.field_uniform(shape, 961, -1.0, 1.0), "f32")
    got, info = run(a, r, "box", cg, "f32", bc, 5, impl="matrixized")
    assert (info["tb"], info["kernels_per_sweep"]) == (tb, kernels)
    check(got, oracle.gather(a, r, cg, bc, 5), 1e-5, f"{shape} r={r} {bc}")
