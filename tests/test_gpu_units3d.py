"""GPU parity of the 3D kernels' work units: units are cut along z by the
grid's size, and the tensor-core kernel's four lane quarters take columns
(y quarter, x tile) in running order, so a unit may straddle two y quarters
or reach past the last column."""
import numpy as np
import pytest

import oracle
import stencil_inputs as si
from gpuutil import TOL, check, run

pytestmark = pytest.mark.gpu

# (nz, ny, nx): one column of one quarter; columns not a multiple of four (the
# last unit reaches below the grid); a unit across two y quarters; y extents
# on and one past a quarter's 30 rows; z extents that leave a short last chunk.
SHAPES = [(3, 3, 4), (64, 64, 64), (37, 31, 20), (5, 61, 200), (131, 30, 36), (97, 90, 100)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind", ["star", "box"])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("impl,dtype", [("matrixized", "f32"), ("gather", "f32"), ("gather", "f64")])
def test_units_of_any_grid(shape, kind, bc, impl, dtype):
    cg = si.coeffs_random(3, 1, kind, 300, dtype=dtype)
    a = si.round_to(si.field_uniform(shape, 301, -1.0, 1.0), dtype)
    got, info = run(a, 1, kind, cg, dtype, bc, 3, impl=impl)
    assert info["device_error"] == 0
    check(got, oracle.gather(a, 1, cg, bc, 3), TOL[dtype], f"{impl} {kind} {bc} {shape} {dtype}")
