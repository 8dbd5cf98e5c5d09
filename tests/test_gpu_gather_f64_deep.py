"""GPU parity of FP64 2D gather sweeps of several steps on both sides of the
line where tiles of 64 rows begin (many tiles; stars only while two CTAs fit)."""
import pytest

import oracle
import stencil_inputs as si
from gpuutil import TOL, check, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(1257, 1998), (1088, 2012)])   # 20 x 63 and 17 x 63 tiles of 64 x 32
@pytest.mark.parametrize("r,kind,tb", [(1, "box", 4), (2, "star", 3), (3, "star", 2), (3, "box", 4), (4, "star", 3),
                                       (4, "box", 2)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_deep_f64_tiles(shape, r, kind, tb, bc):
    cg = si.coeffs_random(2, r, kind, 940 + r, dtype="f64")
    a = si.field_uniform(shape, 941, -1.0, 1.0)
    steps = tb + 1
    got, info = run(a, r, kind, cg, "f64", bc, steps, impl="gather", tb=tb)
    assert info["tb"] == tb
    check(got, oracle.gather(a, r, cg, bc, steps), TOL["f64"], f"{shape} {kind} r={r} tb={tb} {bc}")
