"""GPU parity of 2D tensor-core sweeps that advance several steps at once (the
composed stencil inside, distance-dependent or wrapped weights on the strips
along the faces)."""
import numpy as np
import pytest

import oracle
import paper_2310_16298_gb300 as sx
import stencil_inputs as si
from gpuutil import TOL, check, run

pytestmark = pytest.mark.gpu

# The smallest grid that fuses; odd and unaligned extents (padded grids); one
# and two rows past a tile's rows; ragged column groups at the right face.
SHAPES = [(96, 96), (97, 101), (233, 99), (130, 196), (100, 262)]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("kind,r", [("box", 1), ("star", 1), ("box", 2), ("star", 2), ("box", 3), ("star", 4)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
def test_fused_steps_match_the_oracle(shape, kind, r, bc, prec):
    cg = si.coeffs_random(2, r, kind, 400 + r, dtype="f32")
    a = si.round_to(si.field_uniform(shape, 401, -1.0, 1.0), "f32")
    for steps in (1, 2, 3, 7, 8):   # whole sweeps and every shorter last one
        got, info = run(a, r, kind, cg, "f32", bc, steps, impl="matrixized", prec=prec)
        assert info["tb"] == {1: 4, 2: 2}.get(r, 1) and info["kernels_per_sweep"] == 1
        check(got, oracle.gather(a, r, cg, bc, steps), TOL[prec], f"{shape} {kind} r={r} {bc} {prec} {steps} steps")


@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_fused_steps_signed_weights(bc):
    """Weights of both signs (a diffusion step near its stability limit)."""
    a = si.round_to(si.field_uniform((150, 140), 402, -1.0, 1.0), "f32")
    cg = np.zeros((3, 3))
    cg[0, 1] = cg[2, 1] = cg[1, 0] = cg[1, 2] = 0.24
    cg[1, 1] = 1 - 4 * 0.24
    cg[0, 0] = cg[2, 2] = 0.03125
    cg[0, 2] = cg[2, 0] = -0.03125
    got, info = run(a, 1, "box", cg, "f32", bc, 9, impl="matrixized")
    assert info["tb"] > 1
    check(got, oracle.gather(a, 1, cg, bc, 9), 1e-5, f"signed {bc}")


def test_steps_that_do_not_fuse():
    """An explicit depth of 1, plain precisions, small grids and weights whose
    composition would lose accuracy or range keep one step per sweep."""
    def tb(shape, cg, prec="native", depth=0):
        p = sx.Plan(shape, 1, "box", cg, "f32", impl="matrixized", prec=prec, tb=depth)
        try:
            return p.info["tb"]
        finally:
            p.close()
    avg = np.full((3, 3), 1 / 9)
    wild = np.array([[1.0, -2.0, 1.0], [-2.0, 4.0, -2.0], [1.0, -2.0, 1.0]])
    assert tb((96, 96), avg) == 4
    assert tb((96, 96), avg, depth=1) == 1
    assert tb((96, 95), avg) == tb((95, 96), avg) == 1
    for prec in ("tf32", "bf16", "bf16w2", "bf16x2"):
        assert tb((96, 96), avg, prec=prec) == 1
    assert tb((96, 96), wild) == 1
    assert tb((96, 96), avg * 2.0 ** 25) == tb((96, 96), np.zeros((3, 3))) == 1
