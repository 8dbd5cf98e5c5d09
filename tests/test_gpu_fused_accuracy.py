"""Fused 2D sweeps are no less exact than single ones: relative L2 error of the
same plan with and without fusing (tb = 1), many steps, against FP64."""
import numpy as np
import pytest

import oracle
import paper_2310_16298_gb300 as sx
import stencil_inputs as si

pytestmark = pytest.mark.gpu


def fourth_order_diffusion():
    c = np.zeros((5, 5))
    k = np.array([-1.0, 16.0, -30.0, 16.0, -1.0]) / 12.0 * 0.15
    c[2] += k
    c[:, 2] += k
    c[2, 2] += 1.0
    return c


def advection():   # second order, two directions
    row = lambda a: np.array([a * (a + 1) / 2, 1 - a * a, a * (a - 1) / 2])
    return np.outer(row(0.4), row(0.3))


WEIGHTS = {
    "random1": (1, lambda: si.coeffs_random(2, 1, "box", 103, dtype="f32")),
    "random2": (2, lambda: si.coeffs_random(2, 2, "box", 103, dtype="f32")),
    "jacobi": (1, lambda: np.array([[0, 0.125, 0], [0.125, 0.5, 0.125], [0, 0.125, 0]])),
    "binomial": (2, lambda: np.outer([1, 4, 6, 4, 1], [1, 4, 6, 4, 1]) / 256.0),
    "advection": (1, advection),
    "diffusion4": (2, fourth_order_diffusion),
}


@pytest.mark.parametrize("weights", WEIGHTS)
@pytest.mark.parametrize("prec", ["tf32x3", "bf16x3"])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("lo", [0.0, -1.0])
def test_fusing_loses_no_accuracy(weights, prec, bc, lo):
    import torch
    r, make = WEIGHTS[weights]
    cg, shape = make(), (160, 172)
    a = si.round_to(si.field_uniform(shape, 411, lo, 1.0), "f32")
    x = torch.from_numpy(a).float().cuda()
    for steps in (20, 100):
        want = oracle.gather(a, r, cg, bc, steps)
        err = {}
        for depth in (1, 0):
            plan = sx.Plan(shape, r, "box", cg, "f32", bc=bc, impl="matrixized", prec=prec, tb=depth)
            assert (plan.info["tb"] > 1) == (depth == 0)
            got = plan.apply(x, steps=steps).double().cpu().numpy()
            plan.close()
            err[depth] = np.linalg.norm(got - want) / np.linalg.norm(want)
        # one FP32 rounding of the result is 2^-24 / sqrt(3) relative; no worse beyond that
        assert err[0] <= err[1] + 3.5e-8, (steps, err)
