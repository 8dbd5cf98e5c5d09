"""CPU check of the composition behind fused 2D sweeps, restated in numpy
against the FP64 oracle: k steps are one sweep with the k-fold convolution of
the weights, except within (k-1) r of a face with a zero halo, where the
weights are those of the paths that never leave the grid, by distance class."""
import numpy as np
import pytest

import oracle
import stencil_inputs as si


def compose(r, cg, k, lo, hi):
    """Weights of the input around one output point; offsets outside [lo, hi] per axis are outside the grid."""
    R = k * r
    cur = np.zeros((2 * R + 1,) * 2)
    cur[R, R] = 1.0
    inside = [np.array([l <= o <= h for o in range(-R, R + 1)]) for l, h in zip(lo, hi)]
    for _ in range(k):
        nxt = np.zeros_like(cur)
        for a in range(-r, r + 1):
            for b in range(-r, r + 1):
                nxt += cg[a + r, b + r] * np.roll(cur, (a, b), axis=(0, 1))
        cur = nxt * inside[0][:, None] * inside[1][None, :]
    return cur


def limits(i, n, s):
    far = 1 << 20
    return (-i if i < s else -far), (n - 1 - i if n - 1 - i < s else far)


@pytest.mark.parametrize("r,k", [(1, 2), (1, 3), (1, 4), (2, 2)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
@pytest.mark.parametrize("kind", ["box", "star"])
def test_composed_sweep_equals_single_steps(r, k, bc, kind):
    shape = (17, 20)
    cg = si.coeffs_random(2, r, kind, 7)
    a = si.field_uniform(shape, 8, -1.0, 1.0)
    R, s = k * r, (k - 1) * r if bc == "dirichlet" else 0
    padded = np.pad(a, R, mode="wrap" if bc == "periodic" else "constant")
    got = np.empty(shape)
    for y in range(shape[0]):
        for x in range(shape[1]):
            (ylo, yhi), (xlo, xhi) = limits(y, shape[0], s), limits(x, shape[1], s)
            w = compose(r, cg, k, (ylo, xlo), (yhi, xhi))
            got[y, x] = (w * padded[y:y + 2 * R + 1, x:x + 2 * R + 1]).sum()
    np.testing.assert_allclose(got, oracle.gather(a, r, cg, bc, k), rtol=0, atol=1e-14)
