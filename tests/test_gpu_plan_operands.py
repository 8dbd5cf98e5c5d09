"""A plan holds at most 1 MiB beside its grids: the server's budget counts on it."""
import pytest

import paper_2310_16298_gb300 as sx
import stencil_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(2048, 2048), (100, 130), (160, 96, 128)])
@pytest.mark.parametrize("kind,r", [("box", 1), ("box", 2), ("star", 3), ("box", 4)])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_operands_within_the_charge(shape, kind, r, bc):
    if len(shape) == 3 and r > 3:
        pytest.skip("no tensor-core kernel")
    cg = si.coeffs_random(len(shape), r, kind, 997, dtype="f32")
    for prec in ("tf32x3", "bf16x3", "bf16"):
        plan = sx.Plan(shape, r, kind, cg, "f32", bc=bc, impl="matrixized", prec=prec)
        rows = plan.info["scratch_bytes"]
        plan.close()
        grid = 4
        for n in shape[:-1]:
            grid *= n
        padded = 2 * grid * ((shape[-1] + 3) // 4 * 4)   # rows that are not 16-byte multiples: two padded grids
        aligned = grid * shape[-1]
        held = rows - (aligned if shape[-1] % 4 == 0 else padded)
        assert 0 < held <= 1 << 20, (prec, held)
