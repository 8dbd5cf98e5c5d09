"""GPU parity of the 2D gather kernel on grids with more tiles than resident
CTAs: tiles beyond the first of each CTA are claimed from the plan's counter,
which every launch has to leave at zero."""
import pytest

import oracle
import stencil_inputs as si
from gpuutil import check, run

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("r,kind", [(1, "box"), (3, "star")])
@pytest.mark.parametrize("tb", [1, 2, 4])
@pytest.mark.parametrize("bc", ["dirichlet", "periodic"])
def test_claimed_tiles(r, kind, tb, bc):
    import torch
    shape = (1300, 2312)   # 41 x 19 tiles of 32 x 128, at most three CTAs per SM
    assert 41 * 19 > 3 * torch.cuda.get_device_properties(0).multi_processor_count
    cg = si.coeffs_random(2, r, kind, 950 + r, dtype="f32")
    a = si.round_to(si.field_uniform(shape, 951, -1.0, 1.0), "f32")
    got, info = run(a, r, kind, cg, "f32", bc, 3 * tb + 1, impl="gather", tb=tb)
    assert info["tb"] == tb
    check(got, oracle.gather(a, r, cg, bc, 3 * tb + 1), 1e-5, f"claims {kind} r={r} tb={tb} {bc}")
