"""The widest rows a plan takes: column indexes around the right face of a grid
of nearly 2^31 columns (rows that are not 16-byte multiples: element-loaded
tiles)."""
import numpy as np
import pytest

import oracle
import paper_2310_16298_gb300 as sx
import stencil_inputs as si

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("bc,tb", [("periodic", 2), ("dirichlet", 2)])
def test_rows_of_nearly_two_to_the_31_columns(bc, tb):
    import torch
    ny, nx, E, keep = 3, 2 ** 31 - 1, 300, 290
    need = 3 * ny * nx * 4 + (2 << 30)
    torch.cuda.empty_cache()
    if torch.cuda.mem_get_info()[0] < need:
        pytest.skip(f"needs {need >> 30} GiB of device memory")
    cg = si.coeffs_random(2, 1, "box", 995, dtype="f32")
    ends = si.round_to(si.field_uniform((ny, 2 * E), 996), "f32")   # the last E columns, then the first E
    x = torch.full((ny, nx), 0.5, device="cuda")
    x[:, nx - E:] = torch.from_numpy(ends[:, :E]).float().cuda()
    x[:, :E] = torch.from_numpy(ends[:, E:]).float().cuda()
    plan = sx.Plan((ny, nx), 1, "box", cg, "f32", bc=bc, impl="gather", tb=tb)
    y = plan.apply(x, steps=tb)
    right, left = y[:, nx - keep:].double().cpu().numpy(), y[:, :keep].double().cpu().numpy()
    assert bool((y[:, 1 << 30] > 0).all())
    plan.close()
    del x, y
    torch.cuda.empty_cache()
    if bc == "periodic":   # the two ends are neighbours; far columns do not reach them
        want = oracle.gather(ends, 1, cg, bc, tb)[:, E - keep:E + keep]
        got = np.concatenate([right, left], axis=1)
    else:
        want = np.concatenate([oracle.gather(e, 1, cg, bc, tb)[:, k] for e, k in
                               ((ends[:, :E], slice(E - keep, E)), (ends[:, E:], slice(0, keep)))], axis=1)
        got = np.concatenate([right, left], axis=1)
    np.testing.assert_allclose(got, want, rtol=0, atol=1e-5)
