"""Bursts on a server: plans are built while earlier requests run (their
counters and operands must be in place before their first sweep), and pinned
result buffers come back for later bursts."""
import numpy as np
import pytest

import paper_2310_16298_gb300 as sx
import stencil_inputs as si

pytestmark = pytest.mark.gpu


def solo(shape, kind, cg, steps, h):
    import torch
    p = sx.Plan(shape, 1, kind, cg, "f32")
    try:
        return p.apply(torch.from_numpy(h).cuda(), steps=steps).cpu().numpy()
    finally:
        p.close()


def test_bursts_of_3d_requests_equal_solo_runs():
    # units beyond the first CTA wave need the claims' counter at zero; odd rows repack
    reqs = []
    for k in range(12):
        side = (99, 160, 70, 131)[k % 4]
        kind = "star" if k % 2 else "box"
        cg = si.coeffs_random(3, 1, kind, 900 + k, dtype="f32")
        h = si.field_uniform((side,) * 3, 910 + k).astype(np.float32)
        reqs.append(((side,) * 3, kind, cg, 20 + 7 * k, h))
    want = [solo(*r) for r in reqs]
    srv = sx.stencil_server_create(8 << 30, 16, 16, 8)
    try:
        for _ in range(4):
            made = [sx.make_request(s, 1, kind, cg, "f32", steps, h_in=h) for s, kind, cg, steps, h in reqs]
            ids = [sx.stencil_server_submit(srv, rq) for rq, _ in made]
            for rid, r, w in zip(ids, reqs, want):
                assert sx.stencil_server_wait(srv, rid, 60_000) == sx.OK, sx.stencil_last_error()
                out = np.empty(r[0], np.float32)
                sx.stencil_server_result(srv, rid, out)
                np.testing.assert_allclose(out, w, rtol=0, atol=2e-5)   # the star's cover may be timed anew
    finally:
        sx.stencil_server_destroy(srv)
