"""Applies of one gather plan that may overlap: single sweeps on several streams
touch no scratch grid, and neither stencil_apply_noalloc nor a captured graph of
single sweeps shares one with stencil_apply.  Their tile counters must not be
shared either."""
import pytest

import paper_2310_16298_gb300 as sx
import stencil_inputs as si

pytestmark = pytest.mark.gpu

SHAPE = (1300, 2312)   # more tiles than resident CTAs: tiles are claimed


def make(depth):
    import torch
    cg = si.coeffs_random(2, 1, "box", 990, dtype="f32")
    plan = sx.Plan(SHAPE, 1, "box", cg, "f32", impl="gather", tb=depth)
    x = torch.rand((9,) + SHAPE, device="cuda", generator=torch.Generator("cuda").manual_seed(991))
    return plan, x


@pytest.mark.parametrize("depth", [1, 2])
def test_single_sweeps_on_many_streams(depth):
    import torch
    plan, x = make(depth)
    streams = [torch.cuda.Stream() for _ in range(8)]   # more than a plan keeps counters for
    want = [plan.apply(x[i], steps=depth) for i in range(6)]
    want += [plan.apply(x[i], steps=5 * depth) for i in (6, 7)]
    got = [torch.full_like(x[0], float("nan")) for _ in range(8)]
    torch.cuda.synchronize()
    for _ in range(10):
        for g in got:
            g.fill_(float("nan"))
        torch.cuda.synchronize()
        for i in range(6):
            for _ in range(4):   # back to back on one stream as well
                plan.apply(x[i], got[i], depth, streams[i])
        plan.apply(x[6], got[6], 5 * depth, streams[6])
        sx.stencil_apply_noalloc(plan.handle, x[7].data_ptr(), got[7].data_ptr(), 5 * depth, streams[7].cuda_stream)
        torch.cuda.synchronize()
        for i in range(8):
            assert torch.equal(got[i], want[i]), i
    assert sx.stencil_plan_info(plan.handle)["device_error"] == 0
    plan.close()


def test_captured_single_sweeps_beside_others():
    import torch
    plan, x = make(1)
    want = [plan.apply(x[i], steps=1) for i in range(3)]
    got = [torch.empty_like(x[0]) for _ in range(3)]
    streams = [torch.cuda.Stream() for _ in range(3)]
    plan.apply(x[2], got[2], 1, streams[2])
    graphs = []
    for i in range(2):
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g):
            for _ in range(4):
                plan.apply(x[i], got[i], 1)
        graphs.append(g)
    for _ in range(10):
        for t in got:
            t.fill_(float("nan"))
        torch.cuda.synchronize()
        for i in range(2):
            with torch.cuda.stream(streams[i]):
                graphs[i].replay()
        for _ in range(4):
            plan.apply(x[2], got[2], 1, streams[2])
        torch.cuda.synchronize()
        for i in range(3):
            assert torch.equal(got[i], want[i]), i
    plan.close()


def test_single_sweeps_while_another_thread_captures():
    import threading

    import torch
    plan, x = make(1)
    other = sx.Plan(SHAPE, 1, "box", si.coeffs_random(2, 1, "box", 992, dtype="f32"), "f32", impl="gather")
    want = [plan.apply(x[0], steps=1), other.apply(x[1], steps=1)]
    got = [torch.empty_like(x[0]) for _ in range(2)]
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):   # global mode: other threads' unsafe calls would end the capture
        plan.apply(x[0], got[0], 1)
        t = threading.Thread(target=lambda: [other.apply(x[1], got[1], 1, side) for _ in range(3)])
        t.start()
        t.join()
        plan.apply(x[0], got[0], 1)
    g.replay()
    torch.cuda.synchronize()
    for a, b in zip(got, want):
        assert torch.equal(a, b)
    plan.close()
    other.close()
