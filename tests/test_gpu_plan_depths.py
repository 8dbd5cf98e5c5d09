"""Gather plans of different depths alive at once: they share kernels, so what
one plan sets up must not take shared memory away from another."""
import threading

import pytest

import oracle
import paper_2310_16298_gb300 as sx
import stencil_inputs as si
from gpuutil import TOL, check, torch_dtype

pytestmark = pytest.mark.gpu


class Problem:
    def __init__(self, shape, r, dtype, depth, seed):
        import torch
        self.cg = si.coeffs_random(2, r, "box", 970 + r, dtype=dtype)
        self.a = si.round_to(si.field_uniform(shape, seed), dtype)
        self.x = torch.from_numpy(self.a).to(torch_dtype(dtype)).cuda()
        self.r, self.dtype, self.depth = r, dtype, depth
        self.plan = self.make()

    def make(self):
        return sx.Plan(self.a.shape, self.r, "box", self.cg, self.dtype, impl="gather", tb=self.depth)

    def check(self, what):
        steps = self.depth + 1
        got = self.plan.apply(self.x, steps=steps).double().cpu().numpy()
        check(got, oracle.gather(self.a, self.r, self.cg, "dirichlet", steps), TOL[self.dtype], what)


@pytest.mark.parametrize("dtype,depths", [("f32", (4, 2)), ("f64", (2, 0)), ("f64", (4, 2))])
@pytest.mark.parametrize("r", [1, 2])
@pytest.mark.parametrize("shape", [(90, 132), (700, 900)])   # few tiles (FP64: 16 rows) and many
def test_a_shallower_plan_leaves_a_deeper_one_alone(dtype, depths, r, shape):
    deep = Problem(shape, r, dtype, depths[0], 971)
    shallow = Problem(shape, r, dtype, depths[1], 972)
    try:
        for p, what in ((deep, "deep"), (shallow, "shallow"), (deep, "deep again")):
            p.check(f"{what} {dtype} r={r} {shape}")
    finally:
        deep.plan.close()
        shallow.plan.close()


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_plans_made_by_another_thread(dtype):
    """A thread creates and destroys equal and shallower plans while this one runs its own."""
    deep = Problem((90, 132), 1, dtype, 4, 973)
    shallow = Problem((90, 132), 1, dtype, 2, 974)
    shallow.plan.close()
    stop, failed = threading.Event(), []

    def churn():
        try:
            while not stop.is_set():
                for p in (deep, shallow):
                    p.make().close()
        except Exception as e:   # noqa: BLE001 (reported below)
            failed.append(e)

    t = threading.Thread(target=churn)
    t.start()
    try:
        for _ in range(50):
            deep.check(dtype)
    finally:
        stop.set()
        t.join()
        deep.plan.close()
    assert not failed, failed
