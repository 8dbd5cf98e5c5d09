"""The library's work as its users have it done, for timing and comparison.

Every case goes through the public binding: a solve of one field with a plan
(``Plan.apply``, or ``stencil_apply_host`` for fields in host memory), a batch
of independent problems, or a served stream of requests.  Sizes, boundaries,
step counts and weight recipes are those of ``stencil_inputs.py`` and
``bench.py``; fields are uniform random, weights random and normalised to sum
1 (or the recipe's own symmetric ones), so a field keeps its scale over many
steps.
"""
import math

import numpy as np
import torch

import paper_2310_16298_gb300 as sx

DEV = "cuda"
# Useful operations of the largest listed solves (box27_512_f32, star7_512_f64), which no drawn case exceeds.
MOST_FLOPS = {"f32": 362e9, "f64": 18.7e9}


# --------------------------------------------------------------------- cases
def solve(name, shape, r, stencil, steps, dtype="f32", bc="dirichlet", impl="auto", prec="native", tb=0,
          weights="random", signed=False, host=False):
    """One field advanced by `steps` time steps; `host`: from and to pinned host memory."""
    n = [0] * (3 - len(shape)) + list(shape)
    return {"name": name, "kind": "solve", "ndim": len(shape), "n0": n[0], "n1": n[1], "n2": n[2], "r": r,
            "stencil": stencil, "steps": steps, "dtype": dtype, "bc": bc, "impl": impl, "prec": prec, "tb": tb,
            "weights": weights, "signed": signed, "host": host}


def batch(name, problems, lo, hi, steps_lo, steps_hi):
    """Independent 2D 9-point box problems, sides log-uniform in [lo, hi], packed into one batch."""
    return {"name": name, "kind": "batch", "problems": problems, "lo": lo, "hi": hi, "steps_lo": steps_lo,
            "steps_hi": steps_hi}


def serve(name, requests, lo2, hi2, lo3, hi3, steps_lo, steps_hi):
    """Mixed requests queued at once on a server: 70% 2D, 30% 3D, 10% FP64, fields from host memory."""
    return {"name": name, "kind": "serve", "requests": requests, "lo2": lo2, "hi2": hi2, "lo3": lo3, "hi3": hi3,
            "steps_lo": steps_lo, "steps_hi": steps_hi}


def listed():
    return [
        # The smallest solve: the 5-point Jacobi smoother on a cache-resident FP64
        # grid, ten steps at a time; launches and latency are all of it.
        solve("jacobi_256_f64", (256, 256), 1, "star", 10, dtype="f64", weights="jacobi"),
        # A small FP32 field of the low end of the serving range, advanced for many steps.
        solve("box9_128_f32", (128, 128), 1, "box", 100),
        # A mid-sized FP32 field with odd sides (rows that are not 16-byte multiples), high order.
        solve("star13_1021x1533_f32", (1021, 1533), 3, "star", 40),
        # The headline workload: 25-point box, larger than L2, periodic.
        solve("box25_8192_f32", (8192, 8192), 2, "box", 100, bc="periodic"),
        # The same stencil where FP64 accuracy is needed.
        solve("box25_4096_f64", (4096, 4096), 2, "box", 10, dtype="f64", bc="periodic"),
        # FP32 on the CUDA cores with temporal blocking (several steps per pass over memory).
        solve("gather_tb4_box9_4096_f32", (4096, 4096), 1, "box", 64, impl="gather", tb=4),
        # 3D diffusion-type solves: the two standard 3D stencils on a 512^3 field.
        solve("star7_512_f32", (512, 512, 512), 1, "star", 50, signed=True),
        solve("box27_512_f32", (512, 512, 512), 1, "box", 50, signed=True),
        # A higher-order periodic 3D field that is no power of two.
        solve("star13_200x216x252_f32", (200, 216, 252), 2, "star", 20, bc="periodic", signed=True),
        # Long FP64 3D runs go in pieces of this size.
        solve("star7_512_f64", (512, 512, 512), 1, "star", 10, dtype="f64", weights="symmetric"),
        # Many uneven 2D problems in one packed batch.
        batch("batch_256", 256, 64, 2048, 20, 200),
        # A burst of mixed requests on the server, from submission to results on the host.
        serve("serve_24", 24, 128, 2048, 64, 256, 10, 200),
    ]


def points_of(r, ndim, stencil):
    return 2 * ndim * r + 1 if stencil == "star" else (2 * r + 1) ** ndim


def log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    what = rng.random()
    if what < 0.12:
        lo = log_uniform(rng, 64, 256)
        slo = rng.randint(5, 60)
        c = batch("", log_uniform(rng, 8, 256), lo, log_uniform(rng, 2 * lo, 2048), slo, slo + rng.randint(0, 140))
        while work(c)["flops"] > MOST_FLOPS["f32"] / 2:
            c["problems"] //= 2
    elif what < 0.2:
        c = serve("", log_uniform(rng, 4, 24), 128, log_uniform(rng, 256, 2048), 64, log_uniform(rng, 96, 256), 10,
                  rng.randint(20, 200))
    else:
        ndim = 2 if rng.random() < 0.6 else 3
        stencil = rng.choice(("star", "box"))
        dtype = "f64" if rng.random() < 0.25 else "f32"
        bc = rng.choice(("dirichlet", "periodic"))
        r = rng.choice((1, 1, 2, 2, 3, 4)) if ndim == 2 else rng.choice((1, 1, 1, 2, 3) if stencil == "star" else (1, 1, 2))
        top = (8192 if dtype == "f32" else 4096) if ndim == 2 else 512
        side = log_uniform(rng, 96 if ndim == 2 else 48, top)
        # most fields are near-square; rows of any length, odd ones among them
        shape = [min(top, max(2 * r + 1, int(side * rng.uniform(0.7, 1.4)))) for _ in range(ndim)]
        if rng.random() < 0.5:
            shape[-1] = max(2 * r + 1, shape[-1] // 4 * 4)
        impl, prec, tb = "auto", "native", 0
        if dtype == "f32":
            pick = rng.random()
            if pick < 0.2:
                impl, tb = "gather", rng.choice((0, 0, 2, 3, 4) if ndim == 2 else (0,))
            elif pick < 0.45:
                prec = rng.choice(("tf32", "bf16x2", "bf16x3"))
        host = rng.random() < 0.1
        flops = 2.0 * points_of(r, ndim, stencil) * float(np.prod(shape))
        steps = max(1, min(rng.randint(10, 120), int(MOST_FLOPS[dtype] / flops)))
        c = solve("", shape, r, stencil, steps, dtype, bc, impl, prec, tb, signed=rng.random() < 0.5, host=host)
    del c["name"]
    return c


# --------------------------------------------------------------------- inputs
def star_only(c, r):
    """Zero the weights off the axes."""
    off = sum((np.abs(np.arange(2 * r + 1) - r) > 0).astype(int).reshape([-1 if k == d else 1 for k in range(c.ndim)])
              for d in range(c.ndim))
    return np.where(off <= 1, c, 0.0)


def weights_of(ndim, r, stencil, dtype, recipe, rng):
    if recipe == "jacobi":
        return np.array([[0.0, 0.125, 0.0], [0.125, 0.5, 0.125], [0.0, 0.125, 0.0]])
    if recipe == "symmetric":
        c = np.where(star_only(np.ones((3, 3, 3)), 1) > 0, 0.1, 0.0)
        c[1, 1, 1] = 0.4
        return c
    c = rng.random((2 * r + 1,) * ndim)
    if stencil == "star":
        c = star_only(c, r)
    c = c / c.sum()
    return c.astype(np.float32).astype(np.float64) if dtype == "f32" else c


def torch_type(dtype):
    return torch.float32 if dtype == "f32" else torch.float64


def field_of(shape, dtype, signed, gen):
    x = torch.rand(tuple(shape), dtype=torch_type(dtype), device=DEV, generator=gen)
    return x.mul_(2).sub_(1) if signed else x


def shape_of(case):
    return [case["n1"], case["n2"]] if case["ndim"] == 2 else [case["n0"], case["n1"], case["n2"]]


def solve_problem(case, seed):
    rng = np.random.default_rng([seed, 1])
    gen = torch.Generator(device=DEV).manual_seed(seed)
    shape = shape_of(case)
    cg = weights_of(case["ndim"], case["r"], case["stencil"], case["dtype"], case["weights"], rng)
    return shape, cg, field_of(shape, case["dtype"], case["signed"], gen)


def batch_problems(case, seed):
    """(shape, weights, steps) of every problem; shapes and steps are the case's own, weights the seed's."""
    sizes = np.random.default_rng(4)
    rng = np.random.default_rng([seed, 2])
    out = []
    for _ in range(case["problems"]):
        ny, nx = (int(round(math.exp(sizes.uniform(math.log(case["lo"]), math.log(case["hi"]))))) for _ in range(2))
        steps = int(sizes.integers(case["steps_lo"], case["steps_hi"] + 1))
        out.append(((ny, nx), weights_of(2, 1, "box", "f32", "random", rng), steps))
    return out


def serve_problems(case, seed):
    """(shape, r, stencil, dtype, weights, steps, host field) of every request."""
    sizes = np.random.default_rng(5)
    rng = np.random.default_rng([seed, 3])
    out = []
    for k in range(case["requests"]):
        dtype = "f64" if sizes.random() < 0.1 else "f32"
        stencil = "star" if sizes.random() < 0.5 else "box"
        steps = int(sizes.integers(case["steps_lo"], case["steps_hi"] + 1))
        flat = sizes.random() < 0.7
        lo, hi = (case["lo2"], case["hi2"]) if flat else (case["lo3"], case["hi3"])
        side = int(round(math.exp(sizes.uniform(math.log(lo), math.log(hi)))))
        r = int(sizes.integers(1, 4)) if flat else 1
        shape = (side,) * (2 if flat else 3)
        cg = weights_of(len(shape), r, stencil, dtype, "random", rng)
        h = rng.random(shape, dtype=np.float32 if dtype == "f32" else np.float64)
        out.append((shape, r, stencil, dtype, cg, steps, h))
    return out


# --------------------------------------------------------------------- states
class Solve:
    def __init__(self, case, seed):
        shape, cg, x = solve_problem(case, seed)
        self.plan = sx.Plan(shape, case["r"], case["stencil"], cg, case["dtype"], bc=case["bc"], impl=case["impl"],
                            prec=case["prec"], tb=case["tb"])
        self.steps = case["steps"]
        self.host = case["host"]
        if self.host:
            self.x = x.cpu().pin_memory().numpy()
            self.y = torch.empty_like(x, device="cpu", pin_memory=True).numpy()
        else:
            self.x = x
            self.y = torch.empty_like(x)

    def run(self):
        if self.host:
            sx.stencil_apply_host(self.plan.handle, self.x, self.y, self.steps)
            return self.y
        return self.plan.apply(self.x, out=self.y, steps=self.steps)


class Batch:
    """Inputs and outputs of all problems in one allocation each (problems start on 256-byte boundaries)."""

    def __init__(self, case, seed):
        gen = torch.Generator(device=DEV).manual_seed(seed)
        probs = batch_problems(case, seed)
        at, offs = 0, []
        for shape, _, _ in probs:
            offs.append(at)
            at += (shape[0] * shape[1] + 63) // 64 * 64
        self.x = torch.rand(at, dtype=torch.float32, device=DEV, generator=gen)
        self.y = torch.zeros_like(self.x)
        opts = sx.make_options("native", "dirichlet", "gather", 0)
        self.plans = [sx.stencil_plan_create(shape, 1, "box", cg, "f32", opts) for shape, cg, _ in probs]
        torch.cuda.synchronize()
        self.batch = sx.stencil_batch_create(self.plans, [self.x.data_ptr() + 4 * o for o in offs],
                                             [self.y.data_ptr() + 4 * o for o in offs], [s for _, _, s in probs])

    def run(self):
        sx.stencil_batch_launch(self.batch, torch.cuda.current_stream().cuda_stream)
        return self.y

    def __del__(self):
        if getattr(self, "batch", None):
            sx.stencil_batch_destroy(self.batch)
        for p in getattr(self, "plans", []):
            sx.stencil_plan_destroy(p)


class Serve:
    def __init__(self, case, seed):
        self.server = sx.stencil_server_create(120 * 10**9, 64, 16, 8)
        self.requests, self.out = [], []
        for k, (shape, r, stencil, dtype, cg, steps, h) in enumerate(serve_problems(case, seed)):
            rq, keep = sx.make_request(shape, r, stencil, cg, dtype, steps, h_in=h)
            self.requests.append((rq, keep))
            self.out.append(np.empty_like(h))

    def run(self):
        ids = [sx.stencil_server_submit(self.server, rq) for rq, _ in self.requests]
        for rid, out in zip(ids, self.out):
            if sx.stencil_server_wait(self.server, rid) != sx.OK:
                raise RuntimeError(sx.stencil_last_error())
            sx.stencil_server_result(self.server, rid, out)
        return self.out

    def __del__(self):
        if getattr(self, "server", None):
            sx.stencil_server_destroy(self.server)


def prepare(case, seed):
    return {"solve": Solve, "batch": Batch, "serve": Serve}[case["kind"]](case, seed)


def run(state):
    return state.run()


# --------------------------------------------------------------------- floors and exact values
def work(case):
    """Each field read once and written once, and the stencil's own multiply-adds."""
    if case["kind"] == "solve":
        parts = [(shape_of(case), case["r"], case["stencil"], case["dtype"], case["steps"])]
    elif case["kind"] == "batch":
        parts = [(shape, 1, "box", "f32", steps) for shape, _, steps in batch_problems(case, 0)]
    else:
        parts = [(p[0], p[1], p[2], p[3], p[5]) for p in serve_problems(case, 0)]
    nbytes = flops = 0.0
    for shape, r, stencil, dtype, steps in parts:
        n = float(np.prod(shape))
        nbytes += 2 * n * (4 if dtype == "f32" else 8)
        flops += 2.0 * points_of(r, len(shape), stencil) * n * steps
    return {"bytes": nbytes, "flops": flops}


def exact_solve(x, r, cg, bc, steps):
    """Gather definition in FP64: every output is the weighted sum of its neighbours."""
    a = x.to(torch.float64)
    n = a.shape
    taps = [(o, float(cg[o])) for o in np.ndindex(cg.shape) if cg[o] != 0.0]
    padded = torch.zeros([s + 2 * r for s in n], dtype=torch.float64, device=a.device)
    inside = tuple(slice(r, r + s) for s in n)
    out = torch.empty_like(a)
    for _ in range(steps):
        padded[inside] = a
        if bc == "periodic":   # axis by axis, so that corners wrap too
            for d, s in enumerate(n):
                padded.narrow(d, 0, r).copy_(padded.narrow(d, s, r))
                padded.narrow(d, s + r, r).copy_(padded.narrow(d, r, r))
        out.zero_()
        for o, w in taps:
            out.add_(padded[tuple(slice(k, k + s) for k, s in zip(o, n))], alpha=w)
        a, out = out, a
    return a


def exact(case, seed):
    if case["kind"] == "solve":
        shape, cg, x = solve_problem(case, seed)
        y = exact_solve(x, case["r"], cg, case["bc"], case["steps"])
        return y.cpu() if case["host"] else y
    if case["kind"] == "batch":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        probs = batch_problems(case, seed)
        sizes = [(shape[0] * shape[1] + 63) // 64 * 64 for shape, _, _ in probs]
        x = torch.rand(sum(sizes), dtype=torch.float32, device=DEV, generator=gen)
        y = torch.zeros(x.shape, dtype=torch.float64, device=DEV)
        at = 0
        for (shape, cg, steps), size in zip(probs, sizes):
            n = shape[0] * shape[1]
            y[at:at + n] = exact_solve(x[at:at + n].view(shape), 1, cg, "dirichlet", steps).view(-1)
            at += size
        return y
    return [exact_solve(torch.from_numpy(h).to(DEV), r, cg, "dirichlet", steps).cpu()
            for _, r, _, _, cg, steps, h in serve_problems(case, seed)]
