"""The workloads this library is timed on: sizes, inputs, calls and expected values.

A case is a dict of plain values; ``prepare`` makes the inputs and the plan a
program keeps, ``run`` is one pass through the public entry points, ``work`` the
bytes and operations the pass cannot do without and ``exact`` its outputs in
64 bits from the dense definition of each transform.

Two-dimensional and three-dimensional cases run the forward transform and then
the inverse of its result, as a program that works on the spectrum does, and
return both.
"""

from __future__ import annotations

import math

import torch

from paper_2110_01172_gb300 import MultiPlan, Plan, PoissonSolver, dct2, idct2, inputs


def listed():
    return [
        # one small array through the one-call functions: latency and launches
        {"name": "call_256", "op": "call", "n1": 256, "n2": 256},
        # one image-sized array through a kept plan
        {"name": "plan_1024", "op": "plan", "n1": 1024, "n2": 1024, "batch": 1},
        # the headline size: one array of 64 MiB
        {"name": "plan_4096", "op": "plan", "n1": 4096, "n2": 4096, "batch": 1},
        # the largest square of the benchmark: every array larger than L2
        {"name": "plan_8192", "op": "plan", "n1": 8192, "n2": 8192, "batch": 1},
        # few long rows
        {"name": "plan_1024x8192", "op": "plan", "n1": 1024, "n2": 8192, "batch": 1},
        # an odd number of equal images (filtering or compressing a stack of them)
        {"name": "batch_25x512", "op": "plan", "n1": 512, "n2": 512, "batch": 25},
        # many small tiles in one call
        {"name": "batch_203x64", "op": "plan", "n1": 64, "n2": 64, "batch": 203},
        # the sine transform and its inverse and both mixed kinds, as a field solver uses them
        {"name": "kinds_2048", "op": "kinds", "n1": 2048, "n2": 2048},
        # a volume
        {"name": "volume_256", "op": "volume", "n0": 256, "n1": 256, "n2": 256},
        # the benchmark's batch of uneven sizes between 64 and 1024, replayed as a graph
        {"name": "uneven_512", "op": "uneven", "count": 512, "shapes_seed": 0, "inverse": False},
        # one Poisson solve of a placement density map, the unit of the server
        {"name": "poisson_512", "op": "poisson", "n1": 512, "n2": 512},
        # the tensor-core precision mode
        {"name": "split_1024", "op": "split", "n1": 1024, "n2": 1024, "batch": 1},
    ]


def _batch(rng, elems, most):
    """A number of transforms whose elements stay within `most` (log-uniform, odd ones among them)."""
    return max(1, int(math.exp(rng.uniform(0.0, math.log(max(1, min(512, most // elems)))))))


def draw(rng):
    op = rng.choice(["call", "plan", "plan", "plan", "batch", "batch", "kinds", "volume", "uneven", "poisson", "poisson",
                     "split"])
    side = lambda lo, hi: 1 << rng.randint(lo, hi)  # noqa: E731
    if op == "call":
        return {"op": op, "n1": side(4, 10), "n2": side(4, 10)}
    if op == "plan":
        lg = rng.randint(4, 13)
        return {"op": op, "n1": 1 << lg, "n2": side(4, min(13, 25 - lg)), "batch": 1}
    if op == "batch":
        n1, n2 = side(4, 10), side(4, 10)
        return {"op": "plan", "n1": n1, "n2": n2, "batch": _batch(rng, n1 * n2, 1 << 24)}
    if op == "kinds":
        return {"op": op, "n1": side(6, 11), "n2": side(6, 12)}
    if op == "volume":
        return {"op": op, "n0": side(4, 8), "n1": side(5, 8), "n2": side(5, 9)}
    if op == "uneven":
        return {"op": op, "count": rng.randint(16, 512), "shapes_seed": rng.randint(1, 1 << 20),
                "inverse": rng.random() < 0.5}
    if op == "poisson":
        return {"op": op, "n1": side(6, 11), "n2": side(6, 11)}
    n1, n2 = side(7, 11), side(7, 11)
    return {"op": "split", "n1": n1, "n2": n2, "batch": _batch(rng, n1 * n2, 1 << 22)}


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _uniform(shape, seed):
    """i.i.d. U[-1, 1], the values of the paper's random matrices."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.rand(shape, generator=g, device="cuda", dtype=torch.float32).mul_(2.0).sub_(1.0)


def _density(n1, n2, seed, blobs=400):
    """A nonnegative density map: Gaussian blobs, sigma 1-5 % of the shorter side."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    u = torch.rand((4, blobs), generator=g, device="cuda", dtype=torch.float64)
    sigma = (0.01 + 0.04 * u[2]) * min(n1, n2)
    w = 0.1 + 0.9 * u[3]
    r1 = torch.arange(n1, device="cuda", dtype=torch.float64)[:, None]
    r2 = torch.arange(n2, device="cuda", dtype=torch.float64)[:, None]
    g1 = torch.exp(-0.5 * ((r1 - u[0] * n1) / sigma) ** 2)
    g2 = torch.exp(-0.5 * ((r2 - u[1] * n2) / sigma) ** 2)
    return ((g1 * w) @ g2.T).float().contiguous()


def _shape(case):
    if case["op"] == "volume":
        return (case["n0"], case["n1"], case["n2"])
    batch = case.get("batch", 1)
    return ((batch,) if batch > 1 else ()) + (case["n1"], case["n2"])


def _shapes(case):
    return inputs.batched_shapes(case["count"], seed=case["shapes_seed"])


def prepare(case, seed):
    op = case["op"]
    if op == "poisson":
        rho = _density(case["n1"], case["n2"], seed)
        return {"op": op, "x": rho, "solver": PoissonSolver((case["n1"], case["n2"])),
                "out": [torch.empty_like(rho) for _ in range(3)]}
    if op == "uneven":
        plan = MultiPlan(_shapes(case), graph=True)
        x = _uniform((plan.total,), seed)
        return {"op": op, "plan": plan, "x": x, "out": torch.zeros_like(x), "inverse": case["inverse"]}
    x = _uniform(_shape(case), seed)
    state = {"op": op, "x": x}
    if op == "call":
        return state
    if op == "kinds":
        state["plans"] = [Plan(x.shape, k) for k in ("dst2", "idct_idxst", "idxst_idct")]
        state["out"] = [torch.empty_like(x) for _ in range(4)]
        return state
    state["plan"] = Plan((case["n0"], case["n1"], case["n2"]) if op == "volume" else (case["n1"], case["n2"]), "dct2",
                         batch=case.get("batch", 1))
    if op == "split":
        state["plan"].set_precision("split_bf16")
    state["out"] = [torch.empty_like(x) for _ in range(2)]
    return state


def run(state):
    op, x = state["op"], state["x"]
    if op == "call":
        spectrum = dct2(x)
        return spectrum, idct2(spectrum)
    if op == "poisson":
        return state["solver"].solve(x, *state["out"])
    if op == "uneven":
        plan = state["plan"]
        return (plan.inverse if state["inverse"] else plan.forward)(x, state["out"])
    if op == "kinds":
        sine, cos_sin, sin_cos = state["plans"]
        out = state["out"]
        sine.forward(x, out[0])
        sine.inverse(out[0], out[1])
        cos_sin.inverse(x, out[2])
        sin_cos.inverse(x, out[3])
        return out
    plan, out = state["plan"], state["out"]
    plan.forward(x, out[0])
    plan.inverse(out[0], out[1])
    return out


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def _fft_flops(*sides):
    """Operations of one real transform by FFTs: 2.5 N log2 N and the combination's 7 per value."""
    n = math.prod(sides)
    return n * (2.5 * math.log2(n) + 7.0)


def work(case):
    op = case["op"]
    if op == "uneven":
        shapes = _shapes(case)
        return {"bytes": 8.0 * sum(a * b for a, b in shapes), "flops": sum(_fft_flops(*s) for s in shapes)}
    n = float(math.prod(_shape(case)))
    if op == "poisson":  # the density in, three fields out; four transforms and the scaling
        return {"bytes": 16.0 * n, "flops": 4 * _fft_flops(case["n1"], case["n2"]) + 3 * n}
    if op == "kinds":  # x in, and each of the four results out; the sine spectrum in again
        return {"bytes": 24.0 * n, "flops": 4 * _fft_flops(case["n1"], case["n2"])}
    if op == "split":  # three bf16 products for each of two dense products, both directions
        return {"bytes": 12.0 * n, "flops": 2 * 3 * 2.0 * n * (case["n1"] + case["n2"])}
    sides = _shape(case)[-3:] if op == "volume" else (case["n1"], case["n2"])
    # x in, the spectrum out and in again, the result out
    return {"bytes": 16.0 * n, "flops": 2 * case.get("batch", 1) * _fft_flops(*sides)}


# ---------------------------------------------------------------------------
# expected outputs: dense matrices of the definitions, in 64 bits
# ---------------------------------------------------------------------------

def _cos(num, n):
    """cos(pi num / 2n) for an integer tensor, the angle reduced exactly."""
    return torch.cos((num % (4 * n)).double() * (math.pi / (2 * n)))


def _grid(n):
    k = torch.arange(n, device="cuda", dtype=torch.int64)
    return k[:, None], 2 * k[None, :] + 1


def _dct(n):
    k, m = _grid(n)
    return _cos(k * m, n)


def _dst(n):  # sin(pi m (k+1) / 2n) = cos(pi (m (k+1) - n) / 2n)
    k, m = _grid(n)
    return _cos((k + 1) * m - n, n)


def _idct(n):
    d = _dct(n).T * (2.0 / n)
    d[:, 0] *= 0.5
    return d


def _idst(n):
    d = _dst(n).T * (2.0 / n)
    d[:, n - 1] *= 0.5
    return d


def _idxst(n):
    """x -> (-1)^k IDCT({x_{n-j}})_k with x_n = 0: row k, column j >= 1 is the IDCT's column n - j."""
    d = _idct(n)
    out = torch.zeros_like(d)
    out[:, 1:] = d[:, 1:].flip(1)
    out[1::2] *= -1.0
    return out


def _both(left, x, right):
    return left @ x.double() @ right.T


def exact(case, seed):
    op = case["op"]
    if op == "uneven":
        shapes = _shapes(case)
        plan = MultiPlan(shapes, graph=False)  # its layout only
        x = _uniform((plan.total,), seed)
        out = torch.zeros(plan.total, device="cuda", dtype=torch.float64)
        mats = {n: (_idct(n) if case["inverse"] else _dct(n)) for s in shapes for n in s}
        for off, (a, b) in zip(plan.offsets, shapes):
            out[off:off + a * b] = _both(mats[a], x[off:off + a * b].view(a, b), mats[b]).reshape(-1)
        return out
    n1, n2 = case["n1"], case["n2"]
    if op == "poisson":
        spectrum = _both(_dct(n1), _density(n1, n2, seed), _dct(n2))
        wu = (math.pi / n1) * torch.arange(n1, device="cuda", dtype=torch.float64)[:, None]
        wv = (math.pi / n2) * torch.arange(n2, device="cuda", dtype=torch.float64)[None, :]
        den = wu * wu + wv * wv
        den[0, 0] = 1.0
        a = spectrum / den
        a[0, 0] = 0.0
        return (_both(_idct(n1), a, _idct(n2)), _both(_idxst(n1), a * wu, _idct(n2)),
                _both(_idct(n1), a * wv, _idxst(n2)))
    x = _uniform(_shape(case), seed)
    if op == "kinds":
        return [_both(_dst(n1), x, _dst(n2)), x.double(), _both(_idct(n1), x, _idxst(n2)),
                _both(_idxst(n1), x, _idct(n2))]
    spectrum = _both(_dct(n1), x, _dct(n2))
    if op == "volume":
        spectrum = torch.tensordot(_dct(case["n0"]), spectrum, dims=1)
    return [spectrum, x.double()]
