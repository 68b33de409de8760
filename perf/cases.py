"""The work a user of this framework has it do, as cases that can be timed.

A case is a dict of plain values.  Two kinds:

* ``kind = "plan"``: a ``Plan`` made once, run on device arrays.  ``shape``
  (text, "256x256x256"), ``P`` (virtual processes of the row-wise
  decomposition), ``order`` (a transpose order, or "" for the best one),
  ``dtype`` ("c64", "c128", "c64_tc_fp16", "c64_tc_bf16"), ``batch``
  (transforms per execution), ``direction`` ("forward", "inverse": normalised,
  "roundtrip": both), ``graph`` (replay from a CUDA graph), ``autotune``
  (``Plan.autotune`` once, as a program that runs one shape for long does),
  ``values`` ("uniform": re, im in [-1, 1); "gaussian": N(0, 1)).
* ``kind = "serve"``: a ``Server`` that is given ``requests`` transforms of
  mixed shapes at once (80 % 3-D with each axis from 48 .. 192, 20 % 32^4,
  drawn from ``mix_seed``) and drained.
"""

import math
import random

import torch

import paper_1302_6189_gb300 as md

# line lengths: products of 2, 3 and 5 that the library carries
LENGTHS = (5, 6, 8, 10, 12, 15, 16, 20, 24, 30, 32, 40, 48, 60, 64, 80, 96, 120, 128, 160, 192, 240, 256, 320, 384, 480, 512)
SERVING_AXES = (48, 64, 96, 128, 160, 192)
SERVING_BUDGET = 40 << 30
LARGEST_POINTS = 1 << 27   # points per execution: 512^3, or eight 256^3 volumes
LARGEST_C128 = 1 << 24     # 256^3


def _plan(name, shape, P, dtype="c64", batch=1, direction="forward", order="", graph=False, autotune=False,
          values="uniform"):
    case = {"kind": "plan", "shape": "x".join(str(n) for n in shape), "P": P, "order": order, "dtype": dtype,
            "batch": batch, "direction": direction, "graph": graph, "autotune": autotune, "values": values}
    return dict(case, name=name) if name else case


def _serve(name, requests, mix_seed):
    case = {"kind": "serve", "requests": requests, "mix_seed": mix_seed}
    return dict(case, name=name) if name else case


def listed():
    return [
        # a small grid with ragged, odd axes: nothing but latency and launches
        _plan("c64_30x20x15", (30, 20, 15), 16),
        # the plain method's setting: a small double precision grid on four
        # processes with one given transpose order, there and back
        _plan("c128_32cubed_roundtrip", (32, 32, 32), 4, "c128", direction="roundtrip", order="abc->cab->cba"),
        # a small grid in a time loop, replayed from a CUDA graph
        _plan("c64_64cubed_graph", (64, 64, 64), 64, direction="roundtrip", graph=True),
        # an ordinary grid with unequal axes with odd factors, one volume, the way back
        _plan("c64_60x240x160_inverse", (60, 240, 160), 256, direction="inverse"),
        # five dimensions, one array, plan as made
        _plan("c64_24x5", (24,) * 5, 1024),
        # four dimensions, several arrays per execution, plan autotuned
        _plan("c64_64x4_batch4_tuned", (64,) * 4, 64, batch=4, autotune=True),
        # one volume of the standard grid in each precision
        _plan("c64_256cubed", (256,) * 3, 4096),
        _plan("c128_256cubed", (256,) * 3, 256, "c128"),
        # many volumes of the standard grid, there and back (the headline workload)
        _plan("c64_256cubed_batch8_roundtrip", (256,) * 3, 4096, batch=8, direction="roundtrip"),
        # the largest grid, FP32 arithmetic and split FP16 on the tensor cores
        _plan("c64_512cubed", (512,) * 3, 4096, values="gaussian"),
        _plan("fp16_512cubed", (512,) * 3, 4096, "c64_tc_fp16", values="gaussian"),
        # a burst of requests of mixed shapes through the server
        _serve("serve_200_mixed", 200, 1307),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_shape(rng, M, points, largest):
    """M axis lengths around points^(1/M), unequal, their product near `points` and at most `largest`."""
    while True:
        mean = points ** (1.0 / M)
        shape = []
        for _ in range(M):
            want = mean * math.exp(rng.uniform(-0.7, 0.7))
            shape.append(min(LENGTHS, key=lambda n: abs(math.log(n / want))))
        if math.prod(shape) <= largest:
            return shape


def draw(rng):
    if rng.random() < 0.2:
        return _serve(None, _log_int(rng, 1, 128), rng.randrange(1, 1 << 20))
    dtype = rng.choice(("c64",) * 6 + ("c128",) * 2 + ("c64_tc_fp16", "c64_tc_bf16"))
    largest = LARGEST_C128 if dtype == "c128" else LARGEST_POINTS
    M = rng.choice((3, 3, 3, 4, 5))
    batch = rng.choice((1, 1, 1, 2, 4, 8))
    # rng.uniform over the logarithm: 2^12 points (16^3) up to the largest listed array
    points = 2.0 ** rng.uniform(12.0, math.log2(largest))
    if points < batch << 12:
        batch = 1
    shape = _draw_shape(rng, M, points / batch, largest // batch)
    P = min(_log_int(rng, 4, 4096), math.prod(shape))
    return _plan(None, shape, P, dtype, batch, rng.choice(("forward", "forward", "inverse", "roundtrip")),
                 graph=rng.random() < 0.25, values=rng.choice(("uniform", "gaussian")))


def _shape(case):
    return tuple(int(n) for n in case["shape"].split("x"))


def _requests(case):
    """The request shapes of a serving case, in arrival order."""
    rng = random.Random(case["mix_seed"])
    return [(32,) * 4 if rng.random() < 0.2 else tuple(rng.choice(SERVING_AXES) for _ in range(3))
            for _ in range(case["requests"])]


def _values(n, kind, dtype, seed):
    """n complex values of the seed on the GPU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    real = torch.float64 if dtype == torch.complex128 else torch.float32
    x = torch.empty(n, 2, dtype=real, device="cuda")
    if kind == "gaussian":
        x.normal_(generator=g)
    else:
        x.uniform_(-1.0, 1.0, generator=g)
    return torch.view_as_complex(x)


def _plan_input(case, seed):
    shape = _shape(case)
    full = shape if case["batch"] == 1 else (case["batch"],) + shape
    dtype = torch.complex128 if case["dtype"] == "c128" else torch.complex64
    return _values(math.prod(full), case["values"], dtype, seed).view(full)


def _split(flat, shapes):
    views, at = [], 0
    for s in shapes:
        n = math.prod(s)
        views.append(flat[at:at + n].view(s))
        at += n
    return views


def prepare(case, seed):
    if case["kind"] == "serve":
        shapes = _requests(case)
        flat = _values(sum(math.prod(s) for s in shapes), "uniform", torch.complex64, seed)
        out = torch.empty_like(flat)
        server = md.Server(budget_bytes=SERVING_BUDGET)
        return {"case": case, "server": server, "in": _split(flat, shapes), "out": _split(out, shapes), "flat": out}
    x = _plan_input(case, seed)
    plan = md.Plan(_shape(case), case["P"], case["order"] or None, case["dtype"], batch=case["batch"])
    y = torch.empty_like(x)
    if case["autotune"]:
        plan.autotune(x, y, reps=3)
    z = torch.empty_like(x) if case["direction"] == "roundtrip" else None
    return {"case": case, "plan": plan, "x": x, "y": y, "z": z}


def run(state):
    case = state["case"]
    if case["kind"] == "serve":
        server = state["server"]
        ids = [server.submit(x, y) for x, y in zip(state["in"], state["out"])]
        server.drain()
        for i in ids:
            server.release(i)
        return state["flat"]
    plan, graph = state["plan"], case["graph"]
    if case["direction"] == "inverse":
        return plan.exec(state["x"], state["y"], dir=+1, normalize=True, graph=graph)
    y = plan.exec(state["x"], state["y"], graph=graph)
    if case["direction"] == "forward":
        return y
    return [y, plan.exec(y, state["z"], dir=+1, normalize=True, graph=graph)]


def work(case):
    if case["kind"] == "serve":
        points = [math.prod(s) for s in _requests(case)]
        elem, calls, batch = 8, 1, 1
    else:
        points = [math.prod(_shape(case))]
        elem = 16 if case["dtype"] == "c128" else 8
        calls, batch = (2 if case["direction"] == "roundtrip" else 1), case["batch"]
    # a transform reads its array once and writes its result once; 5 T log2 T operations
    return {"bytes": 2 * elem * sum(points) * calls * batch,
            "flops": 5 * sum(T * math.log2(T) for T in points) * calls * batch}


def exact(case, seed):
    if case["kind"] == "serve":
        shapes = _requests(case)
        flat = _values(sum(math.prod(s) for s in shapes), "uniform", torch.complex64, seed)
        return torch.cat([torch.fft.fftn(x.to(torch.complex128)).reshape(-1) for x in _split(flat, shapes)])
    dims = tuple(range(-len(_shape(case)), 0))
    x = _plan_input(case, seed).to(torch.complex128)
    if case["direction"] == "inverse":
        return torch.fft.ifftn(x, dim=dims)
    y = torch.fft.fftn(x, dim=dims)
    return y if case["direction"] == "forward" else [y, x]
