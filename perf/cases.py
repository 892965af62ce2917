"""What the speed of this framework is measured on: training steps, their halves and inference passes of the
YOLOv2-style stacks, through the calls a user's program makes (`ftp_step`, `ftp_step_grad` + `ftp_sgd`, `ftp_step_host`
with `ftp_prefetch_host`, `ftp_forward`, `ftp_forward` + `ftp_loss_mse` + `ftp_backward`).

Both arithmetic paths are here (fp32, tolerance-critical training; bf16 tensor cores, throughput training), from one
32 x 32 image to 64 images of 608 x 608, with the stacks, tile grids and grouping profiles of `synth.py`, of the
benchmark and of the grouping sweep (one group, one per max-pool, one per layer), maps that are ragged against every
tile size, with and without the delta at the network input.
"""
import math

import torch

import paper_2409_09083_b200 as ftp
from paper_2409_09083_b200 import synth

LR = 1e-3


def _stack(name):
    """The layer stacks: 3 layers (the tiny workload), 8 and 16 (the benchmark's), 23 (the 16 layers and the
    512 -> 1024 -> 512 ones behind them in the same network)."""
    if name == "tiny":
        return synth.stack_tiny()
    if name == "yolo8":
        return synth.stack_yolo8()
    layers = synth.stack_yolo16()
    if name == "yolo23":
        layers += [synth.conv(256, 512, 3), synth.pool(), synth.conv(512, 1024, 3), synth.conv(1024, 512, 1),
                   synth.conv(512, 1024, 3), synth.conv(1024, 512, 1), synth.conv(512, 1024, 3)]
    return layers


def _groups(layers, profile):
    """Grouping profile: "one" group, one per "maxpool", one per "layer", or the benchmark's own cuts after the
    layers named ("4", "4,8")."""
    if profile == "maxpool":
        return synth.groups_per_maxpool(layers)
    if profile == "layer":
        return synth.groups_per_layer(layers)
    cuts = [] if profile == "one" else [int(c) for c in profile.split(",")]
    ends = cuts + [len(layers)]
    return tuple((a + 1, b) for a, b in zip([0] + cuts, ends))


def _case(name, precision, stack, call, n, h, w, grid, groups, dx):
    return {"name": name, "precision": precision, "stack": stack, "call": call, "n": n, "h": h, "w": w,
            "grid_y": grid[0], "grid_x": grid[1], "groups": groups, "dx": dx}


def listed():
    return [
        # a step of the smallest workload: one 32 x 32 image, all latency and launches
        _case("fp32_step_tiny", "fp32", "tiny", "step", 1, 32, 32, (2, 2), "one", True),
        # the 8-layer training step on a small batch, and the 16-layer one on an ordinary batch: the benchmark's fp32 lines
        _case("fp32_step_8l_b4", "fp32", "yolo8", "step", 4, 416, 416, (3, 3), "one", True),
        _case("fp32_step_16l_b16", "fp32", "yolo16", "step", 16, 608, 608, (5, 5), "4,8", True),
        # one data-parallel replica's half step (gradient, then the update) on images of an odd size, no delta at the input
        _case("fp32_grad_8l_ragged", "fp32", "yolo8", "grad", 3, 200, 312, (3, 4), "maxpool", False),
        # inference on one large image
        _case("fp32_forward_16l_b1", "fp32", "yolo16", "forward", 1, 608, 608, (5, 5), "4,8", False),
        # the smallest call on the tensor-core path
        _case("bf16_forward_tiny", "bf16", "tiny", "forward", 1, 32, 32, (2, 2), "one", False),
        # the benchmark's bf16 lines, and the largest batch of the sweep
        _case("bf16_step_8l_b4", "bf16", "yolo8", "step", 4, 416, 416, (3, 3), "one", True),
        _case("bf16_step_16l_b16", "bf16", "yolo16", "step", 16, 608, 608, (5, 5), "4,8", True),
        _case("bf16_step_16l_b64", "bf16", "yolo16", "step", 64, 608, 608, (5, 5), "4,8", False),
        # training from batches in pinned host memory, the next one copied while this one is computed
        _case("bf16_host_8l_b8", "bf16", "yolo8", "host", 8, 416, 416, (4, 4), "4", False),
        # a caller's own loop (forward, loss, backward) on two images whose maps no tile size divides
        _case("bf16_fwdbwd_16l_ragged", "bf16", "yolo16", "fwdbwd", 2, 336, 464, (3, 3), "maxpool", True),
        # the wide end of the network: 512 and 1024 channels on 13 x 13 maps, parameters of 79 MB
        _case("bf16_step_23l_b8", "bf16", "yolo23", "step", 8, 416, 416, (3, 3), "maxpool", False),
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    """One more case of the same ranges: any stack, call, batch of 1 to 64, extents of 32 to 608 pixels that the pools
    divide (the tiny stack: up to 96), tile grid and grouping profile; its arithmetic stays within the largest listed
    case of its precision."""
    most = {p: max(work(c)["flops"] for c in listed() if c["precision"] == p) for p in ("fp32", "bf16")}
    while True:
        precision = rng.choice(["fp32", "bf16"])
        stack = rng.choice(["tiny", "yolo8", "yolo8", "yolo16", "yolo16", "yolo23"])
        step = {"tiny": 2, "yolo8": 8, "yolo16": 16, "yolo23": 32}[stack]
        low, high = {"tiny": (32, 96), "yolo8": (48, 608), "yolo16": (96, 608), "yolo23": (128, 608)}[stack]
        h, w = (int(_log_uniform(rng, low, high + step)) // step * step for _ in range(2))
        n = int(_log_uniform(rng, 1, 65))
        call = rng.choice(["step", "step", "grad", "forward", "fwdbwd", "host"])
        out = min(h, w) // step
        grid = (rng.randint(1, min(6, out)), rng.randint(1, min(6, out)))
        c = _case("drawn", precision, stack, call, n, h, w, grid, rng.choice(["one", "maxpool", "maxpool", "layer"]),
                  call != "forward" and rng.random() < 0.5)
        if work(c)["flops"] <= most[precision]:
            del c["name"]
            return c


def _shape(case):
    layers = _stack(case["stack"])
    return layers, synth.map_shapes(layers, 3, case["h"], case["w"])


def prepare(case, seed):
    """Plan, workspace, parameters (He-normal filters, zero biases), a batch U[0, 1) and an N(0, 1) target."""
    layers, shapes = _shape(case)
    gen = torch.Generator(device="cuda").manual_seed(seed)
    n, h, w = case["n"], case["h"], case["w"]
    plan = ftp.ftp_plan(layers, n, 3, h, w, (case["grid_y"], case["grid_x"]), _groups(layers, case["groups"]),
                        precision=1 if case["precision"] == "bf16" else 0)
    params = torch.zeros(plan.param_floats, device="cuda")
    at = 0
    for l in layers:
        if l.kind == "conv":
            k = l.cout * l.cin * l.k * l.k
            params[at:at + k].normal_(0.0, math.sqrt(2.0 / (l.cin * l.k * l.k)), generator=gen)
            at += k + l.cout
    c, oh, ow = shapes[-1]
    s = {"call": case["call"], "plan": plan, "ws": plan.new_workspace(), "params": params,
         "loss": torch.zeros(1, device="cuda"), "dx": torch.empty((n, 3, h, w), device="cuda") if case["dx"] else None}
    new_x = lambda: torch.rand((n, 3, h, w), device="cuda", generator=gen)                       # noqa: E731
    new_target = lambda: torch.randn((n, c, oh, ow), device="cuda", generator=gen)               # noqa: E731
    if case["call"] == "host":
        # two batches that take turns, as a data loader hands them over
        s["batches"] = [(new_x().cpu().pin_memory(), new_target().cpu().pin_memory()) for _ in range(2)]
        s["loss"] = torch.zeros(1).pin_memory()
        return s
    s["x"] = new_x()
    if case["call"] != "forward":
        s["target"] = new_target()
    if case["call"] in ("forward", "fwdbwd"):
        s["y"] = torch.empty((n, c, oh, ow), device="cuda")
    if case["call"] in ("grad", "fwdbwd"):
        s["dparams"] = torch.empty_like(params)
    if case["call"] == "fwdbwd":
        s["dy"] = torch.empty_like(s["y"])
    return s


def run(state):
    s = state
    plan, ws, params, call = s["plan"], s["ws"], s["params"], s["call"]
    if call == "step":
        ftp.ftp_step(plan, s["x"], params, LR, ws, target=s["target"], loss_out=s["loss"], dx=s["dx"])
        out = {"params": params, "loss": s["loss"]}
    elif call == "grad":
        ftp.ftp_step_grad(plan, s["x"], params, s["dparams"], ws, target=s["target"], loss_out=s["loss"], dx=s["dx"])
        ftp.ftp_sgd(params, s["dparams"], LR)
        out = {"dparams": s["dparams"], "params": params, "loss": s["loss"]}
    elif call == "forward":
        ftp.ftp_forward(plan, s["x"], params, s["y"], ws)
        return {"y": s["y"]}
    elif call == "fwdbwd":
        ftp.ftp_forward(plan, s["x"], params, s["y"], ws)
        ftp.ftp_loss_mse(plan, s["y"], s["target"], s["dy"], s["loss"], ws)
        ftp.ftp_backward(plan, s["x"], s["dy"], params, s["dx"], s["dparams"], ws)
        out = {"y": s["y"], "dparams": s["dparams"], "loss": s["loss"]}
    else:
        (x, t), following = s["batches"]
        ftp.ftp_step_host(plan, x, t, params, LR, s["loss"], ws, dx=s["dx"])
        ftp.ftp_prefetch_host(plan, following[0], following[1], ws)
        s["batches"].reverse()
        out = {"params": params, "loss": s["loss"]}
    if s["dx"] is not None:
        out["dx"] = s["dx"]
    return out


def work(case):
    """Multiply-accumulates of the untiled pass (forward; and for a training pass the filter gradient and the input
    delta of every layer, the first one's only if it is asked for), two operations each; the bytes of the call's inputs
    and outputs."""
    layers, shapes = _shape(case)
    n = case["n"]
    macs = [l.cout * l.cin * l.k * l.k * shapes[i + 1][1] * shapes[i + 1][2] for i, l in enumerate(layers) if l.kind == "conv"]
    x, y, params = (3 * case["h"] * case["w"] * n, shapes[-1][0] * shapes[-1][1] * shapes[-1][2] * n, synth.param_count(layers))
    if case["call"] == "forward":
        return {"bytes": 4 * (x + y + params), "flops": 2 * n * sum(macs)}
    flops = 2 * n * (3 * sum(macs) - (0 if case["dx"] else macs[0]))
    moved = x + y + 2 * params + (x if case["dx"] else 0)
    if case["call"] == "grad":
        moved += params
    if case["call"] == "fwdbwd":
        moved += y
    return {"bytes": 4 * moved, "flops": flops}


# Relative error (2-norm) that correct implementations show, about four times what these calls show against the same step
# in 64 bits (library convolutions, the maps and deltas of the bf16 path rounded where it stores them), measured over 60
# cases of these ranges.  Single layers agree to the rounding of their sums; over a stack a handful of near-ties of the
# pools and of the activations' signs are decided differently and move a whole delta to another pixel, which the delta
# at the network input shows most, the filter gradients (sums over all pixels) less and the parameters after an update
# hardly.  Stacks: tiny, 8, 16, 23 layers.
_REL = {
    ("fp32", "y"): {"tiny": 2e-6, "yolo8": 6e-6, "yolo16": 8e-6, "yolo23": 1.2e-5},
    ("fp32", "params"): {"tiny": 1e-6, "yolo8": 1e-6, "yolo16": 1e-6, "yolo23": 1e-6},
    ("fp32", "dparams"): {"tiny": 1e-4, "yolo8": 1e-4, "yolo16": 2e-4, "yolo23": 2e-3},
    ("fp32", "dx"): {"tiny": 2e-3, "yolo8": 1e-2, "yolo16": 2e-2, "yolo23": 3e-2},
    ("bf16", "y"): {"tiny": 1e-3, "yolo8": 2e-3, "yolo16": 2e-2, "yolo23": 2e-2},
    ("bf16", "params"): {"tiny": 1e-5, "yolo8": 6e-5, "yolo16": 3e-4, "yolo23": 3e-4},
    ("bf16", "dparams"): {"tiny": 2e-3, "yolo8": 2e-3, "yolo16": 2e-2, "yolo23": 3e-2},
    ("bf16", "dx"): {"tiny": 1e-2, "yolo8": 7e-2, "yolo16": 4e-1, "yolo23": 8e-1},
}


def tolerance(case):
    outputs = {"step": ["params"], "host": ["params"], "grad": ["params", "dparams"], "forward": ["y"],
               "fwdbwd": ["y", "dparams"]}[case["call"]] + (["dx"] if case["dx"] else [])
    return {"rel": max(_REL[case["precision"], o][case["stack"]] for o in outputs)}
