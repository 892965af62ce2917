"""fp32 path on the tensor cores (one-conv groups with at least 32 input channels): parity with the fp64 oracle where the
kernels can go wrong, i.e. at the edges of their tiles and chunks and next to groups that run on other kernels.

Accuracy.  An operand is the sum of three bf16 values and a product six bf16 products, exact to 2^-24 in the 2-norm; the
tensor core's accumulator truncates, at most 4 large steps between two additions to fp32 running sums.  A convolution adds
at most 4 steps of 2^-23 and the roundings of the products and of the running sums, together less than 6 x 2^-23 of its
result.  Measured against fp64, relative 2-norm errors of these kernels | of the fp32 multiply-add kernels
(stationary = 1), He-normal filters, cases in which every pool and sign decision agrees:

    8-layer stack,  1 x 64 x 232:    y 2.2e-7 | 6.4e-7     filter gradients 1.4e-7 | 1.0e-7
    16-layer stack, 1 x 192 x 160:   y 4.3e-7 | 1.5e-6     filter gradients 3.1e-7 | 2.4e-7
    16-layer stack, 1 x 96 x 128:    y 4.2e-7 | 1.5e-6     filter gradients 3.2e-7 | 3.5e-7
"""
import numpy as np
import pytest
import torch

import paper_2409_09083_b200 as ftp
from paper_2409_09083_b200 import synth
from _util import FP32_TOL, rel_err, run_gpu, run_oracle

pytestmark = pytest.mark.gpu

W = synth.Workload
conv, pool = synth.conv, synth.pool


def one(n):
    return ((1, n),)


STACKS = {
    # 40, 72, 200, 48 channels: partial slices, chunks and operand rows; odd extents; flat runs that cross image borders
    "odd-channels": W("a", (conv(3, 40, 3), conv(40, 72, 3), conv(72, 200, 1), conv(200, 48, 3)), 3, 3, 47, 61, (2, 2), one(4)),
    # a wide map: tiles instead of flat runs; 32 and 48 input channels (filter gradient by window rows); pool; 33 channels
    "wide-map": W("b", (conv(3, 32, 3), conv(32, 48, 3), pool(), conv(48, 33, 3), conv(33, 130, 3), pool(), conv(130, 32, 1)), 2, 3, 36, 320, (1, 4), one(7)),
    # smallest maps: fewer entries than a block, one row of pixels
    "tiny-map": W("c", (conv(64, 512, 3), conv(512, 160, 1), conv(160, 256, 3)), 1, 64, 2, 150, (1, 2), one(3)),
    "stack-8-ragged": W("d", tuple(synth.stack_yolo8()), 2, 3, 88, 136, (3, 2), ((1, 4), (5, 8))),
    "stack-16": W("e", tuple(synth.stack_yolo16()), 1, 3, 112, 96, (2, 2), ((1, 4), (5, 8), (9, 16))),
    # neighbours on other kernels: pools as groups of their own, a 5x5 layer, a thin layer in the middle
    "per-layer": W("f", tuple(synth.stack_yolo8()), 1, 3, 104, 96, (2, 2), synth.groups_per_layer(synth.stack_yolo8())),
    "five-by-five": W("g", (conv(3, 32, 3), conv(32, 64, 3), pool(), conv(64, 32, 5), conv(32, 8, 3), conv(8, 64, 3), conv(64, 64, 3)), 2, 3, 64, 72, (2, 2), one(7)),
    "first-layer": W("h", (conv(64, 96, 3), pool(), conv(96, 64, 3)), 2, 64, 50, 54, (2, 2), one(3)),
}


def split_layers(plan):
    return [g for i, g in enumerate(plan.exec_groups()) if plan.group_mode(i)[0] == 1]


@pytest.mark.parametrize("name", sorted(STACKS))
def test_split_stacks_match_oracle(name):
    """Dyadic data (the forward pass is exact in any order, so every decision agrees): activations bit for bit, gradients
    within the fp32 tolerance; the workspace starts as NaN, so nothing that is not written is read into a result; the
    second step leaves the same bits."""
    wl = synth.with_slope(STACKS[name], 0.5)
    x, params, target = synth.draw_dyadic(wl, nnz=3)
    ref = run_oracle(wl, x, params, target=target)
    got = run_gpu(wl, x, params, target=target)
    assert np.array_equal(got["y"].astype(np.float64), ref["y"])
    assert rel_err(got["dx"], ref["dx"]) <= FP32_TOL
    assert rel_err(got["dparams"], ref["dparams"]) <= FP32_TOL
    plan = got["plan"]
    assert split_layers(plan)
    ws = plan.new_workspace().fill_(0xff)
    xd, pd, td = (torch.from_numpy(a).cuda() for a in (x, params, target))
    grads = [torch.empty_like(pd) for _ in range(2)]
    dxs = [torch.empty_like(xd) for _ in range(2)]
    for g, dx in zip(grads, dxs):
        ftp.ftp_step_grad(plan, xd, pd, g, ws, target=td, dx=dx)
    plan.check(ws)
    assert torch.equal(grads[0], grads[1]) and torch.equal(dxs[0], dxs[1])
    assert rel_err(grads[0].cpu().numpy(), ref["dparams"]) <= FP32_TOL


@pytest.mark.parametrize("name,convs", [("odd-channels", 8), ("wide-map", 10), ("first-layer", 4)])
def test_split_kernels_keep_fp32_accuracy(name, convs):
    """Paper-like data, slope 1 (no sign decisions; the pools' decisions are the ones of the data): every tensor within the
    bound of the module's docstring for the convolutions a value has gone through (forward and back), in the 2-norm, and
    no further from the oracle than one and a half times the fp32 multiply-add kernels."""
    wl = synth.with_slope(STACKS[name], 1.0)
    if name == "wide-map":
        wl = wl.with_(layers=tuple(l for l in wl.layers if l.kind == "conv"), groups=one(5), H=18, W=320)
    if name == "first-layer":
        wl = wl.with_(layers=tuple(l for l in wl.layers if l.kind == "conv"), groups=one(2))
    x, params, _ = synth.draw(wl, bias_std=0.1)
    c, h, w = synth.map_shapes(wl.layers, wl.C, wl.H, wl.W)[-1]
    dy = np.random.default_rng(4).standard_normal((wl.N, c, h, w)).astype(np.float32)
    ref = run_oracle(wl, x, params, dy=dy)
    got = run_gpu(wl, x, params, dy=dy)
    fma = run_gpu(wl, x, params, dy=dy, stationary=1)
    norm = lambda a, o: float(np.linalg.norm((a.astype(np.float64) - o).ravel()) / np.linalg.norm(o.ravel()))
    for k in ("y", "dx", "dparams"):
        assert norm(got[k], ref[k]) <= convs * 6 * 2.0 ** -23, k
        assert norm(got[k], ref[k]) <= 1.5 * norm(fma[k], ref[k]), k


def test_small_stacks_stay_on_the_multiply_add_kernels():
    """The rule looks at one image's multiply-accumulates, not at the batch: a batch and its halves take the same kernels."""
    plan = lambda n, h, w, **kw: ftp.ftp_plan(tuple(synth.stack_yolo8()), n, 3, h, w, (2, 2), one(8), **kw)
    small, large = plan(64, 64, 96), plan(1, 88, 104)
    assert small.workspace_bytes == plan(64, 64, 96, stationary=0).workspace_bytes
    assert plan(2, 88, 104).workspace_bytes != plan(2, 88, 104, stationary=1).workspace_bytes
    assert large.group_mode(1)[0] == 1
