"""fp32 path on the tensor cores (one-conv groups with at least 32 input channels): parity with the fp64 oracle where the
kernels can go wrong, i.e. at the edges of their tiles and chunks and next to groups that run on other kernels.

Accuracy.  An operand is the sum of three bf16 values and a product six bf16 products, exact to 2^-24 in the 2-norm; the
tensor core's accumulator truncates, at most 4 large steps between two additions to fp32 running sums.  A convolution adds
at most 4 steps of 2^-23 and the roundings of the products and of the running sums, together less than 6 x 2^-23 of its
result.  What the tests below measure against fp64, relative 2-norm errors of these kernels | of the fp32 multiply-add
kernels (stationary = 1):

    one layer, 64 -> 64, 16 x 304 x 304:              y 1.0e-7 | 4.0e-7    dx 1.0e-7 | 4.3e-7    filters 1.0e-7 | 2.2e-7
    one layer, 1024 -> 64, all terms positive:        y 2.1e-7 | 1.4e-6    dx 6.5e-8 | 3.5e-7    filters 4.8e-8 | 1.0e-7
    8 leaky layers with pools, 2 x 88 x 136 (median): y 3.5e-7 | 6.9e-7    dx 2.9e-7 | 7.6e-7    filters 4.6e-7 | 7.8e-7
    16 leaky layers with pools, 1 x 112 x 96:         y 5.6e-7 | 1.7e-6    dx 6.2e-7 | 2.1e-6    filters 6.0e-7 | 1.7e-6
"""
import numpy as np
import pytest
import torch

import paper_2409_09083_b200 as ftp
from paper_2409_09083_b200 import synth
from _util import FP32_TOL, assert_split, kernels, rel_err, run_gpu, run_oracle

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
    assert_split(plan, wl.layers)
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
    assert_split(got["plan"], wl.layers)
    assert all("split" not in k for k in kernels(fma["plan"]).values())
    norm = lambda a, o: float(np.linalg.norm((a.astype(np.float64) - o).ravel()) / np.linalg.norm(o.ravel()))
    for k in ("y", "dx", "dparams"):
        assert norm(got[k], ref[k]) <= convs * 6 * 2.0 ** -23, k
        assert norm(got[k], ref[k]) <= 1.5 * norm(fma[k], ref[k]), k


def test_forward_on_the_row_kernel_leaves_the_input_as_it_is():
    """A first layer with 32 input channels: its forward pass reads the fp32 input, so the conversion to split form, which only the
    filter gradient reads, is no part of ftp_forward (two packing launches and the convolution)."""
    wl = SINGLE["32-channels"]
    x, params, dy = draw_single(wl)
    plan = ftp.ftp_plan(wl.layers, wl.N, wl.C, wl.H, wl.W, wl.grid, wl.groups)
    assert_split(plan, wl.layers)
    ws = plan.new_workspace().fill_(0xff)
    xd, pd, dyd = (torch.from_numpy(a).cuda() for a in (x, params, dy))
    ftp.ftp_forward(plan, xd, pd, None, ws)
    assert plan.launch_count() == 3
    grads = [torch.empty_like(pd) for _ in range(2)]
    for g in grads:                                          # the backward pass can be repeated after one forward pass
        ftp.ftp_backward(plan, xd, dyd, pd, None, g, ws)
    plan.check(ws)
    ref = run_oracle(wl, x, params, dy=dy)
    assert torch.equal(*grads) and rel_err(grads[0].cpu().numpy(), ref["dparams"]) <= FP32_TOL


def test_wait_that_runs_out_is_reported():
    """Split plans have bounded waits on the device: see the test of the same name on the bf16 path."""
    from paper_2409_09083_b200 import binding
    wl = STACKS["stack-8-ragged"]
    x, params, _ = synth.draw(wl)
    plan = ftp.ftp_plan(wl.layers, wl.N, wl.C, wl.H, wl.W, wl.grid, wl.groups)
    ws = plan.new_workspace()
    xd, pd = torch.from_numpy(x).cuda(), torch.from_numpy(params).cuda()
    y = [torch.empty((wl.N,) + tuple(synth.map_shapes(wl.layers, wl.C, wl.H, wl.W)[-1]), device="cuda") for _ in range(2)]
    ftp.ftp_forward(plan, xd, pd, y[0], ws)
    plan.check(ws)
    plan.wait_probe(ws, limit_us=2000)
    with pytest.raises(binding.FtpError) as e:
        plan.check(ws)
    assert e.value.code == -7
    ftp.ftp_forward(plan, xd, pd, y[1], ws)                  # clears the error word
    plan.check(ws)
    assert torch.equal(y[0], y[1])


# one layer on a batch of two, above the 1e8 rule: flat runs; tiles with a pool; a 1x1 layer; tiles of a wide map; the forward pass on
# the row kernel
SINGLE = {
    "flat": W("i", (conv(64, 48, 3),), 2, 64, 66, 70, (2, 2), one(1)),
    "pool": W("j", (conv(64, 48, 3), pool()), 2, 64, 66, 70, (2, 2), one(2)),
    "one-by-one": W("k", (conv(256, 200, 1),), 2, 256, 50, 52, (2, 2), one(1)),
    "wide": W("l", (conv(64, 48, 3),), 2, 64, 20, 320, (2, 2), one(1)),
    "32-channels": W("m", (conv(32, 64, 3), pool()), 2, 32, 88, 90, (2, 2), one(2)),
}
# ... and with maps between the layers, written by an epilogue: without and with a pool, on the row kernel
CHAINS = {
    "chain": W("n", (conv(64, 64, 3), conv(64, 48, 1)), 2, 64, 50, 62, (2, 2), one(2)),
    "chain-pool": W("o", (conv(64, 64, 3), pool(), conv(64, 48, 3)), 2, 64, 52, 64, (2, 2), one(3)),
    "chain-32": W("p", (conv(32, 64, 3), conv(64, 64, 3)), 2, 32, 52, 64, (2, 2), one(2)),
    "chain-32-pool": W("q", (conv(32, 64, 3), pool(), conv(64, 64, 3)), 2, 32, 84, 88, (2, 2), one(3)),
}


def draw_single(wl):
    x, params, _ = synth.draw(wl, bias_std=0.1)
    shape = (wl.N,) + tuple(synth.map_shapes(wl.layers, wl.C, wl.H, wl.W)[-1])
    return x, params, np.random.default_rng(1).standard_normal(shape).astype(np.float32)


def classes(a):
    return np.where(np.isnan(a), 3, np.where(np.isposinf(a), 1, np.where(np.isneginf(a), 2, 0)))


@pytest.mark.filterwarnings("ignore:invalid value encountered")
@pytest.mark.parametrize("where", ["x", "dy"])
@pytest.mark.parametrize("name", sorted(SINGLE))
def test_infinities_and_nans_reach_what_they_reach_in_a_plain_sum(name, where):
    """An infinity stays one: in the last map and the input delta exactly the values of the untiled sums are infinite (with their
    signs) or NaN, the others stay finite and accurate.  In the filter gradient too, but for the window positions that lead
    out of the map from a pixel at its border: there a zero of the padding meets the infinity, and a NaN may stand for the
    finite value (the multiply-add kernels do the same at the edges of their tiles)."""
    wl = SINGLE[name]
    x, params, dy = draw_single(wl)
    if where == "x":
        x[0, 5, 10, 12], x[1, 7, 9, 30], x[0, 9, 15, 40] = np.inf, -np.inf, np.nan
        x[0, 11, 0, 0], x[1, 12, -1, -1], x[0, 13, 3, -1], x[0, 14, -1, 4] = np.inf, np.inf, np.inf, -np.inf
    else:
        dy[0, 5, 5, 6], dy[1, 7, 7, 9], dy[0, 9, 8, 20] = np.inf, -np.inf, np.nan
        dy[0, 11, 0, 0], dy[1, 12, -1, -1] = np.inf, np.inf
    ref, got = run_oracle(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy)
    assert_split(got["plan"], wl.layers)
    for k in ("y", "dx", "dparams"):
        g, r = got[k].astype(np.float64), ref[k]
        cg, cr = classes(g), classes(r)
        if k == "dparams":
            cout, cin, kk = wl.layers[0].cout, wl.layers[0].cin, wl.layers[0].k ** 2
            border = np.zeros((cout, cin, kk), bool)
            if where == "x":
                border[:, 11:15] = True
            else:
                border[11:13] = True
            border = np.concatenate([border.ravel(), np.zeros(cout, bool)])
            cg = np.where(border & (cg == 3) & (cr == 0), 0, cg)
        assert np.array_equal(cg, cr), (k, int((cg != cr).sum()))
        ok = np.isfinite(g) & np.isfinite(r)
        assert np.linalg.norm(g[ok] - r[ok]) <= 2 * 6 * 2.0 ** -23 * np.linalg.norm(r[ok]), k


@pytest.mark.filterwarnings("ignore:invalid value encountered")
@pytest.mark.parametrize("name", sorted(CHAINS))
def test_infinities_and_nans_through_two_layers(name):
    """The same through the maps and deltas that the epilogues write."""
    wl = CHAINS[name]
    x, params, dy = draw_single(wl)
    x[0, 5, 10, 12], x[1, 7, 9, 30], x[0, 9, 15, 40], x[1, 3, 0, 0] = np.inf, -np.inf, np.nan, np.inf
    dy[1, 5, 20, 16], dy[0, 9, 2, 3] = np.inf, np.nan
    ref, got = run_oracle(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy)
    assert_split(got["plan"], wl.layers)
    for k in ("y", "dx"):
        assert np.array_equal(classes(got[k]), classes(ref[k])), k
        ok = np.isfinite(ref[k])
        assert ok.any() and not ok.all()
    assert np.isnan(got["dparams"]).any()


@pytest.mark.parametrize("pooled", [False, True])
@pytest.mark.parametrize("cin", [32, 256])
def test_the_largest_finite_values_between_layers(cin, pooled):
    """A first layer that hands its input on (1x1, identity), so that its epilogue writes values next to the largest fp32."""
    h, w = (200, 64) if cin == 32 else (50, 52)
    layers = (conv(cin, 256, 1),) + ((pool(),) if pooled else ()) + (conv(256, 64, 1),)
    wl = W("r", layers, 2, cin, h, w, (2, 2), one(len(layers)))
    x, params, dy = draw_single(wl)
    params[:256 * cin] = np.eye(256, cin, dtype=np.float32).ravel()
    params[256 * cin:256 * cin + 256] = 0
    params[256 * cin + 256:] *= np.float32(2.0 ** -20)
    x[:, :, 3:9, 5:9] = np.float32(3.395e38) * np.random.default_rng(2).choice(np.float32([1, -1, 0.999]), x[:, :, 3:9, 5:9].shape)
    ref, got = run_oracle(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy)
    assert_split(got["plan"], wl.layers)
    for k in ("y", "dx"):
        assert np.isfinite(got[k]).all(), k
        scale = np.abs(ref[k]).max()
        assert np.linalg.norm((got[k] - ref[k]) / scale) <= 2 * 7 * 2.0 ** -23 * np.linalg.norm(ref[k] / scale), k


@pytest.mark.parametrize("name", sorted(SINGLE))
def test_the_largest_finite_values(name):
    """Inputs within 2^-7 of the largest fp32: their first part is cut instead of rounded up to infinity (bound: see the module's
    docstring, one convolution, and 2^-23 for the bit that the three parts of a cut value may lack)."""
    wl = SINGLE[name]
    x, params, dy = draw_single(wl)
    x[:, :, 3:9, 5:9] = np.float32(3.395e38) * np.random.default_rng(2).choice(np.float32([1, -1, 0.999]), x[:, :, 3:9, 5:9].shape)
    params *= np.float32(2.0 ** -20)
    ref, got = run_oracle(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy)
    assert_split(got["plan"], wl.layers)
    for k in ("y", "dx"):
        assert np.isfinite(got[k]).all(), k
        scale = np.abs(ref[k]).max()
        assert np.linalg.norm((got[k] - ref[k]) / scale) <= 7 * 2.0 ** -23 * np.linalg.norm(ref[k] / scale), k


@pytest.mark.parametrize("name", ["chain", "chain-pool", "chain-32", "chain-32-pool"])
def test_the_smallest_positive_values_count_as_positive(name):
    """Outputs of a first layer down to the smallest fp32 (its input is zero, its bias tiny, of either sign): the derivative of the
    layer is decided by their sign."""
    wl = synth.with_slope(CHAINS[name], 0.25)
    x, params, dy = draw_single(wl)
    x[:] = 0
    l = wl.layers[0]
    at, c = l.cout * l.cin * l.k * l.k, np.arange(l.cout)
    params[at:at + l.cout] = np.where(c % 2, -1, 1) * np.float32(2.0) ** (-149 + c // 2).astype(np.float32)
    assert (params[at:at + l.cout] != 0).all()
    ref, got = run_oracle(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy)
    assert_split(got["plan"], wl.layers)
    assert rel_err(got["dx"], ref["dx"]) <= FP32_TOL
    assert rel_err(got["dparams"], ref["dparams"]) <= FP32_TOL


def test_activations_do_not_depend_on_grid_profile_or_batch_split():
    """Above the 1e8 rule, what the test of the same kind in test_gpu_parity.py shows below it: the same bits in the last map under
    every tile grid and profile that leaves each layer on its kernels, gradients to 1e-5 (sums in another order), the same bits
    from run to run; an image gives the same bits alone and in a batch.  Profiles that fuse layers run on other kernels: then
    the maps agree within both sides' rounding."""
    wl = STACKS["stack-8-ragged"].with_(groups=one(8))
    convs = sum(l.kind == "conv" for l in wl.layers)
    x, params, _ = synth.draw(wl, bias_std=0.1)
    dy = np.random.default_rng(1).standard_normal((wl.N,) + tuple(synth.map_shapes(wl.layers, wl.C, wl.H, wl.W)[-1])).astype(np.float32)
    base, again = run_gpu(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy)
    assert_split(base["plan"], wl.layers)
    for k in ("y", "dx", "dparams"):
        assert np.array_equal(base[k], again[k]), f"{k} differs from run to run"
    variants = [dict(grid=(1, 1)), dict(grid=(4, 2), groups=((1, 4), (5, 8))), dict(grid=(2, 5), groups=synth.groups_per_layer(wl.layers)),
                dict(grid=(11, 17), groups=synth.groups_per_maxpool(wl.layers)), dict(opts=dict(max_group_convs=1)),
                dict(opts=dict(cost_model=1))]
    for v in variants:
        opts = v.get("opts", {})
        got = run_gpu(wl.with_(**{k: v[k] for k in v if k != "opts"}), x, params, dy=dy, **opts)
        assert_split(got["plan"], wl.layers)
        assert np.array_equal(got["y"], base["y"]), v
        assert rel_err(got["dx"], base["dx"]) <= 1e-5, v
        assert rel_err(got["dparams"], base["dparams"]) <= 1e-5, v
    for n in range(wl.N):
        alone = run_gpu(wl.with_(N=1), x[n:n + 1], params, dy=dy[n:n + 1])
        assert np.array_equal(alone["y"][0], base["y"][n])
        assert np.array_equal(alone["dx"][0], base["dx"][n])
    for opts in (dict(strict_groups=True), dict(cost_model=-1), dict(stationary=-1), dict(stationary=1)):
        got = run_gpu(wl, x, params, dy=dy, **opts)
        assert kernels(got["plan"]) != kernels(base["plan"])
        d = np.linalg.norm((got["y"] - base["y"]).astype(np.float64)) / np.linalg.norm(base["y"].astype(np.float64))
        assert d <= 2 * convs * 6 * 2.0 ** -23, opts


@pytest.mark.parametrize("name", sorted(STACKS))
def test_results_do_not_depend_on_what_the_workspace_held(name):
    """Tiles read around the maps they are about: zeros, NaNs or large values there leave the same bits in every result."""
    wl = STACKS[name]
    x, params, target = synth.draw(wl, bias_std=0.1)
    plan = ftp.ftp_plan(wl.layers, wl.N, wl.C, wl.H, wl.W, wl.grid, wl.groups)
    xd, pd, td = (torch.from_numpy(a).cuda() for a in (x, params, target))
    results = []
    for fill in (0x00, 0xff, 0x7e):                          # 0x7e7e7e7e is 8e37, its halves as bf16 too
        ws = plan.new_workspace().fill_(fill)
        y, grad, dx = torch.empty_like(td), torch.empty_like(pd), torch.empty_like(xd)
        ftp.ftp_forward(plan, xd, pd, y, ws)
        ftp.ftp_step_grad(plan, xd, pd, grad, ws, target=td, dx=dx)
        plan.check(ws)
        results.append((y, grad, dx))
    for r in results[1:]:
        assert all(torch.equal(a, b) for a, b in zip(results[0], r))


def norm_err(a, o):
    return float(np.linalg.norm((np.asarray(a, np.float64) - o).ravel()) / np.linalg.norm(np.asarray(o).ravel()))


def window_sums(src, filters, pos):
    """fp64 sums of 3x3 windows of `src` [N, C, H, W] at the positions `pos` (n, y, x arrays) with `filters` [rows, C, 3, 3]."""
    n, y, x = pos
    H, W_ = src.shape[2:]
    out = np.zeros((len(n), filters.shape[0]))
    for ky in range(3):
        for kx in range(3):
            yy, xx = y + ky - 1, x + kx - 1
            ok = (yy >= 0) & (yy < H) & (xx >= 0) & (xx < W_)
            v = src[n, :, np.clip(yy, 0, H - 1), np.clip(xx, 0, W_ - 1)].astype(np.float64) * ok[:, None]
            out += v @ filters[:, :, ky, kx].astype(np.float64).T
    return out


@pytest.mark.parametrize("cin", [32, 64])
def test_many_items_and_stages_a_block(cin):
    """Blocks that take many items (the second halves of the accumulators, the flags of alternate items) and many stages of the
    filter gradient (accumulators of the small products that are emptied every 64 stages) on values with all 24 bits, of
    one sign in the filter gradient, so that truncation would add up: sampled positions and filters against fp64, within the
    docstring's bound for one convolution, and no further off than one and a half times the multiply-add kernels."""
    N, H, W_, cout = (28 if cin == 32 else 16), 304, 304, 64
    rng = np.random.default_rng(3)
    x = rng.random((N, cin, H, W_), dtype=np.float32)
    dy = rng.random((N, cout, H, W_), dtype=np.float32)
    params = np.concatenate([rng.standard_normal(cout * cin * 9) * (2 / (9 * cin)) ** 0.5, rng.standard_normal(cout) * 0.1]).astype(np.float32)
    filters = params[:cout * cin * 9].reshape(cout, cin, 3, 3)
    pos = [rng.integers(0, k, 3000) for k in (N, H, W_)]
    pos[1][:100], pos[2][100:200], pos[1][200:300], pos[2][300:400] = 0, 0, H - 1, W_ - 1
    cos, cis = [0, 17, 63], [0, 5, cin - 1]
    ref_y = window_sums(x, filters, pos) + params[cout * cin * 9:]
    ref_dx = window_sums(dy, np.flip(filters, (2, 3)).transpose(1, 0, 2, 3), pos)
    ref_dw = np.zeros((3, 3, 3, 3))
    for a, co in enumerate(cos):
        d = dy[:, co].astype(np.float64)
        for b, ci in enumerate(cis):
            xp = np.pad(x[:, ci].astype(np.float64), ((0, 0), (1, 1), (1, 1)))
            for ky in range(3):
                for kx in range(3):
                    ref_dw[a, b, ky, kx] = np.vdot(d, xp[:, ky:ky + H, kx:kx + W_])
    ref_db = dy.astype(np.float64).sum((0, 2, 3))
    err = {}
    for kind, opts in (("split", {}), ("rows", dict(stationary=1))):
        wl = W("s", (conv(cin, cout, 3, leaky=1.0),), N, cin, H, W_, (2, 2), one(1))
        got = run_gpu(wl, x, params, dy=dy, **opts)
        if kind == "split":
            assert_split(got["plan"], wl.layers)
            assert N * (H + 1) * (W_ + 1) / 1024 > 2 * 148                        # an item is at most 8 blocks of 128 entries
            assert (N * (H + 1) - 1) * (W_ + 1) / 64 / got["plan"].group_mode(0)[1] > 128   # stages of 64 entries at most; a set is a share of them
        dw = got["dparams"][:cout * cin * 9].reshape(cout, cin, 3, 3)[np.ix_(cos, cis)]
        err[kind] = [norm_err(got["y"][pos[0], :, pos[1], pos[2]], ref_y), norm_err(got["dx"][pos[0], :, pos[1], pos[2]], ref_dx),
                     norm_err(dw, ref_dw), norm_err(got["dparams"][cout * cin * 9:], ref_db)]
    for s, r in zip(err["split"], err["rows"]):
        assert s <= max(6 * 2.0 ** -23, 1.5 * r), err


@pytest.mark.parametrize("cin", [512, 1024])
def test_long_contractions_of_one_sign(cin):
    """9 x 512 and 9 x 1024 terms a sum, all positive: what truncation takes from the accumulators of an item has one sign."""
    wl = W("t", (conv(cin, 64, 3, leaky=1.0),), 2, cin, 26, 24, (2, 2), one(1))
    rng = np.random.default_rng(5)
    x = rng.random((2, cin, 26, 24), dtype=np.float32)
    dy = rng.random((2, 64, 26, 24), dtype=np.float32)
    params = rng.random(64 * cin * 9 + 64, dtype=np.float32) * np.float32(1 / cin)
    ref = run_oracle(wl, x, params, dy=dy)
    got, fma = run_gpu(wl, x, params, dy=dy), run_gpu(wl, x, params, dy=dy, stationary=1)
    assert_split(got["plan"], wl.layers)
    err = {k: (norm_err(got[k], ref[k]), norm_err(fma[k], ref[k])) for k in ("y", "dx", "dparams")}
    for s, r in err.values():
        assert s <= max(6 * 2.0 ** -23, 1.5 * r), err


@pytest.mark.parametrize("name", ["stack-8-ragged", "stack-16", "wide-map"])
def test_whole_stacks_are_as_close_to_fp64_as_the_multiply_add_kernels(name):
    """Leaky slopes, pools, ordinary data: distance from fp64 in the 2-norm, the median over seven draws (about one draw in five
    has a near-tie of a pool or a sign that either arithmetic decides against fp64; that moves a whole delta and says
    nothing about the sums)."""
    wl = STACKS[name]
    convs = sum(l.kind == "conv" for l in wl.layers)
    err = {"split": [], "rows": []}
    for seed in range(100, 107):
        w = wl.with_(seed=seed)
        x, params, _ = synth.draw(w, bias_std=0.1)
        shape = (w.N,) + tuple(synth.map_shapes(w.layers, w.C, w.H, w.W)[-1])
        dy = np.random.default_rng(seed).standard_normal(shape).astype(np.float32)
        ref = run_oracle(w, x, params, dy=dy)
        for kind, opts in (("split", {}), ("rows", dict(stationary=1))):
            got = run_gpu(w, x, params, dy=dy, **opts)
            assert (kind == "split") == any("split" in k for k in kernels(got["plan"]).values())
            err[kind].append([norm_err(got[k], ref[k]) for k in ("y", "dx", "dparams")])
    split, rows = (np.median(np.array(err[k]), axis=0) for k in ("split", "rows"))
    assert (split <= 1.1 * rows).all()
    assert (split <= 6 * 2.0 ** -23 * convs * np.array([1, 2, 2])).all()
