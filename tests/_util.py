"""Shared helpers of the GPU parity tests: run the CUDA path through the C-ABI
binding and the fp64 oracle on the same seeded inputs and compare per tensor."""
import numpy as np
import torch

import paper_2409_09083_b200 as ftp
from oracle import reference as orc
from paper_2409_09083_b200 import synth

# Tolerance of the fp32 path: per tensor, max_i |a_i - o_i| / max_j |o_j| <= 1e-4.
FP32_TOL = 1e-4


def rel_err(a, o):
    a = np.asarray(a, dtype=np.float64)
    o = np.asarray(o, dtype=np.float64)
    scale = np.abs(o).max()
    if scale == 0.0:
        return float(np.abs(a).max())
    return float(np.abs(a - o).max() / scale)


def run_gpu(wl, x, params, target=None, dy=None, want_dx=True, **plan_opts):
    """forward + backward through the library; returns dict of numpy arrays."""
    dev = "cuda"
    plan = ftp.ftp_plan(wl.layers, x.shape[0], wl.C, wl.H, wl.W, wl.grid, wl.groups, **plan_opts)
    ws = plan.new_workspace(dev)
    xd = torch.from_numpy(x).to(dev)
    pd = torch.from_numpy(params).to(dev)
    c, h, w = synth.map_shapes(wl.layers, wl.C, wl.H, wl.W)[-1]
    y = torch.empty((x.shape[0], c, h, w), dtype=torch.float32, device=dev)
    ftp.ftp_forward(plan, xd, pd, y, ws)
    torch.cuda.synchronize()
    yh = y.cpu().numpy()
    if dy is None:
        M = yh.size
        dy = (2.0 * (yh.astype(np.float64) - target.astype(np.float64)) / M).astype(np.float32)
    dyd = torch.from_numpy(np.ascontiguousarray(dy)).to(dev)
    dx = torch.empty_like(xd) if want_dx else None
    dparams = torch.empty_like(pd)
    ftp.ftp_backward(plan, xd, dyd, pd, dx, dparams, ws)
    torch.cuda.synchronize()
    return dict(plan=plan, y=yh, dy=dy, dx=None if dx is None else dx.cpu().numpy(),
                dparams=dparams.cpu().numpy())


def run_gpu_step(wl, x, params, target, lr, want_dx=True, **plan_opts):
    dev = "cuda"
    plan = ftp.ftp_plan(wl.layers, x.shape[0], wl.C, wl.H, wl.W, wl.grid, wl.groups, **plan_opts)
    ws = plan.new_workspace(dev)
    xd = torch.from_numpy(x).to(dev)
    pd = torch.from_numpy(params.copy()).to(dev)
    td = torch.from_numpy(target).to(dev)
    loss = torch.zeros(1, dtype=torch.float32, device=dev)
    dx = torch.empty_like(xd) if want_dx else None
    ftp.ftp_step(plan, xd, pd, lr, ws, target=td, loss_out=loss, dx=dx)
    torch.cuda.synchronize()
    return dict(plan=plan, loss=float(loss.item()), new_params=pd.cpu().numpy(),
                dx=None if dx is None else dx.cpu().numpy())


def run_oracle(wl, x, params, target=None, dy=None, lr=0.0, store=None):
    return orc.step(list(wl.layers), x.astype(np.float64), params.astype(np.float64), lr,
                    target=None if target is None else target.astype(np.float64),
                    dy=None if dy is None else dy.astype(np.float64), store=store)


def bf16_grid(a):
    """The same array with every value moved to the nearest bfloat16 (still float32): inputs that a
    bf16 path and the oracle can both take without an input-rounding difference."""
    return torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).to(torch.bfloat16).to(torch.float32).numpy()


def per_layer_errors(layers, got, ref):
    """Relative error of each conv layer's filter and bias gradient."""
    out = []
    for i, (g, r) in enumerate(zip(orc.unpack_params(layers, got), orc.unpack_params(layers, ref))):
        if g is None:
            continue
        out.append((i + 1, rel_err(g[0], r[0]), rel_err(g[1], r[1])))
    return out


def decision_margin(layers, ref):
    """Smallest relative margin of the discrete decisions the oracle took: |Z| of every
    leaky-ReLU input and the gap between the two largest values of every pooling window, each
    relative to the largest magnitude of its map.  A case whose margin is far above fp32
    rounding takes the same decisions in fp32 and fp64."""
    worst = np.inf
    maps = ref["maps"]
    for i, l in enumerate(layers):
        out = maps[i + 1]
        if l.kind == "conv":
            worst = min(worst, np.abs(out).min() / max(np.abs(out).max(), 1e-300))
        else:
            X = maps[i]
            N, C, H, W = X.shape
            w = X.reshape(N, C, H // 2, 2, W // 2, 2).transpose(0, 1, 2, 4, 3, 5).reshape(N, C, H // 2, W // 2, 4)
            s = np.sort(w, axis=-1)
            worst = min(worst, (s[..., 3] - s[..., 2]).min() / max(np.abs(X).max(), 1e-300))
    return float(worst)


def draw_unambiguous(wl, bias_std=0.5, tau=2e-5, tries=200, store=None):
    """First seed >= wl.seed whose oracle decisions all have a margin above tau; returns
    (workload with that seed, x, params, target, oracle result).  store="bf16": inputs on the
    bf16 grid, oracle with bf16 feature-map storage."""
    for s in range(wl.seed, wl.seed + tries):
        w = wl.with_(seed=s)
        x, params, target = synth.draw(w, bias_std=bias_std)
        if store:
            x, params = bf16_grid(x), bf16_grid(params)
        ref = run_oracle(w, x, params, target=target, store=store)
        if decision_margin(list(w.layers), ref) > tau:
            return w, x, params, target, ref
    raise RuntimeError("no seed with unambiguous decisions found")


def kernels(plan):
    """{layers of an executed group: (kernels of its forward pass, of its backward pass)}."""
    return {g: (plan.group_kernels(i, 0), plan.group_kernels(i, 1)) for i, g in enumerate(plan.exec_groups())}


def assert_split(plan, layers):
    """Every conv layer with a 1x1 or 3x3 window and 32 input channels or more runs on the split kernels (with exactly 32 its
    forward pass on the row kernel), no other layer does."""
    for (a, b), k in kernels(plan).items():
        convs = [l for l in layers[a - 1:b] if l.kind == "conv"]
        if any(l.k in (1, 3) and l.cin >= 32 for l in convs):
            assert len(convs) == 1, (a, b, k)
            assert k == ("rows" if convs[0].cin == 32 else "split", "split"), (a, b, k)
        else:
            assert "split" not in k, (a, b, k)
    assert any("split" in k for k in kernels(plan).values())
