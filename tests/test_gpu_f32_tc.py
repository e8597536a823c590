"""Gradients and training of FP32 networks on the tensor cores (operands split into 16-bit parts)
against FP64, at the sizes where the tiles can go wrong.

Tolerance.  u = 2^-24.  A sine layer adds a sine error of at most 8u (5e-7) and a contraction whose
rounding stays below 8u of its result's scale; the layers that follow may amplify both by the gain
of an untrained network, taken as 4.  Over k + 1 sine layers the root mean square error of the
gradient is below 64 u (k + 1) of the gradients' root mean square.
"""
import numpy as np
import pytest
import torch

import oracle
from paper_2201_09147_gb300 import inputs

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
NETS = {"64x1": (64, 1, 3), "64x3": (64, 3, 3), "128x2": (128, 2, 3), "256x1": (256, 1, 3), "256x4": (256, 4, 3),
        "128x2_t": (128, 2, 4), "256x3_t": (256, 3, 4)}


def rel_rms(a, b):
    return float(np.sqrt(np.mean((a.astype(np.float64) - b) ** 2) / np.mean(b ** 2)))


def net_bytes(name):
    w, k, d = NETS[name]
    return inputs.net_to_bytes(inputs.siren_init(11, w, k, in_dim=d))


def points(n, seed=5):
    return (2.0 * inputs.uniform01(seed, 3 * n).reshape(3, n) - 1.0).astype(np.float32)


# one point, the edges of a 32-point tile and of a CTA's two tiles, and more tiles than CTAs
@pytest.mark.parametrize("n", [1, 31, 32, 33, 64, 65, 152 * 32 + 1, 2 * 152 * 64 + 33])
@pytest.mark.parametrize("name", ["64x1", "128x2", "256x1", "256x4"])
def test_gradients(sdf, name, n):
    b, pts = net_bytes(name), points(n)
    g = sdf.normals(sdf.Net(b, sdf.SDF_FP32), torch.from_numpy(pts).cuda())
    sdf.sync_status()
    check = np.unique(np.concatenate([np.arange(min(n, 70)), np.arange(max(0, n - 70), n)]))
    ref = oracle.Net(b).grad_batch(pts[:, check].astype(np.float64))
    assert np.isfinite(g.cpu().numpy()).all()
    assert rel_rms(g.cpu().numpy()[:, check], ref) <= 64 * U * (NETS[name][1] + 1)


@pytest.mark.parametrize("name", ["64x3", "128x2_t", "256x3_t"])
def test_masked_and_timed(sdf, name):
    n = 4133
    b, pts = net_bytes(name), points(n)
    mask = (inputs.uniform01(9, n) < 0.3).astype(np.uint8)
    net, p = sdf.Net(b, sdf.SDF_FP32), torch.from_numpy(pts).cuda()
    full = sdf.normal_map(net, p)
    part = sdf.normal_map(net, p, torch.from_numpy(mask).cuda())
    keep = torch.from_numpy(mask.astype(bool)).cuda()
    assert torch.equal(part[:, keep], full[:, keep]) and not part[:, ~keep].any()
    if NETS[name][2] == 4:
        const = sdf.normal_map_timed(net, p, torch.zeros(n, device="cuda"))
        assert rel_rms(const.cpu().numpy(), full.cpu().numpy().astype(np.float64)) <= 64 * U * (NETS[name][1] + 1)
    sdf.sync_status()


def scaled(b, layer, factor):
    """The image of a folded network with hidden layer `layer`'s weights and biases times `factor`."""
    shape, theta = sdfnn_theta(b)
    d, w, k = shape
    o = w * d + w + (layer - 1) * (w * w + w)
    theta = theta.copy()
    theta[o:o + w * w + w] *= np.float32(factor)
    return sdfnn_image(shape, theta)


def sdfnn_theta(b):
    from paper_2201_09147_gb300 import sdfnn
    return sdfnn.theta_from_sdfn(b)


def sdfnn_image(shape, theta):
    from paper_2201_09147_gb300 import sdfnn
    return sdfnn.sdfn_from_theta(shape, theta)


# weights far from 1: 2^-40 is rescaled into half's range; 2^-70 is beyond the scales and takes the
# SIMT kernels.  The network's values are then linear in the scaled layer.
@pytest.mark.parametrize("log2", [-70, -40, -20])
def test_small_weights(sdf, log2):
    b = scaled(net_bytes("128x2"), 2, 2.0 ** log2)
    pts = points(500)
    g = sdf.normals(sdf.Net(b, sdf.SDF_FP32), torch.from_numpy(pts).cuda()).cpu().numpy()
    sdf.sync_status()
    ref = oracle.Net(b).grad_batch(pts.astype(np.float64))
    s = 2.0 ** -log2
    assert rel_rms(g.astype(np.float64) * s, ref * s) <= 64 * U * 3


def reference_training(shape, theta, pts, time, d_f, d_g):
    """f, grad f and dL/dtheta of L = <d_f, f> + <d_g, grad f> in float64 (torch autograd)."""
    d, w, k = shape
    th = torch.from_numpy(theta).double().cuda().requires_grad_(True)
    x = torch.from_numpy(pts).double().cuda()
    if d == 4:
        x = torch.cat([x, torch.from_numpy(time).double().cuda()[None]])
    o, h, g = 0, x, None
    for layer in range(k + 1):
        fan = d if layer == 0 else w
        W, b = th[o:o + w * fan].reshape(w, fan), th[o + w * fan:o + w * fan + w]
        o += w * fan + w
        z = W @ h + b[:, None]
        c, h = torch.cos(z), torch.sin(z)
        g = [W[:, i:i + 1] * c for i in range(3)] if layer == 0 else [(W @ t) * c for t in g]
    f = th[o:o + w] @ h + th[o + w]
    grad = torch.stack([th[o:o + w] @ t for t in g])
    loss = (f * torch.from_numpy(d_f).double().cuda()).sum() + (grad * torch.from_numpy(d_g).double().cuda()).sum()
    return f.detach(), grad.detach(), torch.autograd.grad(loss, th)[0]


# one point, the edges of a K block (16 points), of a tile (32) and of a CTA's two tiles, and a batch whose
# weight-gradient blocks do not divide evenly over the CTAs.  d_theta adds a third contraction (over the batch)
# and the sums of the backward to the forward's errors: 128 u (k + 1).
@pytest.mark.parametrize("n", [1, 15, 17, 33, 64, 65, 3001])
@pytest.mark.parametrize("name", ["64x1", "64x3", "128x2_t", "256x1", "256x4"])
def test_training_gradients(sdf, name, n):
    w, k, d = NETS[name]
    shape, theta = sdfnn_theta(net_bytes(name))
    pts, time = points(n), inputs.uniform01(7, n).astype(np.float32)
    z = (2.0 * inputs.uniform01(8, 4 * n) - 1.0).astype(np.float32) / n
    d_f, d_g = z[:n].copy(), z[n:].reshape(3, n).copy()
    dev = lambda a: torch.from_numpy(a).cuda()
    th, tm = dev(theta), dev(time) if d == 4 else None
    f, g, ws = sdf.train_forward(shape, th, dev(pts), pt_time=tm)
    d_theta = sdf.train_backward(shape, th, dev(pts), dev(d_f), dev(d_g), ws, pt_time=tm)
    sdf.sync_status()
    rf, rg, rt = reference_training(shape, theta, pts, time, d_f, d_g)
    host = lambda t: t.cpu().numpy().astype(np.float64)
    assert rel_rms(host(f), host(rf)) <= 64 * U * (k + 1)
    assert rel_rms(host(g), host(rg)) <= 64 * U * (k + 1)
    assert rel_rms(host(d_theta), host(rt)) <= 128 * U * (k + 1)
