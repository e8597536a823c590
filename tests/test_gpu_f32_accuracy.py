"""FP32 gradients and training on the tensor cores against the same networks' FMA chains
(sdf_fit_forward), on networks whose layers are far from those of an untrained SIREN.

Tolerance.  Both paths share the layers' sines (their error) and the networks; the split operands miss a
float by half a unit at most and their products are summed with fewer roundings than the chain's.  So the
root mean square error against FP64 is at most 1.5 times the chain's (one and a half: two samples of errors
of a size), plus u = 2^-24 of the gradients' root mean square for the roundings after the last layer.
"""
import numpy as np
import pytest
import torch

from paper_2201_09147_gb300 import inputs, sdfnn
from test_gpu_f32_tc import reference_training

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def rms(x):
    return float(np.sqrt(np.mean(np.square(x, dtype=np.float64))))


def points(n, seed=5):
    return (2.0 * inputs.uniform01(seed, 3 * n).reshape(3, n) - 1.0).astype(np.float32)


def layers(shape, theta):
    """Views of theta: the hidden layers' (W, b), and the weights that read each (the next layer's, or w_out)."""
    d, w, k = shape
    o, ws, bs = w * d + w, [], []
    for _ in range(k):
        ws.append(theta[o:o + w * w].reshape(w, w))
        bs.append(theta[o + w * w:o + w * w + w])
        o += w * w + w
    return ws, bs, theta[o:o + w]


def unbalanced(width, hidden, s):
    """A SIREN in which one unit of every hidden layer has its weights times s and the weights that read it over s."""
    shape, theta = sdfnn.theta_from_sdfn(inputs.net_to_bytes(inputs.siren_init(11, width, hidden)))
    theta = theta.copy()
    ws, _, out = layers(shape, theta)
    for l in range(hidden):
        j = (37 * l + 5) % width
        ws[l][j] *= np.float32(s)
        if l + 1 < hidden:
            ws[l + 1][:, j] /= np.float32(s)
        else:
            out[j] /= np.float32(s)
    return shape, theta


def small_layers(width, hidden, exponents):
    """A SIREN with hidden layer l's weights and biases times 2^exponents[l]."""
    shape, theta = sdfnn.theta_from_sdfn(inputs.net_to_bytes(inputs.siren_init(11, width, hidden)))
    theta = theta.copy()
    ws, bs, _ = layers(shape, theta)
    for w, b, e in zip(ws, bs, exponents):
        w *= np.float32(2.0 ** e)
        b *= np.float32(2.0 ** e)
    return shape, theta


def compare_training(shape, theta, n=3001):
    """f, grad f and dL/dtheta of sdf_train_forward / _backward are as near to FP64 as those of the FMA chains'
    forward and the same backward."""
    pts = points(n)
    z = (2.0 * inputs.uniform01(8, 4 * n) - 1.0).astype(np.float32) / n
    d_f, d_g = z[:n].copy(), z[n:].reshape(3, n).copy()
    dev = lambda a: torch.from_numpy(a).cuda()
    th, x = dev(theta), dev(pts)

    def run(entry):
        f, g, ws = sdfnn._forward(entry, shape, th, x, None, None, None, sdfnn.SDF_FP32)
        d = sdfnn.train_backward(shape, th, x, dev(d_f), dev(d_g), ws)
        return [t.cpu().numpy().astype(np.float64) for t in (f, g, d)]

    tc, fma = run(sdfnn.lib().sdf_train_forward), run(sdfnn.lib().sdf_fit_forward)
    sdfnn.sync_status()
    ref = [t.cpu().numpy() for t in reference_training(shape, theta, pts, None, d_f, d_g)]
    # (b_out, the last entry, is a plain sum of d_f in the order of atomics on both sides)
    tc[2], fma[2], ref[2] = tc[2][:-1], fma[2][:-1], ref[2][:-1]
    for name, a, b, r in zip(("f", "grad f", "dL/dtheta"), tc, fma, ref):
        assert np.isfinite(a).all(), name
        assert rms(a - r) <= 1.5 * rms(b - r) + U * rms(r), name


@pytest.mark.parametrize("s", [1.0, 16.0, 32.0, 1024.0])
@pytest.mark.parametrize("width,hidden", [(64, 2), (128, 3), (256, 4)])
def test_training_of_unbalanced_networks(sdf, width, hidden, s):
    compare_training(*unbalanced(width, hidden, s))


# a layer at 2^-70 alone, and layers whose product is (beyond a half's exponents, or a scale of 2^60)
@pytest.mark.parametrize("exponents", [(0, -70), (-40, -40), (-25, -25), (20, -50)])
def test_training_of_small_layers(sdf, exponents):
    compare_training(*small_layers(128, 2, exponents))


@pytest.mark.parametrize("width,hidden", [(64, 3), (128, 2), (256, 2)])
def test_repeated_calls_give_the_same_bits(sdf, width, hidden):
    """The chains of products meet in a fixed order: nothing may depend on how instructions overlap.  (16 points: one
    CTA adds to each entry of dL/dtheta.)"""
    shape, theta = unbalanced(width, hidden, 1.0)
    th, net = torch.from_numpy(theta).cuda(), sdf.Net(sdfnn.sdfn_from_theta(shape, theta), sdf.SDF_FP32)
    for n in (16, 20011):
        x = torch.from_numpy(points(n)).cuda()
        c = torch.from_numpy((2.0 * inputs.uniform01(8, 4 * n) - 1.0).astype(np.float32)).cuda()
        first = None
        for _ in range(20):
            f, g, ws = sdf.train_forward(shape, th, x)
            out = [sdf.normals(net, x), f, g]
            if n == 16:
                out.append(sdf.train_backward(shape, th, x, c[:n].contiguous(), c[n:].reshape(3, n).contiguous(), ws))
            first = first or out
            assert all(torch.equal(a, b) for a, b in zip(out, first))
    sdf.sync_status()


@pytest.mark.parametrize("s", [1.0, 16.0, 32.0, 1024.0, 2.0 ** 18])
@pytest.mark.parametrize("width,hidden", [(64, 2), (128, 3), (256, 4)])
def test_normals_of_unbalanced_networks(sdf, width, hidden, s):
    """The last factor is beyond the scales of the split operands: the network runs on the FMA units."""
    shape, theta = unbalanced(width, hidden, s)
    pts = points(3001)
    x = torch.from_numpy(pts).cuda()
    g = sdf.normals(sdf.Net(sdfnn.sdfn_from_theta(shape, theta), sdf.SDF_FP32), x).cpu().numpy().astype(np.float64)
    fma = sdfnn._forward(sdfnn.lib().sdf_fit_forward, shape, torch.from_numpy(theta).cuda(), x, None, None, None,
                         sdfnn.SDF_FP32)[1].cpu().numpy().astype(np.float64)
    sdf.sync_status()
    zero = np.zeros(3001, np.float32)
    ref = reference_training(shape, theta, pts, None, zero, np.zeros((3, 3001), np.float32))[1].cpu().numpy()
    assert rms(g - ref) <= 1.5 * rms(fma - ref) + U * rms(ref)


def permuted(width, hidden):
    """Hidden layers that pass one unit on to one unit: contractions of a single product, where a correction of the
    mean error of long sums would show as a gain."""
    shape, theta = sdfnn.theta_from_sdfn(inputs.net_to_bytes(inputs.siren_init(11, width, hidden)))
    theta = theta.copy()
    for l, w in enumerate(layers(shape, theta)[0]):
        w[:] = 0.0
        w[np.arange(width), (5 * np.arange(width) + 3 * l) % width] = 0.75
    return shape, theta


# A product alone is rounded to within u of itself and a sum of such products in either direction: over k + 1 layers
# the gain stays within u (k + 1) of the FMA chains' (the sines' error is common to both), with the backward's and
# the weight gradients' contractions within 3 u (k + 1) of it.
@pytest.mark.parametrize("width,hidden", [(64, 3), (128, 4), (256, 4)])
def test_single_products_have_no_gain(sdf, width, hidden):
    shape, theta = permuted(width, hidden)
    n = 4096
    pts = points(n)
    z = (2.0 * inputs.uniform01(8, 4 * n) - 1.0).astype(np.float32) / n
    d_f, d_g = z[:n].copy(), z[n:].reshape(3, n).copy()
    dev = lambda a: torch.from_numpy(a).cuda()
    th, x = dev(theta), dev(pts)
    host = lambda t: t.cpu().numpy().astype(np.float64)
    normals = host(sdf.normals(sdf.Net(sdfnn.sdfn_from_theta(shape, theta), sdf.SDF_FP32), x))
    f, g, ws = sdf.train_forward(shape, th, x)
    d = host(sdf.train_backward(shape, th, x, dev(d_f), dev(d_g), ws))
    _, fma, _ = sdfnn._forward(sdfnn.lib().sdf_fit_forward, shape, th, x, None, None, None, sdfnn.SDF_FP32)
    sdf.sync_status()
    _, rg, rd = (t.cpu().numpy() for t in reference_training(shape, theta, pts, None, d_f, d_g))
    gain = lambda a, r: float((a * r).sum() / (r * r).sum()) - 1.0
    base, tol = gain(host(fma), rg), U * (hidden + 1)
    assert abs(gain(normals, rg) - base) <= tol
    assert abs(gain(host(g), rg) - base) <= tol
    assert abs(gain(d, rd) - base) <= 3 * tol


def test_accuracy_of_the_split_products(sdf):
    """On untrained SIRENs of every width: gradients and training against the FMA chains, and every block of
    dL/dtheta against a plain FP32 evaluation.  That one has the sines of the math library; the kernels' sines are
    off by up to 8 u each, so a block may be off by 8 u (k + 1) of its root mean square more than twice its error."""
    for width, hidden in [(64, 1), (128, 2), (256, 1), (256, 3)]:
        shape, theta = unbalanced(width, hidden, 1.0)
        compare_training(shape, theta, n=6001)
        n = 6001
        pts = points(n)
        z = (2.0 * inputs.uniform01(8, 4 * n) - 1.0).astype(np.float32) / n
        d_f, d_g = z[:n].copy(), z[n:].reshape(3, n).copy()
        dev = lambda a: torch.from_numpy(a).cuda()
        th, x = dev(theta), dev(pts)
        _, _, ws = sdf.train_forward(shape, th, x)
        d = sdf.train_backward(shape, th, x, dev(d_f), dev(d_g), ws).cpu().numpy().astype(np.float64)
        plain = plain_training(shape, theta, pts, d_f, d_g).cpu().numpy().astype(np.float64)
        ref = reference_training(shape, theta, pts, None, d_f, d_g)[2].cpu().numpy()
        o, bounds = 0, []
        for fan in [3] + [width] * hidden:
            bounds += [(o, o + width * fan), (o + width * fan, o + width * fan + width)]
            o += width * fan + width
        bounds += [(o, o + width), (o + width, o + width + 1)]
        for lo, hi in bounds[:-1]:  # (b_out is a plain sum of d_f)
            r = ref[lo:hi]
            assert rms(d[lo:hi] - r) <= 2.0 * rms(plain[lo:hi] - r) + 8 * U * (hidden + 1) * rms(r), (width, hidden, lo)


def plain_training(shape, theta, pts, d_f, d_g):
    """dL/dtheta in FP32 by torch's own operations."""
    d, w, k = shape
    torch.backends.cuda.matmul.allow_tf32 = False
    th = torch.from_numpy(theta).cuda().requires_grad_(True)
    o, h, g = 0, torch.from_numpy(pts).cuda(), None
    for layer in range(k + 1):
        fan = d if layer == 0 else w
        W, b = th[o:o + w * fan].reshape(w, fan), th[o + w * fan:o + w * fan + w]
        o += w * fan + w
        z = W @ h + b[:, None]
        c, h = torch.cos(z), torch.sin(z)
        g = [W[:, i:i + 1] * c for i in range(3)] if layer == 0 else [(W @ t) * c for t in g]
    f = th[o:o + w] @ h + th[o + w]
    grad = torch.stack([th[o:o + w] @ t for t in g])
    loss = (f * torch.from_numpy(d_f).cuda()).sum() + (grad * torch.from_numpy(d_g).cuda()).sum()
    return torch.autograd.grad(loss, th)[0]
