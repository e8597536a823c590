"""Calls of few points or rays, which run on other launch shapes or kernels, equal, bit for bit, the
same points or rays in a larger call."""
import numpy as np
import pytest
import torch

from paper_2201_09147_gb300 import inputs

pytestmark = pytest.mark.gpu

SMS32 = 152 * 32  # points of one half-tile on every SM: the most that are spread that way


@pytest.mark.parametrize("n", [1, 31, 33, 300, SMS32 - 31, SMS32, SMS32 + 1])
@pytest.mark.parametrize("width,hidden,precision", [(64, 1, "SDF_BF16"), (128, 2, "SDF_FP8"), (256, 3, "SDF_FP16")])
def test_spread_points_match_a_larger_call(sdf, width, hidden, precision, n):
    net = sdf.Net(inputs.net_to_bytes(inputs.siren_init(3, width, hidden)), getattr(sdf, precision))
    pts = torch.from_numpy(inputs.random_points(4, 3 * SMS32)).cuda()
    few = pts[:, :n].contiguous()
    mask = torch.zeros(pts.shape[1], dtype=torch.uint8, device="cuda")
    mask[:n] = 1
    ref = sdf.normals(net, pts)
    assert torch.equal(sdf.normals(net, few), ref[:, :n])
    unit = sdf.normal_map(net, pts)
    assert torch.equal(sdf.normal_map(net, few), unit[:, :n])
    masked = sdf.normal_map(net, pts, mask)
    assert torch.equal(masked[:, :n], unit[:, :n]) and not masked[:, n:].any()
    sdf.sync_status()


# Rays: width 64 changes kernel at 256 rays per SM, width 256 its tiles at 128 per SM; a whole of 300 per SM
# against parts at the edges of a 128-ray tile and of both lines.
RAYS = 300 * 152


@pytest.mark.parametrize("width,hidden,in_dim,precision", [
    (64, 1, 3, "SDF_BF16"), (64, 3, 4, "SDF_FP16"), (128, 2, 3, "SDF_FP16"), (128, 1, 4, "SDF_BF16"),
    (256, 2, 3, "SDF_BF16"), (256, 1, 4, "SDF_FP16"), (256, 2, 3, "SDF_FP8"), (64, 2, 4, "SDF_FP32"),
    (128, 2, 3, "SDF_FP32"), (256, 1, 4, "SDF_FP32")])
def test_few_rays_match_a_larger_call(sdf, width, hidden, in_dim, precision):
    b = inputs.net_to_bytes(inputs.siren_init(5, width, hidden, in_dim=in_dim, out_scale=30.0, out_shift=0.1))
    net = sdf.Net(b, getattr(sdf, precision))
    u = inputs.uniform01(31, 5 * RAYS).reshape(5, RAYS)
    orig = np.stack([3.0 * u[0] - 1.5, 3.0 * u[1] - 1.5, np.full(RAYS, 2.5)])
    d = np.stack([u[2] - 0.5, u[3] - 0.5, np.zeros(RAYS)]) - orig
    orig, d = (torch.from_numpy(x.astype(np.float32)).cuda() for x in (orig, d / np.linalg.norm(d, axis=0)))
    time = torch.from_numpy(u[4].astype(np.float32)).cuda() if in_dim == 4 else None

    def trace(a, e):
        return sdf.trace_multiscale([net], [0.0], [9], 1e-2, orig[:, a:e].contiguous(), d[:, a:e].contiguous(),
                                    step_scale=[0.7], ray_time=None if time is None else time[a:e].contiguous())

    whole = trace(0, RAYS)
    assert 0 < int(whole[2].sum()) < RAYS
    a = 0
    for n in (1, 127, 129, 1000, 128 * 152 - 1, 128 * 152 + 1):
        pos, t, hit, iters = trace(a, a + n)
        assert torch.equal(pos, whole[0][:, a:a + n]) and torch.equal(t, whole[1][a:a + n])
        assert torch.equal(hit, whole[2][a:a + n]) and torch.equal(iters, whole[3][a:a + n])
        a += n
    sdf.sync_status()
