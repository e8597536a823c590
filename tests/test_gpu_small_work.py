"""Gradients of few points (a half-tile of 32 per CTA) equal, bit for bit, the same points in a larger call."""
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
