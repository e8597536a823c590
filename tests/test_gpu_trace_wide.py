"""The trace kernel with several threads per ray at the ends of its work: levels without a step, and
tails whose rays end turns apart, in which the warps of a CTA see the list run dry at different times."""
import numpy as np
import pytest
import torch

from paper_2201_09147_gb300 import inputs

pytestmark = pytest.mark.gpu

# one tile, and (width 256) two tiles that regroup their rays; 128 and 256 rays per SM on any part
CASES = [(64, 2, 3, "SDF_BF16"), (64, 1, 4, "SDF_FP16"), (128, 2, 3, "SDF_FP16"), (256, 1, 3, "SDF_BF16"),
         (256, 2, 4, "SDF_FP16"), (256, 3, 3, "SDF_FP8")]


def rays(n, in_dim):
    u = inputs.uniform01(17, 5 * n).reshape(5, n)
    orig = np.stack([3.0 * u[0] - 1.5, 3.0 * u[1] - 1.5, np.full(n, 2.5)])
    d = np.stack([u[2] - 0.5, u[3] - 0.5, np.zeros(n)]) - orig
    orig, d = (torch.from_numpy(x.astype(np.float32)).cuda() for x in (orig, d / np.linalg.norm(d, axis=0)))
    return orig, d, torch.from_numpy(u[4].astype(np.float32)).cuda() if in_dim == 4 else None


@pytest.mark.parametrize("per_sm", [5, 127, 131, 300])
@pytest.mark.parametrize("width,hidden,in_dim,precision", CASES)
def test_levels_without_a_step_change_nothing(sdf, width, hidden, in_dim, precision, per_sm):
    """A level of cap 0 before, between or after others passes its rays on: the same bits as without it (a last
    level of cap 0 leaves no hit).  Caps of 1 to 61 end the rays of a tile together or far apart."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count + 7
    b = inputs.net_to_bytes(inputs.siren_init(5, width, hidden, in_dim=in_dim, out_scale=30.0, out_shift=0.1))
    net = sdf.Net(b, getattr(sdf, precision))
    orig, d, time = rays(n, in_dim)

    def trace(caps):
        k = len(caps)
        return sdf.trace_multiscale([net] * k, [0.01] * (k - 1) + [0.0], caps, 1e-2, orig, d, step_scale=[0.3] * k, ray_time=time)

    for cap in (1, 9, 61):
        one = trace([cap])
        assert 0 < int(one[2].sum()) < n or cap == 1
        for caps in ([0, cap], [0, 0, cap]):
            assert all(torch.equal(x, y) for x, y in zip(trace(caps), one))
        assert all(torch.equal(x, y) for x, y in zip(trace([cap]), one))
    none = trace([0])
    assert not none[2].any() and not none[3].cpu().numpy().any()
    after = trace([9, 0])
    assert not after[2].any()
    sdf.sync_status()


@pytest.mark.parametrize("per_sm", [1, 31, 33, 64, 97])
@pytest.mark.parametrize("width,hidden,in_dim,precision", CASES)
def test_calls_of_few_rays_match_a_larger_call(sdf, width, hidden, in_dim, precision, per_sm):
    """The fewer warps of a CTA take rays, at the edges of one, two, ... warps per CTA: the same bits as the same rays
    among more.  (Rays of the first call that miss the box leave work for the warps that held back.)"""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, whole = per_sm * sms + 3, 128 * sms
    b = inputs.net_to_bytes(inputs.siren_init(5, width, hidden, in_dim=in_dim, out_scale=30.0, out_shift=0.1))
    net = sdf.Net(b, getattr(sdf, precision))
    orig, d, time = rays(whole, in_dim)

    def trace(k):
        return sdf.trace_multiscale([net], [0.0], [25], 1e-2, orig[:, :k].contiguous(), d[:, :k].contiguous(),
                                    step_scale=[0.3], ray_time=None if time is None else time[:k].contiguous())

    few, all_ = trace(n), trace(whole)
    for x, y in zip(few, all_):
        assert torch.equal(x, y[..., :n])
    sdf.sync_status()
