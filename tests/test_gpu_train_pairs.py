"""16-bit training on batches of more than one half-tile per SM, whose half-tiles run in pairs, against the
same points in calls small enough to run spread (checked against FP64 and FP32 in test_gpu_train_tc.py).

A point's f and grad f do not depend on the call: equal bits.  dL/dtheta sums the same products in another
order in FP32 (both objectives' adjoints are scaled by powers of two): 1e-5 of its norm, as for chunks of one call.
"""
import pytest
import torch

from paper_2201_09147_gb300 import inputs

pytestmark = pytest.mark.gpu


# the edges of the spread range, a ragged larger batch, and one whose weight gradients keep an accumulator for more
# than 32 K blocks (512 points per SM and layer)
@pytest.mark.parametrize("per_sm,extra", [(32, -1), (32, 0), (32, 1), (131, 5), (700, 3)])
@pytest.mark.parametrize("precision", ["SDF_BF16", "SDF_FP16"])
@pytest.mark.parametrize("width,hidden,in_dim", [(64, 1, 3), (128, 2, 4), (256, 3, 3)])
def test_pairs_match_spread_calls(sdf, width, hidden, in_dim, precision, per_sm, extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n, chunk, prec = per_sm * sms + extra, 27 * sms + 13, getattr(sdf, precision)
    shape, theta = sdf.theta_from_sdfn(inputs.net_to_bytes(inputs.siren_init(11, width, hidden, in_dim=in_dim)))
    th = torch.from_numpy(theta).cuda()
    pts = torch.from_numpy(inputs.random_points(21, n)).cuda()
    time = torch.from_numpy(inputs.uniform01(22, n).astype("float32")).cuda() if in_dim == 4 else None
    z = torch.from_numpy((2.0 * inputs.uniform01(23, 4 * n) - 1.0).astype("float32") / n).cuda()
    d_f, d_g = z[:n].contiguous(), z[n:].reshape(3, n).contiguous()
    f, g, ws = sdf.train_forward(shape, th, pts, pt_time=time, precision=prec)
    whole = sdf.train_backward(shape, th, pts, d_f, d_g, ws, pt_time=time, precision=prec)
    parts = torch.zeros_like(whole, dtype=torch.float64)
    for lo in range(0, n, chunk):
        hi = min(n, lo + chunk)
        p, t = pts[:, lo:hi].contiguous(), None if time is None else time[lo:hi].contiguous()
        cf, cg, cw = sdf.train_forward(shape, th, p, pt_time=t, precision=prec)
        assert torch.equal(cf, f[lo:hi]) and torch.equal(cg, g[:, lo:hi])
        parts += sdf.train_backward(shape, th, p, d_f[lo:hi].contiguous(), d_g[:, lo:hi].contiguous(), cw, pt_time=t,
                                    precision=prec)
    sdf.sync_status()
    assert ((whole - parts).norm() / parts.norm()).item() <= 1e-5
