"""The trace kernel with several threads per ray at the ends of its work: levels without a step, and
tails whose rays end turns apart, in which the warps of a CTA see the list run dry at different times."""
import numpy as np
import pytest
import torch

from paper_2201_09147_gb300 import inputs, workloads

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


@pytest.mark.parametrize("in_dim,precision,line", [(3, "SDF_BF16", 2700), (4, "SDF_FP16", 256), (4, "SDF_FP8", 1000)])
def test_one_hidden_layer_of_256_in_large_calls(sdf, in_dim, precision, line):
    """Later levels of calls of more than 256 rays per SM, and first levels of more than 2,700 (E4M3: 1,000), run on a
    kernel of their own: the same bits as in calls of fewer, with and without levels that do no step."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    n = line * sms + 33
    b = inputs.net_to_bytes(inputs.siren_init(5, 256, 1, in_dim=in_dim, out_scale=30.0, out_shift=0.1))
    net = sdf.Net(b, getattr(sdf, precision))
    orig, d, time = rays(n, in_dim)

    def trace(lo, hi, caps):
        k = len(caps)
        return sdf.trace_multiscale([net] * k, [0.01] * (k - 1) + [0.0], caps, 1e-2, orig[:, lo:hi].contiguous(),
                                    d[:, lo:hi].contiguous(), step_scale=[0.3] * k,
                                    ray_time=None if time is None else time[lo:hi].contiguous())

    for caps in ([25], [3, 25], [0, 25], [25, 0], [2, 3, 4]):
        whole = trace(0, n, caps)
        for lo, hi in ((0, line * sms), (line * sms, n)):
            assert all(torch.equal(x[..., lo:hi], y) for x, y in zip(whole, trace(lo, hi, caps)))
    assert 0 < int(trace(0, n, [25])[2].sum()) < n
    sdf.sync_status()


@pytest.mark.parametrize("width,height", [(150, 129), (180, 170), (200, 195)])
def test_queued_frames_match_direct_calls(sdf, width, height):
    """Frames overlapped on two streams take other kernels from 128 rays per SM on: the same bits as direct calls."""
    wl = workloads.get("three_level_512", width, height)
    nets = [sdf.Net((workloads.SCENES / x).read_bytes(), sdf.SDF_BF16) for x in wl.levels]
    fine = sdf.Net((workloads.SCENES / wl.fine).read_bytes(), sdf.SDF_BF16)
    n = width * height
    orig, d, _ = rays(n, 3)
    host = [x.cpu().pin_memory() for x in (orig, d)]
    out = [(torch.empty(3, n).pin_memory(), torch.empty(n, dtype=torch.uint8).pin_memory(), torch.empty(3, n).pin_memory())
           for _ in range(4)]
    queue = sdf.FrameQueue(nets, wl.delta, wl.caps, wl.eps, fine, n, depth=3, step_scale=wl.step_scale,
                           final_mode=wl.final_mode)
    for o in out:
        queue.submit(*host, *o)
    queue.wait()
    pos, _, hit, _ = sdf.trace_multiscale(nets, wl.delta, wl.caps, wl.eps, orig, d, step_scale=wl.step_scale,
                                          final_mode=wl.final_mode)
    normal = sdf.normal_map(fine, pos, hit)
    sdf.sync_status()
    assert hit.any()
    for o in out:
        assert all(torch.equal(a, b.cpu()) for a, b in zip(o, (pos, hit, normal)))


@pytest.mark.parametrize("per_sm,most", [(3, 1), (256, 1), (257, 6)])
def test_autotuned_plans_report_what_they_run(sdf, per_sm, most):
    """The tile count of a plan is a count that its launches use: one for the calls of few rays, whose kernel has
    one launch shape."""
    n = per_sm * torch.cuda.get_device_properties(0).multi_processor_count
    net = sdf.Net(inputs.net_to_bytes(inputs.siren_init(5, 64, 1, out_scale=30.0, out_shift=0.1)), sdf.SDF_BF16)
    orig, d, _ = rays(n, 3)
    plan = sdf.Plan([net], [0.0], [9], 1e-2, orig, d, step_scale=[0.3], autotune=True)
    tiles, _ = plan.info()
    assert 1 <= tiles[0] <= most
    plan.launch()
    direct = sdf.trace_multiscale([net], [0.0], [9], 1e-2, orig, d, step_scale=[0.3])
    assert torch.equal(plan.pos, direct[0]) and torch.equal(plan.hit, direct[2])
    plan.close()
    sdf.sync_status()
