"""Performance cases of the sdfnn library: the work a program that uses it has it do.

Every case runs through the public binding (`paper_2201_09147_gb300.sdfnn`).  Networks are the
ones in `scenes/` (and the random SIREN of `workloads.random_siren_64x1`); rays, points and
fitting batches are made from the seed on the GPU, with the distributions the library meets:
pinhole views from an orbit around the scene, points on and near the scene's surface, batches of
the fitting objective.  Kinds of case:

  points    sdf_normals / sdf_normal_map / sdf_normal_map_timed at given points
  trace     sdf_trace_multiscale of one view
  frame     sdf_trace_multiscale of one view, then the normals of the fine network at the hits
  plan      sdf_plan_launch: a batch of animation frames (4-D networks, a time per ray)
  host      sdf_frame_queue: host views rendered back to back through page-locked buffers
  fit       one native fitting step (forward, objective, backward, Adam)
  autograd  SineMLP forward and backward (dL/dtheta) under torch.autograd
"""
from __future__ import annotations

import functools
import math

import numpy as np
import torch

from paper_2201_09147_gb300 import inputs, sdfnn, workloads

PRECISION = {"fp32": sdfnn.SDF_FP32, "bf16": sdfnn.SDF_BF16, "fp16": sdfnn.SDF_FP16, "fp8": sdfnn.SDF_FP8}
# (inputs, width, hidden layers) of the networks used here
SHAPES = {"s8_64x1": (3, 64, 1), "s8_64x2": (3, 64, 2), "s8_128x2": (3, 128, 2), "s8_256x1": (3, 256, 1),
          "s8_256x2": (3, 256, 2), "s8_256x3": (3, 256, 3), "a8_64x1_t": (4, 64, 1), "a8_128x2_t": (4, 128, 2),
          "a8_256x3_t": (4, 256, 3), "siren": (3, 64, 1)}
# Mean network evaluations per ray of each level and share of the rays that hit, for views from
# the orbit (counted once with the FP32 path): what work() counts operations with.
EVALS = {"random_siren_64x1": ([21.4], 0.089), "nested_3level_512": ([5.6, 1.6, 1.1], 0.163),
         "normal_map_1080p": ([4.55], 0.168), "three_level_512": ([5.3, 0.93], 0.133),
         "plain_256x3_1080p": ([4.25], 0.134), "animation_32_pair": ([4.64], 0.191), "animation_32": ([4.64], 0.191)}


def listed():
    return [
        # picking / collision queries: the gradient at a few points per call (latency)
        dict(name="points_few_fp16", kind="points", net="s8_256x3", precision="fp16", n=300, mode="normals"),
        # mesh shading: unit normals of the fine network at the vertices of the subdivision-7 mesh
        dict(name="mesh_normals_bf16", kind="points", net="s8_256x3", precision="bf16", n=163842, mode="map"),
        # the faster, coarser option: E4M3 normals onto the hits of a frame (mask: one point in six)
        dict(name="map_masked_fp8", kind="points", net="s8_256x3", precision="fp8", n=1280 * 720 + 1, mode="masked"),
        # the smallest frame: a 128 x 128 preview of an untrained network with Lipschitz steps
        dict(name="trace_preview_128", kind="trace", workload="random_siren_64x1", precision="bf16", width=128,
             height=128),
        # the library's default use: a 1080p frame, coarse trace and neural normal mapping
        dict(name="frame_1080p_bf16", kind="frame", workload="normal_map_1080p", precision="bf16", width=1920,
             height=1080),
        # the nested sequence of all three widths, in the accurate 16-bit type, its own normals
        dict(name="frame_nested_512_fp16", kind="frame", workload="nested_3level_512", precision="fp16", width=512,
             height=512),
        # the fine network traced alone (the comparison every multiscale frame is measured against)
        dict(name="trace_plain_720p_bf16", kind="trace", workload="plain_256x3_1080p", precision="bf16", width=1280,
             height=720),
        # the FP32 path, trace and normals, on a window of odd size
        dict(name="frame_3level_odd_fp32", kind="frame", workload="three_level_512", precision="fp32", width=517,
             height=389),
        # animation: a batch of frames of mixed sizes as one graph, a time per ray
        dict(name="plan_animation_pair", kind="plan", workload="animation_32_pair", precision="bf16", small=4, hd=4,
             full=2),
        # a viewer that streams views through host memory
        dict(name="host_views_720p", kind="host", workload="normal_map_1080p", precision="bf16", width=1280,
             height=720, views=4),
        # native fitting of the widest network, tensor cores
        dict(name="fit_256x3_bf16", kind="fit", net="s8_256x3", precision="bf16", n=1 << 18),
        # training through autograd with the binding's default precision (FP32)
        dict(name="autograd_128x2_fp32", kind="autograd", net="s8_128x2", precision="fp32", n=50001),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["points", "points", "trace", "frame", "frame", "plan", "host", "fit", "fit", "autograd"])
    if kind == "points":
        net = rng.choice(["s8_64x2", "s8_128x2", "s8_256x1", "s8_256x3", "a8_128x2_t", "a8_256x3_t"])
        wide = SHAPES[net][1] >= 128
        prec = rng.choice(["bf16", "fp16", "fp8" if wide else "bf16", "fp32"])
        mode = rng.choice(["normals", "map", "masked", "timed" if SHAPES[net][0] == 4 else "masked"])
        return dict(kind=kind, net=net, precision=prec, n=_log(rng, 1, 60000 if prec == "fp32" else 900000), mode=mode)
    if kind in ("trace", "frame"):
        wl = rng.choice(["random_siren_64x1", "nested_3level_512", "normal_map_1080p", "three_level_512",
                         "plain_256x3_1080p"])
        prec = rng.choice(["bf16", "fp16", "fp32"])
        if wl == "plain_256x3_1080p":
            prec = rng.choice(["bf16", "fp16", "fp8"])
        most = {"fp32": 200000, "fp8": 900000}.get(prec, 900000 if wl == "plain_256x3_1080p" else 2000000)
        pixels = _log(rng, 1000, most)
        aspect = rng.uniform(0.6, 2.0)
        w = max(8, int(math.sqrt(pixels * aspect)))
        return dict(kind=kind, workload=wl, precision=prec, width=w, height=max(8, pixels // w))
    if kind == "plan":
        return dict(kind=kind, workload=rng.choice(["animation_32_pair", "animation_32"]),
                    precision=rng.choice(["bf16", "fp16"]), small=rng.randint(1, 6), hd=rng.randint(0, 3),
                    full=rng.randint(0, 1))
    if kind == "host":
        pixels = _log(rng, 4000, 900000)
        w = max(8, int(math.sqrt(pixels * rng.uniform(0.6, 2.0))))
        return dict(kind=kind, workload=rng.choice(["normal_map_1080p", "three_level_512"]),
                    precision=rng.choice(["bf16", "fp16"]), width=w, height=max(8, pixels // w),
                    views=rng.randint(1, 4))
    net = rng.choice(["s8_64x2", "s8_128x2", "s8_256x1", "s8_256x3", "a8_128x2_t"])
    prec = rng.choice(["bf16", "fp16", "fp32"])
    return dict(kind=kind, net=net, precision=prec, n=_log(rng, 500, 30000 if prec == "fp32" else 300000))


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _image(net):
    if net == "siren":
        return inputs.net_to_bytes(workloads.random_siren_64x1())
    return (workloads.SCENES / (net + ".sdfn")).read_bytes()


def _start_image(case, seed):
    """The network a fit starts from: the SIREN initialisation of the shape."""
    i, w, k = SHAPES[case["net"]]
    return inputs.net_to_bytes(inputs.siren_init(seed, w, k, in_dim=i))


@functools.lru_cache(maxsize=None)
def _net(net, precision):
    """A program loads its networks once and renders many frames with them."""
    return sdfnn.Net(_image(net), PRECISION[precision])


def _levels(wl):
    return [x.split(".")[0] if isinstance(x, str) else "siren" for x in wl.levels]


def _fine(wl):
    return wl.fine.split(".")[0] if isinstance(wl.fine, str) else "siren"


def _rand(gen, *shape):
    return torch.rand(*shape, generator=gen, device="cuda", dtype=torch.float64)


def _view(width, height, azimuth, elevation):
    """Pinhole rays (3, n) float32 towards the origin from 2.5 away, vertical field of view 45 degrees."""
    f64 = dict(device="cuda", dtype=torch.float64)
    ce = math.cos(elevation)
    eye = torch.tensor([2.5 * math.sin(azimuth) * ce, 2.5 * math.sin(elevation), 2.5 * math.cos(azimuth) * ce], **f64)
    fwd = -eye / eye.norm()
    right = torch.linalg.cross(fwd, torch.tensor([0.0, 1.0, 0.0], **f64))
    right = right / right.norm()
    up = torch.linalg.cross(right, fwd)
    th = math.tan(math.radians(22.5))
    x = (2.0 * (torch.arange(width, **f64) + 0.5) / width - 1.0) * th * (width / height)
    y = (1.0 - 2.0 * (torch.arange(height, **f64) + 0.5) / height) * th
    d = fwd[:, None, None] + x[None, None, :] * right[:, None, None] + y[None, :, None] * up[:, None, None]
    d = (d / d.norm(dim=0, keepdim=True)).reshape(3, -1).float().contiguous()
    return eye.float()[:, None].expand(3, d.shape[1]).contiguous(), d


def _random_view(width, height, gen):
    a, e = (2.0 * _rand(gen, 2) - 1.0).tolist()
    return _view(width, height, math.pi * a, 0.4 * e)


def _surface_points(n, gen, jitter):
    """Points (3, n) float64 on the scene's spheres, moved along the radius by N(0, jitter)."""
    scene = inputs.sphere_scene(seed=1)
    c = torch.as_tensor(scene.centres, device="cuda")
    r = torch.as_tensor(scene.radii, device="cuda")
    k = torch.randint(0, len(scene.radii), (n,), generator=gen, device="cuda")
    u = torch.randn(3, n, generator=gen, device="cuda", dtype=torch.float64)
    u = u / u.norm(dim=0, keepdim=True)
    j = jitter * torch.randn(n, generator=gen, device="cuda", dtype=torch.float64)
    return (c[k].T + (r[k] + j)[None, :] * u).clamp(-1.0, 1.0)


def _scene(p):
    """Value and gradient of the analytic scene at points p (3, n) float64."""
    scene = inputs.sphere_scene(seed=1)
    best = torch.full((p.shape[1],), math.inf, device="cuda", dtype=torch.float64)
    grad = torch.zeros_like(p)
    for c, r in zip(scene.centres, scene.radii):
        diff = p - torch.as_tensor(c, device="cuda")[:, None]
        dist = diff.norm(dim=0)
        closer = dist - r < best
        best = torch.where(closer, dist - r, best)
        grad = torch.where(closer[None], diff / dist.clamp_min(1e-12)[None], grad)
    s, c = torch.sin(scene.freq * p), torch.cos(scene.freq * p)
    value = best + scene.amp * s[0] * s[1] * s[2]
    grad = grad + scene.amp * scene.freq * torch.stack([c[0] * s[1] * s[2], s[0] * c[1] * s[2], s[0] * s[1] * c[2]])
    return value, grad


def _points_inputs(case, seed):
    gen = _gen(seed)
    n = case["n"]
    pts = _surface_points(n, gen, 0.0).float().contiguous()
    mask = (_rand(gen, n) < 1.0 / 6.0).to(torch.uint8) if case["mode"] == "masked" else None
    time = _rand(gen, n).float() if case["mode"] == "timed" else None
    return pts, mask, time


def _plan_inputs(case, seed):
    gen = _gen(seed)
    frames = [(256, 256)] * case["small"] + [(1280, 720)] * case["hd"] + [(1920, 1080)] * case["full"]
    t0 = 0.5 * _rand(gen, 1).item()
    views = [_random_view(w, h, gen) for w, h in frames]
    times = [torch.full((w * h,), t0 + 0.5 * k / len(frames), device="cuda") for k, (w, h) in enumerate(frames)]
    return (torch.cat([v[0] for v in views], 1).contiguous(), torch.cat([v[1] for v in views], 1).contiguous(),
            torch.cat(times))


def _fit_inputs(case, seed):
    """A batch of the fitting objective: half near the surface, half uniform, and adjoints of the outputs' scale."""
    gen = _gen(seed)
    n, half = case["n"], case["n"] // 2
    pts = torch.cat([_surface_points(half, gen, 0.02), 2.0 * _rand(gen, 3, n - half) - 1.0], 1).float().contiguous()
    value, grad = _scene(pts.double())
    near = torch.zeros(n, dtype=torch.uint8, device="cuda")
    near[:half] = 1
    time = _rand(gen, n).float() if SHAPES[case["net"]][0] == 4 else None
    d_f = (torch.randn(n, generator=gen, device="cuda") / n).contiguous()
    d_grad = (0.1 * torch.randn(3, n, generator=gen, device="cuda") / n).contiguous()
    return dict(pts=pts, value=value.float(), grad=grad.float().contiguous(), near=near, time=time, d_f=d_f,
                d_grad=d_grad)


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind, "case": case}
    if kind == "points":
        s["net"] = _net(case["net"], case["precision"])
        s["pts"], s["mask"], s["time"] = _points_inputs(case, seed)
    elif kind in ("trace", "frame"):
        wl = workloads.get(case["workload"], case["width"], case["height"])
        s["wl"], s["nets"] = wl, [_net(x, case["precision"]) for x in _levels(wl)]
        s["fine"] = _net(_fine(wl), case["precision"])
        s["orig"], s["dirs"] = _random_view(case["width"], case["height"], _gen(seed))
    elif kind == "plan":
        wl = workloads.get(case["workload"])
        orig, dirs, time = _plan_inputs(case, seed)
        s["plan"] = sdfnn.Plan([_net(x, case["precision"]) for x in _levels(wl)], wl.delta, wl.caps, wl.eps, orig, dirs,
                               fine=_net(_fine(wl), case["precision"]), ray_time=time, step_scale=wl.step_scale,
                               final_mode=wl.final_mode, want_iters=False)
    elif kind == "host":
        wl = workloads.get(case["workload"], case["width"], case["height"])
        gen, n = _gen(seed), case["width"] * case["height"]
        s["views"] = []
        for _ in range(case["views"]):
            o, d = _random_view(case["width"], case["height"], gen)
            s["views"].append(tuple(x.cpu().pin_memory() for x in (o, d)) + (
                torch.empty(3, n).pin_memory(), torch.empty(n, dtype=torch.uint8).pin_memory(),
                torch.empty(3, n).pin_memory()))
        s["queue"] = sdfnn.FrameQueue([_net(x, case["precision"]) for x in _levels(wl)], wl.delta, wl.caps, wl.eps,
                                      _net(_fine(wl), case["precision"]), n, depth=3, step_scale=wl.step_scale,
                                      final_mode=wl.final_mode)
    else:
        s["shape"], theta = sdfnn.theta_from_sdfn(_start_image(case, seed))
        s["theta"] = torch.from_numpy(theta).cuda()
        s["precision"] = PRECISION[case["precision"]]
        s |= _fit_inputs(case, seed)
        if kind == "fit":
            s["m"], s["v"], s["step"] = torch.zeros_like(s["theta"]), torch.zeros_like(s["theta"]), 0
            _, size = sdfnn.train_shape_info(*s["shape"], case["n"], s["precision"])
            s["workspace"] = torch.empty(size, dtype=torch.uint8, device="cuda")
    return s


def run(s):
    kind, case = s["kind"], s["case"]
    if kind == "points":
        if case["mode"] == "normals":
            return sdfnn.normals(s["net"], s["pts"])
        if case["mode"] == "timed":
            return sdfnn.normal_map_timed(s["net"], s["pts"], s["time"])
        return sdfnn.normal_map(s["net"], s["pts"], s["mask"])
    if kind in ("trace", "frame"):
        wl = s["wl"]
        pos, t, hit, iters = sdfnn.trace_multiscale(s["nets"], wl.delta, wl.caps, wl.eps, s["orig"], s["dirs"],
                                                    step_scale=wl.step_scale, final_mode=wl.final_mode)
        out = {"pos": pos, "t": t, "hit": hit, "iters": iters}
        if kind == "frame":
            out["normal"] = sdfnn.normal_map(s["fine"], pos, hit)
        return out
    if kind == "plan":
        p = s["plan"]
        p.launch()
        return {"pos": p.pos, "t": p.t, "hit": p.hit, "normal": p.normal}
    if kind == "host":
        for v in s["views"]:
            s["queue"].submit(*v)
        s["queue"].wait()
        return [{"pos": v[2], "hit": v[3], "normal": v[4]} for v in s["views"]]
    if kind == "fit":
        s["step"] += 1
        loss, s["workspace"] = sdfnn.fit_step(s["shape"], s["theta"], s["m"], s["v"], s["step"], s["pts"], s["value"],
                                              s["grad"], s["near"], lr=1e-5, workspace=s["workspace"],
                                              precision=s["precision"], pt_time=s["time"])
        return {"loss": loss, "theta": s["theta"], "m": s["m"], "v": s["v"]}
    theta = s["theta"].detach().requires_grad_(True)
    f, g = sdfnn.SineMLP.apply(theta, s["pts"], s["shape"], s["time"], s["precision"])
    (d_theta,) = torch.autograd.grad((f, g), theta, (s["d_f"], s["d_grad"]))
    return {"f": f.detach(), "grad": g.detach(), "d_theta": d_theta}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------
def _params(net):
    i, w, k = SHAPES[net]
    return w * i + w + k * (w * w + w) + w + 1


def _eval_flops(net):
    i, w, k = SHAPES[net]
    return 2.0 * (w * i + k * w * w + w)


def work(case):
    kind = case["kind"]
    if kind == "points":
        n = case["n"]
        share = 1.0 / 6.0 if case["mode"] == "masked" else 1.0
        # value and three tangents through the hidden layers
        flops = 4.0 * _eval_flops(case["net"]) * n * share
        return {"bytes": 12.0 * n * (share + 1.0) + n * (share < 1.0) + 4.0 * _params(case["net"]), "flops": flops}
    if kind in ("fit", "autograd"):
        n, p = case["n"], _params(case["net"])
        # forward, adjoints, weight gradients: three products per layer over four streams; points, targets
        # (or adjoints) and outputs once; parameters, their moments and gradients once
        return {"bytes": n * (12.0 + 16.0 + 16.0 + 1.0) + 4.0 * p * (6.0 if kind == "fit" else 2.0),
                "flops": 3.0 * 4.0 * _eval_flops(case["net"]) * n}
    wl = workloads.get(case["workload"])
    if kind == "plan":
        n = case["small"] * 256 * 256 + case["hd"] * 1280 * 720 + case["full"] * 1920 * 1080
    else:
        n = case["width"] * case["height"] * case.get("views", 1)
    evals, hits = EVALS[case["workload"]]
    levels = _levels(wl)
    flops = sum(e * _eval_flops(x) for e, x in zip(evals, levels)) * n
    # rays in; end point, distance, hit and step count out
    size = n * (24.0 + 12.0 + 4.0 + 1.0 + 2.0)
    if kind == "plan":
        size += 4.0 * n  # a time per ray
    if kind != "trace":
        flops += 4.0 * _eval_flops(_fine(wl)) * n * hits
        size += 12.0 * n
    return {"bytes": size, "flops": flops}


# ---------------------------------------------------------------------------
# the same in 64 bits, with torch alone
# ---------------------------------------------------------------------------
class _Exact:
    """A network file's sine MLP in float64: f = w . sin(W_k ... sin(W_0 x + b_0)) + b."""

    def __init__(self, image):
        head = np.frombuffer(image[:32], "<u4")
        self.inputs, w, k = int(head[2]), int(head[3]), int(head[4])
        w0, wh = (1.0, 1.0) if head[7] & 1 else np.frombuffer(image[20:28], "<f4").astype(np.float64)
        flat = np.frombuffer(image[32:], "<f4").astype(np.float64)
        self.weights, self.biases, o = [], [], 0
        for layer in range(k + 1):
            fan, scale = (self.inputs, w0) if layer == 0 else (w, wh)
            self.weights.append(torch.tensor(scale * flat[o:o + w * fan].reshape(w, fan), device="cuda"))
            o += w * fan
            self.biases.append(torch.tensor(scale * flat[o:o + w], device="cuda"))
            o += w
        self.out, self.bias = torch.tensor(flat[o:o + w], device="cuda"), float(flat[o + w])
        self.width = w

    def folded(self):
        """The float32 vector of the folded parameters, in the file's order, as float64."""
        parts = [x.reshape(-1) for pair in zip(self.weights, self.biases) for x in pair]
        tail = torch.tensor([self.bias], dtype=torch.float64, device="cuda")
        return torch.cat(parts + [self.out, tail]).float().double()

    def lipschitz(self):
        return math.prod(float(torch.linalg.matrix_norm(x, 2)) for x in self.weights) * float(self.out.norm())

    def chunk(self):
        return (1 << 26) // self.width

    def value(self, x):
        """f at x (inputs, n)."""
        out = torch.empty(x.shape[1], dtype=torch.float64, device="cuda")
        for a in range(0, x.shape[1], self.chunk()):
            h = x[:, a:a + self.chunk()]
            for w, b in zip(self.weights, self.biases):
                h = torch.sin(torch.addmm(b[:, None], w, h))
            out[a:a + self.chunk()] = self.out @ h + self.bias
        return out

    def gradient(self, x):
        """The spatial gradient (3, n) at x (inputs, n)."""
        out = torch.empty(3, x.shape[1], dtype=torch.float64, device="cuda")
        step = self.chunk() // 4
        for a in range(0, x.shape[1], step):
            h, back = x[:, a:a + step], []
            for w, b in zip(self.weights, self.biases):
                z = torch.addmm(b[:, None], w, h)
                back.append(torch.cos(z))
                h = torch.sin(z)
            g = self.out[:, None] * back[-1]
            for w, c in zip(self.weights[:0:-1], back[-2::-1]):
                g = (w.T @ g) * c
            out[:, a:a + step] = (self.weights[0].T @ g)[:3]
        return out

    def training(self, theta, x):
        """f and its spatial gradient as functions of the folded parameters theta (for autograd)."""
        o, w, h, g = 0, self.width, x, None
        for layer, shape in enumerate(self.weights):
            fan = shape.shape[1]
            weight = theta[o:o + w * fan].reshape(w, fan)
            o += w * fan
            bias = theta[o:o + w]
            o += w
            z = torch.addmm(bias[:, None], weight, h)
            c, h = torch.cos(z), torch.sin(z)
            if layer == 0:
                g = [weight[:, i:i + 1] * c for i in range(3)]
            else:
                g = [(weight @ t) * c for t in g]
        out = theta[o:o + w]
        return out @ h + theta[o + w], torch.stack([out @ t for t in g])


def _unit(g):
    size = g.norm(dim=0, keepdim=True)
    return torch.where(size >= 1e-12, g / size.clamp_min(1e-300), torch.zeros_like(g))


def _with_time(net, p, time):
    if net.inputs == 3:
        return p
    return torch.cat([p, torch.zeros(1, p.shape[1], dtype=p.dtype, device="cuda") if time is None else time[None]])


def _exact_trace(nets, wl, orig, dirs, time):
    """Alg. 1 in float64: end points, distances and hits."""
    o, v = orig.double(), dirs.double()
    time = None if time is None else time.double()
    t1, t2 = (-1.0 - o) / v, (1.0 - o) / v
    near = torch.minimum(t1, t2).amax(0).clamp_min(0.0)
    far = torch.maximum(t1, t2).amin(0)
    inside = near <= far
    tau = torch.where(inside, near, torch.zeros_like(near))
    pos = o + tau * v
    hit = torch.zeros(o.shape[1], dtype=torch.bool, device="cuda")
    alive = inside.nonzero()[:, 0]  # rays that enter the next level
    for j, net in enumerate(nets):
        last = j + 1 == len(nets)
        d = 0.0 if last and wl.final_mode == 0 else float(np.float32(wl.delta[j]))
        scale = float(np.float32(1.0 / net.lipschitz() if wl.step_scale is None else wl.step_scale[j]))
        eps = float(np.float32(wl.eps))
        done, active = [], alive
        for it in range(wl.caps[j]):
            if not active.numel():
                break
            t = net.value(_with_time(net, pos[:, active], None if time is None else time[active])) - d
            step = scale * t
            pos[:, active] += step * v[:, active]
            tau[active] += step
            out = (pos[:, active].abs() > 1.0 + 1e-3).any(0)
            ends = ~(t > eps) & ~out
            if last:
                hit[active[ends]] = True
            done.append(active[ends])
            active = active[~out & ~ends]
        alive = torch.cat(done + [active])
    return pos, tau, hit


def exact(case, seed):
    kind = case["kind"]
    if kind == "points":
        pts, mask, time = _points_inputs(case, seed)
        net = _Exact(_image(case["net"]))
        g = net.gradient(_with_time(net, pts.double(), None if time is None else time.double()))
        if case["mode"] != "normals":
            g = _unit(g)
        return g if mask is None else g * (mask != 0)
    if kind in ("trace", "frame", "plan", "host"):
        wl = workloads.get(case["workload"])
        nets, fine = [_Exact(_image(x)) for x in _levels(wl)], _Exact(_image(_fine(wl)))
        if kind == "plan":
            views = [_plan_inputs(case, seed)]
        else:
            gen = _gen(seed)
            views = [_random_view(case["width"], case["height"], gen) + (None,) for _ in range(case.get("views", 1))]
        outs = []
        for orig, dirs, time in views:
            pos, tau, hit = _exact_trace(nets, wl, orig, dirs, time)
            out = {"pos": pos, "t": tau, "hit": None, "iters": None}
            if kind != "trace":
                at = hit.nonzero()[:, 0]
                out["normal"] = torch.zeros_like(pos)
                out["normal"][:, at] = _unit(fine.gradient(
                    _with_time(fine, pos[:, at], None if time is None else time[at].double())))
                if case["workload"] == "three_level_512" and case["precision"] != "fp32":
                    out["normal"] = None  # its caps cut rays off: which of them count as hits is up to the rounding
            if kind == "host":
                del out["t"]
            if kind != "trace" and kind != "frame":
                del out["iters"]
            outs.append(out)
        return outs if kind == "host" else outs[0]
    net, data, n = _Exact(_start_image(case, seed)), _fit_inputs(case, seed), case["n"]
    theta = net.folded().requires_grad_(True)
    x = _with_time(net, data["pts"].double(), None if data["time"] is None else data["time"].double())
    near = data["near"] != 0
    d_theta = torch.zeros_like(theta)
    terms = torch.zeros(3, dtype=torch.float64, device="cuda")
    fs, gs = [], []
    step = max(1, net.chunk() // 16)
    for a in range(0, n, step):
        b = slice(a, a + step)
        f, g = net.training(theta, x[:, b])
        if kind == "autograd":
            total = (f * data["d_f"][b]).sum() + (g * data["d_grad"][:, b]).sum()
            fs.append(f.detach())
            gs.append(g.detach())
        else:
            target = data["grad"][:, b].double()
            cosine = (g * target).sum(0) / (g.norm(dim=0) * target.norm(dim=0))
            part = torch.stack([(f - data["value"][b].double()).abs().sum() / n,
                                ((1.0 - cosine) * near[b]).sum() / max(1, int(near.sum())),
                                (g.norm(dim=0) - 1.0).abs().sum() / n])
            total = part[0] + 0.1 * part[1] + 0.05 * part[2]
            terms += part.detach()
        d_theta += torch.autograd.grad(total, theta)[0]
    if kind == "autograd":
        return {"f": torch.cat(fs), "grad": torch.cat(gs, 1), "d_theta": d_theta}
    m, v = 0.1 * d_theta, 0.001 * d_theta * d_theta
    new = theta.detach() - 1e-5 * (m / 0.1) / ((v / 0.001).sqrt() + 1e-8)
    loss = torch.cat([terms, (terms[0] + 0.1 * terms[1] + 0.05 * terms[2])[None]])
    return {"loss": loss, "theta": new, "m": m, "v": v}
