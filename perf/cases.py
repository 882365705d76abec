"""The work a program has this package do, as cases that can be timed.

Each case goes through the public entry points: `gftorf.Renderer` (eager
calls, a captured CUDA graph, or `render_ctof` under autograd),
`fit.FitLoop`, `mlp.DeformationMLP` and `gftorf.sort_footprints`.  Scenes
follow the synthetic workloads of `scenes.py` (its sizes, distributions and
options), drawn here on the GPU from the seed alone.  `exact` is a plain
torch restatement in 64 bits that uses none of the package's code.
"""
import math

import numpy as np
import torch

DEV = "cuda"
C_LIGHT = 299792458.0
QUARTET = (0.0, math.pi / 2, math.pi, 3 * math.pi / 2)
FREQS = (30e6, 80e6)
# the constants of gftorf.make_consts, as single precision holds them
DILATION, ALPHA_MAX, ALPHA_MIN, T_MIN, GUARD, SIGMA_CUT, NEAR = (
    float(np.float32(v)) for v in (0.3, 0.99, 1.0 / 255.0, 1e-4, 1.3, 3.0, 0.2))
# fit.LEARNING_RATES and fit.BOUNDS
FIT_LRS = {"means": 1.6e-4, "coeffs": 8e-4, "scales": 5e-3 * 0.05, "quats": 1e-3,
           "opacity": 5e-2 * 0.2, "amplitude": 1.6e-4}
FIT_BOUNDS = {"opacity": (1e-3, 1.0), "scales": (1e-5, 10.0), "amplitude": (0.0, 10.0)}
BLOCK = 64  # pixels across the blocks that exact() composites at once
MLP_WIDTH, MLP_DEPTH, MLP_IN, MLP_USED, MLP_BANDS = 256, 8, 128, 84, 10


def _render(name, n, frames, width, height, tile, **more):
    case = dict(kind="render", n=n, frames=frames, width=width, height=height, tile_w=tile[0],
                tile_h=tile[1], ppt=4 if tile[0] >= 32 else 0, persistent=False, freqs=1,
                moving=True, hidden=frames > 1, backward=True, how="graph", sh=-1, extra=False,
                posed=False, asynchronous=False, z0=1.0, z1=3.0)
    case.update(more)
    if name:
        case["name"] = name
    return case


def listed():
    return [
        # an interactive preview: the smallest scene, one eager forward (latency, launches)
        _render("view_1k", 1000, 1, 64, 64, (16, 16), how="eager", moving=False, backward=False),
        # a differentiable render inside somebody's own torch model, at a small size
        _render("grad_5k", 5000, 3, 96, 64, (16, 16), how="autograd"),
        # one frame of a mid-sized scene per step, as online fitting takes it
        _render("frame_100k", 100_000, 1, 640, 480, (32, 32)),
        # the benchmark's step: 16 timesteps of 300k dynamic Gaussians, one captured graph
        _render("batch_300k", 300_000, 16, 640, 480, (64, 64)),
        # the two-frequency capture (phase wrapping), the largest scene
        _render("twofreq_500k", 500_000, 8, 640, 576, (64, 64), freqs=2, z0=0.5, z1=6.0),
        # every model option: view-dependent reflectivity, phasor and depth channels, a moved
        # camera, eager calls
        _render("options_200k", 200_000, 4, 640, 480, (32, 32), how="eager", sh=3, extra=True,
                posed=True),
        # rendering an asynchronous raw sequence of a fitted scene, ragged image, default tiles
        _render("async_view", 120_000, 12, 517, 389, (16, 16), how="eager", backward=False,
                asynchronous=True),
        # a whole fitting iteration over the captured sequence, replayed as a graph
        dict(name="fit_300k", kind="fit", n=300_000, frames=60, width=640, height=480, tile_w=64,
             tile_h=64, persistent=False),
        # the deformation network: training at one timestep, at the batch's 16 timesteps, and
        # inference for a rendered frame
        dict(name="mlp_train_300k", kind="mlp", n=300_000, frames=1, train=True),
        dict(name="mlp_train_4800k", kind="mlp", n=300_000, frames=16, train=True),
        dict(name="mlp_infer_300k", kind="mlp", n=300_000, frames=1, train=False),
        # binning of footprints that a caller projected itself
        dict(name="bin_100k", kind="bin", n=100_000, frames=4, width=640, height=480, tile_w=16,
             tile_h=16),
    ]


def draw(rng):
    def spread(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(("render",) * 5 + ("fit", "mlp", "mlp", "bin"))
    width, height = rng.choice(((640, 480), (640, 576), (spread(64, 640), spread(48, 480))))
    if kind == "mlp":
        return dict(kind="mlp", n=spread(1000, 300_000), frames=spread(1, 16),
                    train=rng.random() < 0.6)
    if kind == "bin":
        tile = rng.choice(((8, 8), (16, 16), (16, 32), (32, 32), (64, 64)))
        return dict(kind="bin", n=spread(1000, 100_000), frames=spread(1, 4), width=width,
                    height=height, tile_w=tile[0], tile_h=tile[1])
    if kind == "fit":
        tile = rng.choice(((16, 16), (32, 32), (64, 64)))
        return dict(kind="fit", n=spread(5000, 300_000), frames=spread(4, 24), width=width,
                    height=height, tile_w=tile[0], tile_h=tile[1], persistent=rng.random() < 0.5)
    tile = rng.choice(((16, 16), (16, 32), (32, 32), (64, 32), (64, 64)))
    frames = spread(1, 16)
    asynchronous = rng.random() < 0.2
    return _render(None, spread(1000, 300_000), frames, width, height, tile,
                   how=rng.choice(("eager", "graph", "autograd")), backward=rng.random() < 0.75,
                   persistent=rng.random() < 0.3, freqs=1 if asynchronous else rng.choice((1, 2)),
                   sh=rng.choice((-1, -1, 1, 3)), extra=rng.random() < 0.3,
                   posed=rng.random() < 0.3, asynchronous=asynchronous)


# --- inputs ------------------------------------------------------------------------
def _generator(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1_000_003 + 17)
    return g


def _uniform(g, shape, lo, hi):
    return torch.empty(shape, device=DEV).uniform_(lo, hi, generator=g)


def _normal(g, shape, std=1.0, mean=0.0):
    return torch.empty(shape, device=DEV).normal_(mean, std, generator=g)


def _focal(width):
    return float(np.float32(width / (2.0 * math.tan(math.radians(60.0) / 2.0))))


def _pose(case):
    """[R | t], single precision: the identity, or a turned and shifted camera."""
    if not case.get("posed"):
        return np.concatenate([np.eye(3), np.zeros((3, 1))], 1).astype(np.float32)
    a, b, c = (math.radians(v) for v in (4.0, -6.0, 3.0))
    rx = np.array([[1, 0, 0], [0, math.cos(a), -math.sin(a)], [0, math.sin(a), math.cos(a)]])
    ry = np.array([[math.cos(b), 0, math.sin(b)], [0, 1, 0], [-math.sin(b), 0, math.cos(b)]])
    rz = np.array([[math.cos(c), -math.sin(c), 0], [math.sin(c), math.cos(c), 0], [0, 0, 1]])
    r = rz @ ry @ rx
    centre = np.array([0.1, -0.05, -0.2])
    return np.concatenate([r, (-r @ centre)[:, None]], 1).astype(np.float32)


def _frames_of(case):
    """Per frame: (time, phase offset, interpolation bracket or None)."""
    b = case["frames"]
    if case.get("asynchronous"):
        tick = 1.0 / max(b - 1, 1)
        return [(i * tick, (math.pi / 2) * (i % 4), (4 * (i // 4) * tick, 4 * (i // 4) * tick + 4 * tick))
                for i in range(b)]
    return [(i / max(b - 1, 1) if b > 1 else 0.37, 0.0, None) for i in range(b)]


def _offsets(case):
    return (0.0,) if case.get("asynchronous") else QUARTET


def _channels(case):
    f = case.get("freqs", 1)
    return f * len(_offsets(case)) + 1 + (2 * f + 1 if case.get("extra") else 0)


def _gaussians(case, g):
    n, w, h = case["n"], case["width"], case["height"]
    z0, z1 = (1.0, 6.0) if case["kind"] == "fit" else (case["z0"], case["z1"])
    z = _uniform(g, (n,), z0, z1)
    half = torch.tensor([w / 2 / _focal(w), h / 2 / _focal(w)], device=DEV)
    means = torch.cat([_uniform(g, (n, 2), -1, 1) * half * z[:, None], z[:, None]], 1)
    if case.get("posed"):
        rt = torch.as_tensor(_pose(case), device=DEV).double()
        means = ((means.double() - rt[:, 3]) @ rt[:, :3]).float()
    p = dict(means=means.contiguous(), scales=_normal(g, (n, 3), 0.3, -3.5).exp(),
             quats=torch.nn.functional.normalize(_normal(g, (n, 4)), dim=1).contiguous(),
             opacity=torch.sigmoid(_normal(g, (n,))), amplitude=_uniform(g, (n,), 0.1, 1.0),
             coeffs=None, delta=None, sh=None)
    if case["kind"] == "fit":
        p["amplitude"] = torch.full((n,), 0.1, device=DEV)
        p["coeffs"] = torch.zeros((n, 3, 3), device=DEV)
        return p
    if case["moving"]:
        p["coeffs"] = _normal(g, (n, 3, 3), 0.05)
    if case["hidden"]:  # uneven visible counts: the rest is moved out of sight
        share = _uniform(g, (case["frames"], 1), 0.3, 1.0)
        p["delta"] = torch.zeros((case["frames"], n, 3), device=DEV)
        p["delta"][..., 0] = 10.0 * (_uniform(g, (case["frames"], n), 0, 1) >= share)
    if case["sh"] >= 0:
        sh = _normal(g, (n, (case["sh"] + 1) ** 2), 0.03)
        sh[:, 0] = (p["amplitude"] - 0.5) * (2.0 * math.sqrt(math.pi))
        p["sh"], p["amplitude"] = sh, None
    return p


def _raw_frames(case, g):
    """Captured raw quartets of a slanted wall and a disc moving before it."""
    b, w, h = case["frames"], case["width"], case["height"]
    y, x = torch.meshgrid(torch.linspace(-1, 1, h, device=DEV), torch.linspace(-1, 1, w, device=DEV),
                          indexing="ij")
    t = torch.linspace(0, 1, b, device=DEV)[:, None, None]
    disc = ((x - 1.2 * (t - 0.5)) ** 2 + (y - 0.2) ** 2) < 0.1
    d = torch.where(disc, 2.5, 4.5 + 0.4 * x + 0.2 * y)
    a = torch.where(disc, 0.8, 0.5) / d ** 2
    psi = (4 * math.pi * FREQS[0] / C_LIGHT) * d
    q = [a * torch.sin(psi + o) for o in QUARTET] + [a]
    return torch.stack(q, 1) + _normal(g, (b, len(q), h, w), 0.002)


def _render_inputs(case, seed):
    g = _generator(seed)
    p = _gaussians(case, g)
    bg = _uniform(g, (case["frames"], _channels(case)), -1, 1)
    dout = None
    if case["backward"]:
        dout = _normal(g, (case["frames"], _channels(case), case["height"], case["width"]))
    return p, bg, dout


def _mlp_inputs(case, seed):
    """Packed parameters ([W, b] per layer, the head last), positions, dL/d(offset)."""
    g = _generator(seed)
    parts = []
    for layer in range(MLP_DEPTH):
        fan = MLP_USED if layer == 0 else MLP_WIDTH
        wt = torch.zeros((MLP_WIDTH, MLP_IN if layer == 0 else MLP_WIDTH), device=DEV)
        wt[:, :fan] = _normal(g, (MLP_WIDTH, fan), math.sqrt(2.0 / (fan + MLP_WIDTH)))
        parts += [wt.reshape(-1), _normal(g, (MLP_WIDTH,), 0.01)]
    parts += [_normal(g, (3 * MLP_WIDTH,), 0.02), _normal(g, (3,), 0.01)]
    means = _uniform(g, (case["n"], 3), -2.0, 4.0)
    times = [float(t) for t in np.linspace(0, 1, case["frames"]).astype(np.float32)]
    dd = _normal(g, (case["frames"], case["n"], 3)) if case["train"] else None
    return torch.cat(parts), means, times, dd


def _footprints(case, seed):
    """A caller's footprints: one set of discs, the seed's own order and depths (so that
    the lists' total length, and with it the outputs' shape, is the case's own)."""
    g = _generator(0)
    shape = (case["frames"], case["n"])
    u = _uniform(g, shape, -0.05, 1.05) * case["width"]
    v = _uniform(g, shape, -0.05, 1.05) * case["height"]
    sigma = _normal(g, shape, 0.3, -3.4).exp() * _focal(case["width"]) / _uniform(g, shape, 1.0, 3.0)
    radius = torch.ceil(SIGMA_CUT * sigma).to(torch.int32)
    radius = torch.where(_uniform(g, shape, 0, 1) < 0.1, 0, radius)
    g = _generator(seed + 1)
    order = torch.argsort(_uniform(g, shape, 0, 1), dim=1)
    u, v, radius = (t.gather(1, order).contiguous() for t in (u, v, radius))
    return u, v, radius, _uniform(g, shape, 1.0, 3.0)


def prepare(case, seed):
    from paper_2505_05356_gb300 import fit, gftorf, mlp

    if case["kind"] == "bin":
        return dict(case=case, args=_footprints(case, seed))
    if case["kind"] == "mlp":
        theta, means, times, dd = _mlp_inputs(case, seed)
        net = mlp.DeformationMLP(case["n"], case["frames"], 1.0 / mlp.unambiguous_range(FREQS[0]))
        return dict(case=case, net=net, theta=theta, means=means, times=times, dd=dd)

    cam, focal = _pose(case), _focal(case["width"])
    frames = [gftorf.make_frame(focal, focal, case["width"] / 2, case["height"] / 2, cam, NEAR, t,
                                phase, bracket) for t, phase, bracket in _frames_of(case)]
    consts = gftorf.make_consts()
    tile = (case["tile_w"], case["tile_h"])
    if case["kind"] == "fit":
        g = _generator(seed)
        p = _gaussians(case, g)
        loop = fit.FitLoop(p, frames, gftorf.make_sensor(FREQS[:1], QUARTET), consts,
                           _raw_frames(case, g), tile=tile, render_mode=int(case["persistent"]),
                           seed=int(seed))
        loop.capture()
        return dict(case=case, loop=loop)

    p, bg, dout = _render_inputs(case, seed)
    flags = gftorf.FLAG_PHASOR | gftorf.FLAG_DEPTH if case["extra"] else 0
    r = gftorf.Renderer(case["n"], case["frames"], case["width"], case["height"], case["freqs"],
                        len(_offsets(case)), tile=tile, render_mode=int(case["persistent"]),
                        pixels_per_thread=case["ppt"], flags=flags,
                        n_sh=0 if case["sh"] < 0 else (case["sh"] + 1) ** 2)
    sensor = gftorf.make_sensor(FREQS[:case["freqs"]], _offsets(case))
    r.fit_capacity(p, frames, sensor, consts, bg)
    s = dict(case=case, r=r, p=p, bg=bg, dout=dout, setup=(frames, sensor, consts))
    if case["how"] == "autograd":
        s["leaves"] = [t.requires_grad_() for t in [bg] + [p[k] for k in sorted(p)] if t is not None]
    elif case["how"] == "graph":
        out = torch.empty((case["frames"], r.C, case["height"], case["width"]), device=DEV)
        grads = r.alloc_grads(p, bg) if case["backward"] else None

        def step():
            r.preprocess(p, *s["setup"])
            r.render_fwd(bg, out)
            if grads is not None:
                r.render_bwd(p, bg, dout, grads)

        step()
        torch.cuda.synchronize()
        s["graph"] = torch.cuda.CUDAGraph()
        with torch.cuda.graph(s["graph"]):
            step()
        s["result"] = dict(out=out, grads=grads)
    return s


def run(s):
    from paper_2505_05356_gb300 import gftorf

    case = s["case"]
    if case["kind"] == "bin":
        return gftorf.sort_footprints(*s["args"], case["width"], case["height"],
                                      tile=(case["tile_w"], case["tile_h"]))
    if case["kind"] == "mlp":
        net, args = s["net"], (s["theta"], s["means"], s["times"])
        if not case["train"]:
            return net.infer(*args)
        delta = net.forward(*args)
        d_theta, d_means = net.backward(*args, s["dd"])
        return dict(delta=delta, d_theta=d_theta, d_means=d_means)
    if case["kind"] == "fit":
        loop = s["loop"]
        loop.run(1)
        return dict(out=loop.out, grads=loop.param_grads(), params=loop.p)
    r, p, bg = s["r"], s["p"], s["bg"]
    if case["how"] == "graph":
        s["graph"].replay()
        return s["result"]
    if case["how"] == "autograd":
        out = gftorf.render_ctof(r, *s["setup"], bg, p)
        if not case["backward"]:
            return dict(out=out)
        grads = torch.autograd.grad(out, s["leaves"], s["dout"])
        return dict(out=out, grads=dict(zip(["bg"] + [k for k in sorted(p) if p[k] is not None],
                                            grads)))
    r.preprocess(p, *s["setup"])
    out = r.render_fwd(bg)
    if not case["backward"]:
        return dict(out=out)
    return dict(out=out, grads=r.render_bwd(p, bg, s["dout"]))


# --- what a pass cannot do without ----------------------------------------------------
def _pairs(case):
    """Estimated (pixel, Gaussian) pairs a frame's pixels composite or reject near the
    edge: those that reach alpha_min, until the pixel is opaque (about 70 at the
    benchmark's opacities)."""
    f = _focal(case["width"])
    z0, z1 = (1.0, 6.0) if case["kind"] == "fit" else (case["z0"], case["z1"])
    per_px = case["n"] * 0.65 * math.pi * 8.0 * (0.032 * f) ** 2 / (z0 * z1) / (
        case["width"] * case["height"])
    return case["frames"] * case["width"] * case["height"] * min(per_px, 70.0)


def work(case):
    n, b = case["n"], case["frames"]
    if case["kind"] == "mlp":
        macs = MLP_WIDTH * (MLP_USED + (MLP_DEPTH - 1) * MLP_WIDTH + 3)
        params = 4 * (MLP_WIDTH * (MLP_IN + 1) + (MLP_DEPTH - 1) * MLP_WIDTH * (MLP_WIDTH + 1) +
                      3 * (MLP_WIDTH + 1))
        if not case["train"]:
            return dict(bytes=12 * n + 12 * n * b + params, flops=2 * macs * n * b)
        return dict(bytes=24 * n + 24 * n * b + 2 * params, flops=6 * macs * n * b)
    if case["kind"] == "bin":
        f = _focal(case["width"])
        r = SIGMA_CUT * 0.035 * f / 2.0
        tiles = (2 * r / case["tile_w"] + 1) * (2 * r / case["tile_h"] + 1)
        return dict(bytes=16 * n * b + 12 * 0.9 * n * b * tiles, flops=0)
    px = b * case["width"] * case["height"]
    if case["kind"] == "fit":  # parameters, both moments, gradients; raw frames; image and its gradient
        return dict(bytes=84 * n * 7 + 4 * 5 * px * 3, flops=80 * _pairs(case))
    per_g = 4 * (11 + (9 if case["moving"] else 0) +
                 (1 if case["sh"] < 0 else (case["sh"] + 1) ** 2))
    data = per_g * n + (12 * n * b if case["hidden"] else 0)
    image = 4 * _channels(case) * px
    if not case["backward"]:
        return dict(bytes=data + image, flops=20 * _pairs(case))
    return dict(bytes=2 * data + 2 * image, flops=80 * _pairs(case))


# --- the same in 64 bits, in plain torch ---------------------------------------------
def _sh_basis(w):
    """Real spherical harmonics of degree 0..3, orthonormal, no Condon-Shortley phase."""
    x, y, z = w.unbind(-1)
    pi = math.pi
    k1, k2, k3 = math.sqrt(3 / (4 * pi)), math.sqrt(15 / pi) / 2, math.sqrt(21 / (2 * pi)) / 4
    a, c = math.sqrt(35 / (2 * pi)) / 4, math.sqrt(105 / pi) / 2
    return torch.stack([
        torch.full_like(x, 1 / (2 * math.sqrt(pi))), k1 * y, k1 * z, k1 * x, k2 * x * y, k2 * y * z,
        math.sqrt(5 / pi) / 4 * (2 * z * z - x * x - y * y), k2 * x * z, k2 / 2 * (x * x - y * y),
        a * y * (3 * x * x - y * y), c * x * y * z, k3 * y * (4 * z * z - x * x - y * y),
        math.sqrt(7 / pi) / 4 * z * (2 * z * z - 3 * x * x - 3 * y * y),
        k3 * x * (4 * z * z - x * x - y * y), c / 2 * z * (x * x - y * y),
        a * x * (x * x - 3 * y * y)], -1)


def _project(case, p, b):
    """(record (N, 6 + features + 1): u, v, conic, opacity, features, distance; sort
    depth; visible; tile rectangle; half extents of the alpha_min ellipse) of frame b."""
    w, h, f = case["width"], case["height"], _focal(case["width"])
    cam = torch.as_tensor(_pose(case), device=DEV).double()
    rot, tr = cam[:, :3], cam[:, 3]
    t, _, bracket = (float(np.float32(v)) if isinstance(v, float) else v for v in _frames_of(case)[b])
    x = p["means"]
    if p.get("coeffs") is not None:
        if bracket is not None:
            t0, t1 = (float(np.float32(v)) for v in bracket)
            tp = [((t1 - t) * t0 ** k + (t - t0) * t1 ** k) / (t1 - t0) for k in (1, 2, 3)]
        else:
            tp = [t, t ** 2, t ** 3]
        x = x + sum(p["coeffs"][:, k] * tp[k] for k in range(3))
    if p.get("delta") is not None:
        x = x + p["delta"][b]
    q = x @ rot.T + tr
    z = q[:, 2]
    e = x + rot.T @ tr
    d = e.norm(dim=1)
    a, i, j, k = torch.nn.functional.normalize(p["quats"], dim=1).unbind(1)
    rq = torch.stack([1 - 2 * (j * j + k * k), 2 * (i * j - a * k), 2 * (i * k + a * j),
                      2 * (i * j + a * k), 1 - 2 * (i * i + k * k), 2 * (j * k - a * i),
                      2 * (i * k - a * j), 2 * (j * k + a * i), 1 - 2 * (i * i + j * j)],
                     1).reshape(-1, 3, 3)
    m = rq * p["scales"][:, None, :]
    tx = (q[:, 0] / z).clamp(-GUARD * 0.5 * w / f, GUARD * 0.5 * w / f)
    ty = (q[:, 1] / z).clamp(-GUARD * 0.5 * h / f, GUARD * 0.5 * h / f)
    zero = torch.zeros_like(z)
    jac = torch.stack([f / z, zero, -f * tx / z, zero, f / z, -f * ty / z], 1).reshape(-1, 2, 3)
    jm = (jac @ rot) @ m
    cov = jm @ jm.transpose(1, 2)
    c00, c01, c11 = cov[:, 0, 0] + DILATION, cov[:, 0, 1], cov[:, 1, 1] + DILATION
    det = c00 * c11 - c01 * c01
    u, v = f * q[:, 0] / z + w / 2, f * q[:, 1] / z + h / 2
    refl = p.get("amplitude")
    if p.get("sh") is not None:
        basis = _sh_basis(e / d[:, None])[:, :p["sh"].shape[1]]
        refl = (0.5 + (p["sh"] * basis).sum(1)).clamp(min=0.0)
    amp = refl / d ** 2
    feats = []
    for fr in FREQS[:case.get("freqs", 1)]:
        psi = 4 * math.pi * float(np.float32(fr)) / C_LIGHT * d
        feats += [amp * torch.sin(psi), amp * torch.cos(psi)]
    rec = torch.stack([u, v, c11 / det, -c01 / det, c00 / det, p["opacity"]] + feats + [amp, d], 1)
    with torch.no_grad():
        mid = 0.5 * (c00 + c11)
        rad = torch.ceil(SIGMA_CUT * torch.sqrt(mid + torch.sqrt((mid * mid - det).clamp(min=0.1))))
        rect = []
        for at, size, tiles in ((u, case["tile_w"], -(-w // case["tile_w"])),
                                (v, case["tile_h"], -(-h // case["tile_h"]))):
            c, r = at.float(), rad.float()
            rect += [torch.floor((c - r) / size).clamp(0, tiles),
                     (torch.floor((c + r) / size) + 1).clamp(0, tiles)]
        kappa = 2 * torch.log(p["opacity"] / ALPHA_MIN)
        ext = [torch.sqrt(kappa.clamp(min=0) * c) + 1.0 for c in (c00, c11)]
        visible = (z > NEAR) & (det > 0) & (kappa >= 0) & (rect[0] < rect[1]) & (rect[2] < rect[3])
    return rec, z.detach().float(), visible, rect, ext


def _composite(r, member, px, py, state):
    """Adds records r (front to back) to the per-pixel state (features, depth, T)."""
    acc, acc_d, trans, alive = state
    dx, dy = r[:, 0, None] - px, r[:, 1, None] - py
    power = -0.5 * (r[:, 2, None] * dx * dx + r[:, 4, None] * dy * dy) - r[:, 3, None] * dx * dy
    alpha = (r[:, 5, None] * torch.exp(power)).clamp(max=ALPHA_MAX)
    alpha = torch.where(member & (power <= 0) & (alpha >= ALPHA_MIN), alpha, 0.0)
    with torch.no_grad():
        after = trans * torch.exp(torch.cumsum(torch.log1p(-alpha), 0))
        on = alive & (after >= T_MIN)  # once below, a pixel stays below
    alpha = alpha * on
    logs = torch.cumsum(torch.log1p(-alpha), 0)
    before = trans * torch.exp(torch.cat([torch.zeros_like(logs[:1]), logs[:-1]]))
    at = alpha * before
    feats = r[:, 6:-1]
    return (acc + feats.T @ (at * before), acc_d + r[:, -1] @ at, trans * torch.exp(logs[-1]), on[-1])


def _image(case, state, bg, b):
    acc, acc_d, trans, _ = state
    freqs, phase = case.get("freqs", 1), float(np.float32(_frames_of(case)[b][1]))
    out, c = [], 0
    for f in range(freqs):
        for o in _offsets(case):
            phi = float(np.float32(o)) + phase
            out.append(math.cos(phi) * acc[2 * f] + math.sin(phi) * acc[2 * f + 1] + bg[c] * trans)
            c += 1
    out.append(acc[2 * freqs] + bg[c] * trans)
    if case.get("extra"):
        for f in range(freqs):
            out += [2 * acc[2 * f + 1] + bg[c + 1] * trans, 2 * acc[2 * f] + bg[c + 2] * trans]
            c += 2
        out.append(acc_d)
    return torch.stack(out)


def _exact_frame(case, p, bg, b, dout_of):
    """Frame b's image; with dout_of (image block, y slice, x slice -> dL/d image
    block) also its gradients, added to the leaves' .grad."""
    w, h = case["width"], case["height"]
    rec, z, visible, rect, ext = _project(case, p, b)
    flat, order = rec.detach(), torch.argsort(z, stable=True)
    order = order[visible[order]]
    keys = [t[order] for t in rect + ext] + [flat[order, 0], flat[order, 1]]
    grad, bg_b = torch.zeros_like(flat), bg[b].detach()
    image = torch.empty((_channels(case), h, w), device=DEV, dtype=torch.float64)
    g_bg = torch.zeros_like(bg_b)
    tw, th = case["tile_w"], case["tile_h"]
    xa, xb, ya, yb, ex, ey, u, v = keys
    for y0 in range(0, h, BLOCK):
        for x0 in range(0, w, BLOCK):
            ys, xs = slice(y0, min(y0 + BLOCK, h)), slice(x0, min(x0 + BLOCK, w))
            hit = ((xa <= (xs.stop - 1) // tw) & (xb > x0 // tw) & (ya <= (ys.stop - 1) // th) &
                   (yb > y0 // th) & (u + ex >= x0) & (u - ex <= xs.stop) & (v + ey >= y0) &
                   (v - ey <= ys.stop)).nonzero()[:, 0]
            py, px = torch.meshgrid(torch.arange(y0, ys.stop, device=DEV, dtype=torch.float64) + 0.5,
                                    torch.arange(x0, xs.stop, device=DEV, dtype=torch.float64) + 0.5,
                                    indexing="ij")
            px, py = px.reshape(-1), py.reshape(-1)
            tx, ty = torch.floor(px / tw), torch.floor(py / th)
            one = torch.ones_like(px)
            state = (torch.zeros((flat.shape[1] - 7, px.numel()), device=DEV, dtype=torch.float64),
                     torch.zeros_like(px), one, one > 0)
            parts = []
            back = bg_b.clone().requires_grad_(dout_of is not None)
            with torch.set_grad_enabled(dout_of is not None):
                for at in range(0, hit.numel(), 384):
                    k = hit[at:at + 384]
                    # a pixel sees the records whose tile rectangle holds its tile
                    member = ((xa[k, None] <= tx) & (xb[k, None] > tx) & (ya[k, None] <= ty) &
                              (yb[k, None] > ty))
                    r = flat[order[k]].requires_grad_(dout_of is not None)
                    state = _composite(r, member, px, py, state)
                    parts.append((order[k], r))
                    if not bool(state[3].any()):
                        break
                out = _image(case, state, back, b)
            part = out.detach().reshape(-1, ys.stop - y0, xs.stop - x0)
            image[:, ys, xs] = part
            if dout_of is not None:
                got = torch.autograd.grad(out, [back] + [r for _, r in parts],
                                          dout_of(part, ys, xs).reshape(out.shape))
                g_bg += got[0]
                for (i, _), gr in zip(parts, got[1:]):
                    grad.index_add_(0, i, gr)
    if dout_of is not None:
        bg.grad[b] += g_bg
        rec.backward(torch.where(visible[:, None], grad, 0.0))
    return image


def _double(p):
    return {k: None if t is None else t.detach().double().requires_grad_() for k, t in p.items()}


def _exact_render(case, seed):
    p32, bg32, dout = _render_inputs(case, seed)
    p, bg = _double(p32), bg32.double().requires_grad_()
    for t in [bg] + [t for t in p.values() if t is not None]:
        t.grad = torch.zeros_like(t)
    out = []
    for b in range(case["frames"]):
        of = None if dout is None else (lambda part, ys, xs, b=b: dout[b, :, ys, xs].double())
        with torch.set_grad_enabled(dout is not None):
            out.append(_exact_frame(case, p, bg, b, of))
    out = torch.stack(out)
    if dout is None:
        return dict(out=out)
    return dict(out=out, grads={k: t.grad for k, t in list(p.items()) + [("bg", bg)] if t is not None})


def _background(seed, count):
    """The first iteration's background: SplitMix64's first `count` outputs, 24 bits each."""
    with np.errstate(over="ignore"):
        x = np.uint64(seed) + np.arange(1, count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x = x ^ (x >> np.uint64(31))
    return (x >> np.uint64(40)).astype(np.float64) * 2.0 ** -23 - 1.0


def _exact_fit(case, seed):
    g = _generator(seed)
    p = _double(_gaussians(case, g))
    raw = _raw_frames(case, g)
    b, c = case["frames"], len(QUARTET) + 1
    bg = torch.as_tensor(_background(int(seed), b * c), device=DEV).reshape(b, c).requires_grad_()
    for t in [bg] + [t for t in p.values() if t is not None]:
        t.grad = torch.zeros_like(t)
    mean = 2.0 / (b * (c - 1) * case["width"] * case["height"])

    def loss_grad(part, ys, xs, i):
        d = mean * (part - raw[i, :, ys, xs].double())
        d[c - 1] = 0.0  # the ambient channel is not in the loss
        return d

    out = torch.stack([_exact_frame(case, p, bg, i, lambda part, ys, xs, i=i: loss_grad(part, ys, xs, i))
                       for i in range(b)])
    grads = {k: p[k].grad for k in FIT_LRS}
    params = {k: None if t is None else t.detach() for k, t in p.items()}
    for k, lr in FIT_LRS.items():  # Adam's first step: both moments are the gradient's own
        lo, hi = FIT_BOUNDS.get(k, (-math.inf, math.inf))
        params[k] = (params[k] - lr * grads[k] / (grads[k].abs() + 1e-15)).clamp(lo, hi)
    return dict(out=out, grads=grads, params=params)


def _exact_mlp(case, seed):
    """In 64 bits but for the network's own BF16 operands: encoding, weights,
    activations and back-propagated pre-activation gradients are rounded where the
    mixed-precision network rounds them."""
    theta, means, times, dd = _mlp_inputs(case, seed)
    scale = float(np.float32(2.0 * FREQS[0] / C_LIGHT))

    def bf(t):
        return t.to(torch.bfloat16).double()

    layers, at = [], 0
    for rows, cols in [(MLP_WIDTH, MLP_IN)] + [(MLP_WIDTH, MLP_WIDTH)] * (MLP_DEPTH - 1) + [(3, MLP_WIDTH)]:
        wt = bf(theta[at:at + rows * cols]).reshape(rows, cols)
        layers.append((wt, theta[at + rows * cols:at + rows * (cols + 1)].double()))
        at += rows * (cols + 1)
    grads = [[torch.zeros_like(wt), torch.zeros_like(bias)] for wt, bias in layers]
    delta, d_means = [], torch.zeros((case["n"], 3), device=DEV, dtype=torch.float64)
    band = (2.0 ** torch.arange(MLP_BANDS, device=DEV, dtype=torch.float64)) * math.pi
    for b, t in enumerate(times):
        x = means.double() * scale
        arg = band[None, :, None] * x[:, None, :]
        enc = torch.zeros((case["n"], MLP_IN), device=DEV, dtype=torch.float64)
        enc[:, :3] = x
        enc[:, 3:63] = torch.stack([torch.sin(arg), torch.cos(arg)], 2).reshape(-1, 60)
        enc[:, 63] = t
        enc[:, 64:84] = torch.stack([torch.sin(band * t), torch.cos(band * t)], 1).reshape(-1)
        hidden = [bf(enc)]
        for wt, bias in layers[:-1]:
            hidden.append(bf((hidden[-1] @ wt.T + bias).clamp(min=0)))
        delta.append(hidden[-1] @ layers[-1][0].T + layers[-1][1])
        if dd is None:
            continue
        dz = bf(dd[b])
        for i in range(MLP_DEPTH, -1, -1):
            grads[i][0] += dz.T @ hidden[i]
            grads[i][1] += dz.sum(0)
            dh = dz @ layers[i][0]
            dz = bf(dh * (hidden[i] > 0)) if i else dh
        d_arg = dz[:, 3:63].reshape(-1, MLP_BANDS, 2, 3)
        d_means += scale * (dz[:, :3] + (band[None, :, None] * (
            d_arg[:, :, 0] * torch.cos(arg) - d_arg[:, :, 1] * torch.sin(arg))).sum(1))
    delta = torch.stack(delta)
    if dd is None:
        return delta
    return dict(delta=delta, d_means=d_means,
                d_theta=torch.cat([t.reshape(-1) for pair in grads for t in pair]))


def exact(case, seed):
    if case["kind"] == "bin":  # whole numbers
        return None
    if case["kind"] == "mlp":
        # 64-bit products run near 1 TFLOP/s
        return _exact_mlp(case, seed) if work(case)["flops"] <= 8e12 else None
    # blocks of pixels, each a few milliseconds
    blocks = case["frames"] * -(-case["width"] // BLOCK) * -(-case["height"] // BLOCK)
    if blocks > 3000:
        return None
    return _exact_fit(case, seed) if case["kind"] == "fit" else _exact_render(case, seed)
