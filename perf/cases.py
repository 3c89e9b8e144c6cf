"""The work a user of this framework has it do, as cases that can be timed.

Kinds of case (field "kind"):

* step      one training step of the fused render: forward, loss, adjoint, the
            gradients of grid, probes and MLP (the loop of fit.fit_appearance).
* view      one rendered image without gradients, uniform samples.
* proposed  one image with samples placed by the learned proposal (the
            real-time form, fit.render_proposed).
* two_pass  one image by node shading and a march over the node colours.
* proposal  one training step of the proposal (the loop of fit.train_proposal).
* terms     the grid-level part of a training step: Gaussian smoothing, the
            regularisers, probe smoothness, transposed smoothing, Adam.

Scenes have the shapes of the framework's own workloads (an object in a cube,
a standing body in a 1 x 2 x 1 box); all inputs are made on the GPU.
"""
from __future__ import annotations

import math

import torch

import paper_2412_10084_gb300 as ps
from paper_2412_10084_gb300 import fit

DEV = "cuda"
LAMBDAS = dict(sdf=0.2, eik=0.1, normal=0.05, features=0.05, probes=0.2)


def _case(name, kind, **kw):
    """A case with every field: grid nodes per axis (rx, ry, rz), probes per
    axis (px, py, pz), layout of the features (nodes, bf16, planes, bricks),
    sharpness tau, rays, samples per ray,
    share of the bricks that are stored."""
    c = dict(kind=kind, scene="object", rx=256, ry=256, rz=256, px=32, py=32, pz=32,
             layout="nodes", half=False, sh_l=3, n_ang=4, width=32, view_dir=False, tau=64.0,
             rays=1 << 18, samples=256, autograd=False, mask_loss=False, bins=16, occ=64,
             band=0.1, stored=0.0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the smallest configuration: a 64^3 sphere, 4096 rays, through autograd as a
        # script would call it; launches and latency count
        _case("step_sphere64", "step", scene="sphere", rx=64, ry=64, rz=64, px=16, py=16, pz=16,
              width=16, rays=4096, samples=128, autograd=True),
        # the default training step of an object capture, FP32
        _case("step_object256", "step"),
        # human capture in reduced precision: BF16 features, FP16 probes and MLP
        _case("step_human384", "step", scene="body", rx=384, ry=768, rz=384, px=48, py=96, pz=48,
              layout="bf16", half=True, rays=1 << 19),
        # high resolution, 8 angular channels, 512 samples (a quarter of the stress batch)
        _case("step_stress512", "step", rx=512, ry=512, rz=512, px=64, py=64, pz=64,
              layout="bf16", n_ang=8, rays=1 << 18, samples=512),
        # tile tri-plane features, with a mask loss on the weight sum
        _case("step_planes256", "step", layout="planes", mask_loss=True),
        # a 1024^3 grid stored as sparse bricks around the surface
        _case("step_bricks1024", "step", rx=1024, ry=1024, rz=1024, px=64, py=64, pz=64,
              layout="bricks", stored=0.27, tau=256.0),
        # a 1080p frame, FP32, 256 uniform samples
        _case("view_1080p", "view", rays=1920 * 1080),
        # the real-time form of the same frame: reduced precision, 128 placed samples
        _case("proposed_1080p", "proposed", layout="bf16", half=True, rays=1920 * 1080,
              samples=128),
        # the viewer form: shade the nodes near the surface, then march their colours
        _case("two_pass_1080p", "two_pass", rays=1920 * 1080),
        # training the proposal on a batch of rays of the training rig
        _case("proposal_step", "proposal", rays=1 << 15),
        # grid-level terms of a dense training step
        _case("terms_256", "terms"),
        # the same on sparse bricks of a 512^3 grid
        _case("terms_bricks512", "terms", rx=512, ry=512, rz=512, layout="bricks", stored=0.35),
    ]


def _spread(rng, lo, hi):
    """An integer spread over the logarithm of [lo, hi]."""
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "view", "proposed", "two_pass", "proposal",
                       "terms"])
    c = dict(kind=kind, scene=rng.choice(["object", "sphere"]))
    top = 320 if kind in ("step", "terms") else 256
    for a in "xyz":
        c["r" + a] = _spread(rng, 24, top)
        c["p" + a] = rng.randint(4, 40)
    c["view_dir"] = rng.random() < 0.2
    c["tau"] = float(rng.choice([32.0, 64.0, 128.0, 256.0]))
    if kind == "step":
        c["rays"] = _spread(rng, 600, 1 << 18)
        c["samples"] = rng.choice([33, 64, 100, 128, 200, 256, 257])
        c["layout"] = rng.choice(["nodes", "nodes", "bf16", "planes", "bricks"])
        c["autograd"] = rng.random() < 0.5
        c["mask_loss"] = rng.random() < 0.5
        if c["layout"] == "nodes":
            c["width"], c["n_ang"], c["sh_l"] = rng.choice([(16, 4, 3), (32, 4, 3), (32, 8, 3),
                                                            (32, 4, 4)])
        elif c["layout"] == "bf16":
            c["half"] = rng.random() < 0.6
            c["n_ang"] = 4 if c["half"] else 8
            c["autograd"] = False
        elif c["layout"] == "planes":
            c["width"], c["sh_l"] = rng.choice([(16, 3), (32, 3), (32, 4)])
    elif kind in ("view", "proposed", "two_pass"):
        w, h = rng.choice([(320, 180), (641, 479), (800, 600), (1280, 720), (1921, 1079)])
        c["rays"] = w * h - rng.randint(0, 31)
        c["samples"] = rng.choice([64, 96, 128, 160, 192])
        if kind == "proposed":
            c["layout"], c["half"] = rng.choice([("bf16", True), ("nodes", False)])
            c["bins"], c["occ"] = rng.choice([(8, 32), (16, 64), (16, 32)])
        else:
            c["layout"] = rng.choice(["nodes", "bricks"])
            c["band"] = rng.choice([0.02, 0.1, 0.25])
    elif kind == "proposal":
        c["rays"] = _spread(rng, 1000, 1 << 16)
        c["bins"], c["occ"] = rng.choice([(8, 32), (16, 64), (16, 33)])
        c["samples"] = rng.choice([64, 128, 256])
    else:
        c["layout"] = rng.choice(["nodes", "bf16", "planes", "bricks"])
    if c.get("layout") == "bricks":
        c["stored"] = rng.choice([0.3, 0.5, 0.7])
        for a in "xyz":
            c["r" + a] = 16 * rng.randint(4, 20)
    return _case(None, c.pop("kind"), **c)


# ---------------------------------------------------------------------------
# Inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed))
    return g


def _uni(g, *shape, lo=0.0, hi=1.0):
    return torch.rand(*shape, generator=g, device=DEV) * (hi - lo) + lo


def _box(case):
    return (0.0, 0.0, 0.0), ((1.0, 2.0, 1.0) if case["scene"] == "body" else (1.0, 1.0, 1.0))


def _shapes(case, g):
    """Segments with radii (a sphere is a segment of length zero): a, b [n,3], r [n]."""
    if case["scene"] == "sphere":
        c = _uni(g, 1, 3, lo=0.47, hi=0.53)
        return c, c, _uni(g, 1, lo=0.38, hi=0.42)
    if case["scene"] == "body":
        y = torch.linspace(0.3, 1.7, 15, device=DEV)[:, None]
        x = _uni(g, 15, 1, lo=0.38, hi=0.62)
        z = _uni(g, 15, 1, lo=0.42, hi=0.58)
        a = torch.cat([x, y, z], 1)
        return a, a + _uni(g, 15, 3, lo=-0.14, hi=0.14), _uni(g, 15, lo=0.05, hi=0.1)
    a = _uni(g, 32, 3, lo=0.25, hi=0.75)
    long = (torch.arange(32, device=DEV) % 2)[:, None]
    b = a + long * _uni(g, 32, 3, lo=-0.15, hi=0.15)
    return a, b, _uni(g, 32, lo=0.05, hi=0.15)


def _distance(P, shapes, k=0.05):
    """Smooth-min union of the segments at points P [..., 3]."""
    acc = None
    for a, b, r in zip(*shapes):
        ab = b - a
        h = (((P - a) @ ab) / (ab @ ab).clamp(min=1e-12)).clamp(0.0, 1.0)
        d = (P - a - h[..., None] * ab).norm(dim=-1) - r
        if acc is None:
            acc = d
        else:
            m = (k - (acc - d).abs()).clamp(min=0.0) / k
            acc = torch.minimum(acc, d) - m * m * (0.25 * k)
    return acc


def _axes(case):
    lo, hi = _box(case)
    return [torch.linspace(lo[a], hi[a], case["r" + "xyz"[a]], device=DEV) for a in range(3)]


def _sdf(case, shapes, noise, g):
    X, Y, Z = _axes(case)
    out = torch.empty(Z.numel(), Y.numel(), X.numel(), device=DEV)
    for z in range(0, Z.numel(), 32):
        P = torch.stack(torch.meshgrid(Z[z:z + 32], Y, X, indexing="ij")[::-1], -1)
        out[z:z + 32] = _distance(P, shapes)
    if noise:
        out += noise * torch.randn(out.shape, generator=g, device=DEV)
    return out


def _stored(case):
    """Number of stored bricks."""
    return max(1, int(case["stored"] * (case["rx"] * case["ry"] * case["rz"] // 4096)))


def _bricks(case, shapes):
    """Boolean [Bz,By,Bx] of the stored bricks, those nearest to the surface,
    and their SDF [n,16,16,16]."""
    ax = _axes(case)
    B = [x.view(-1, 16) for x in ax]
    mid = [0.5 * (b[:, 0] + b[:, -1]) for b in B]
    P = torch.stack(torch.meshgrid(mid[2], mid[1], mid[0], indexing="ij")[::-1], -1)
    far = _distance(P, shapes).abs()
    keep = torch.zeros_like(far, dtype=torch.bool)
    keep.view(-1)[far.view(-1).topk(_stored(case), largest=False).indices] = True
    bz, by, bx = torch.nonzero(keep, as_tuple=True)
    sdf = torch.empty(bz.numel(), 16, 16, 16, device=DEV)
    for i in range(0, bz.numel(), 4096):
        s = slice(i, i + 4096)
        n = bz[s].numel()
        P = torch.stack([B[0][bx[s]].view(n, 1, 1, 16).expand(n, 16, 16, 16),
                         B[1][by[s]].view(n, 1, 16, 1).expand(n, 16, 16, 16),
                         B[2][bz[s]].view(n, 16, 1, 1).expand(n, 16, 16, 16)], -1)
        sdf[s] = _distance(P, shapes)
    return keep, sdf


def _mlp(g, *sizes):
    """Xavier-uniform layers with small biases, packed W1 b1 W2 b2 W3 b3."""
    parts = []
    for fi, fo in zip(sizes[:-1], sizes[1:]):
        a = math.sqrt(6.0 / (fi + fo))
        parts += [_uni(g, fo * fi, lo=-a, hi=a), _uni(g, fo, lo=-0.05, hi=0.05)]
    return torch.cat(parts)


def _scene(case, g):
    """The packed scene of a case and its SDF (dense [Rz,Ry,Rx] or bricks)."""
    shapes = _shapes(case, g)
    lo, hi = _box(case)
    dims = (case["rx"], case["ry"], case["rz"])
    probes = 0.1 * torch.randn(case["pz"], case["py"], case["px"], case["sh_l"] ** 2,
                               case["n_ang"], generator=g, device=DEV)
    mlp = _mlp(g, 3 + case["n_ang"] + 3, case["width"], case["width"], 3)
    if case["layout"] == "bricks":
        keep, sdf = _bricks(case, shapes)
        feat = 0.1 * torch.randn(*sdf.shape, 3, generator=g, device=DEV)
        scene = ps.sparse_scene(keep.cpu(), sdf, feat, probes, mlp, dims, lo, hi, case["sh_l"],
                                case["width"], empty_sdf=1.0, device=DEV)
        return scene, sdf
    sdf = _sdf(case, shapes, 0.01 if case["scene"] == "sphere" and case["rx"] <= 64 else 0.0, g)
    layout, dtype = ps.FEAT_NODES, ps.F32
    if case["layout"] == "planes":
        tx, ty, tz = ps.tri_tiles(dims)
        layout = ps.FEAT_TRIPLANE
        feat = 1.0 + 0.3 * torch.randn(tz, ty, tx, 3, 16, 16, 3, generator=g, device=DEV)
    else:
        feat = 0.1 * torch.randn(*sdf.shape, 3, generator=g, device=DEV)
        dtype = ps.BF16 if case["layout"] == "bf16" else ps.F32
    grid = ps.pack_grid(ps.grid_desc(dims, lo, hi, 3, dtype, layout), sdf, feat)
    half = ps.F16 if case["half"] else ps.F32
    scene = ps.Scene(grid=grid, probes=probes.half() if case["half"] else probes, mlp=mlp,
                     dims=dims, box_min=lo, box_max=hi, sh_l=case["sh_l"], width=case["width"],
                     feat_dtype=dtype, feat_layout=layout, probe_dtype=half, mlp_dtype=half)
    return scene, sdf


def _look(case, eye):
    """Camera frames (forward, right, up) [n,3] at eye [n,3] towards the box centre."""
    lo, hi = _box(case)
    centre = torch.tensor([(a + b) / 2 for a, b in zip(lo, hi)], device=DEV)
    up = torch.tensor([0.0, 1.0, 0.0] if case["scene"] == "body" else [0.0, 0.0, 1.0], device=DEV)
    f = torch.nn.functional.normalize(centre - eye, dim=-1)
    r = torch.nn.functional.normalize(torch.linalg.cross(f, up.expand_as(f)), dim=-1)
    return centre, f, r, torch.linalg.cross(r, f)


def _eyes(case, g, n):
    """Camera centres on a rig around the box (a ring for a body, else a band
    of the upper hemisphere)."""
    az = 2 * math.pi * _uni(g, n)
    if case["scene"] == "body":
        return torch.stack([0.5 + 2.5 * az.cos(), torch.ones_like(az), 0.5 + 2.5 * az.sin()], -1)
    el = _uni(g, n, lo=0.1, hi=1.2)
    return 0.5 + 2.0 * torch.stack([el.cos() * az.cos(), el.cos() * az.sin(), el.sin()], -1)


def _pixels(case, g, n):
    """n random pixels of 49 cameras (a training batch): origins, directions."""
    eye = _eyes(case, g, 49)
    _, f, r, u = _look(case, eye)
    cam = torch.randint(0, 49, (n,), generator=g, device=DEV)
    tan = math.tan(math.radians(45.0 if case["scene"] != "sphere" else 50.0) / 2)
    x = _uni(g, n, 1, lo=-1.0, hi=1.0) * tan * (1.0 if case["scene"] == "body" else 4 / 3)
    y = _uni(g, n, 1, lo=-1.0, hi=1.0) * tan
    d = torch.nn.functional.normalize(f[cam] + x * r[cam] + y * u[cam], dim=-1)
    return eye[cam].contiguous(), d.contiguous()


def _image(case, g, n):
    """The first n pixels of one 16:9 view, row by row: origins, directions, eye."""
    eye = 0.5 + 1.15 * (_eyes(case, g, 1) - 0.5)
    _, f, r, u = _look(case, eye)
    w = max(1, math.ceil(math.sqrt(n * 16 / 9)))
    h = math.ceil(n / w)
    i = torch.arange(n, device=DEV)
    tan = math.tan(math.radians(45.0) / 2)
    x = ((2 * ((i % w) + 0.5) / w - 1) * tan * w / h)[:, None]
    y = ((1 - 2 * ((i // w) + 0.5) / h) * tan)[:, None]
    d = torch.nn.functional.normalize(f + x * r + y * u, dim=-1)
    return eye.expand(n, 3).contiguous(), d.contiguous(), tuple(float(v) for v in eye[0])


def _params(case, **kw):
    return ps.render_params(case["tau"], case["samples"],
                            ps.DIR_VIEW if case["view_dir"] else ps.DIR_REFLECT, 3, **kw)


def prepare(case, seed):
    g = _gen(seed)
    scene, sdf = _scene(case, g)
    s = {"case": case, "scene": scene, "params": _params(case)}
    kind, n = case["kind"], case["rays"]
    if kind == "step":
        s["o"], s["d"] = _pixels(case, g, n)
        s["target"] = _uni(g, n, 3)
        s["mask"] = (_uni(g, n) < 0.5).float()
        if case["autograd"]:
            for t in (scene.grid, scene.probes, scene.mlp):
                t.requires_grad_(True)
        else:
            s["grads"] = scene.grad_buffers()
    elif kind in ("view", "proposed", "two_pass"):
        s["o"], s["d"], s["eye"] = _image(case, g, n)
        if kind == "two_pass":
            s["colours"] = torch.zeros(case["rz"], case["ry"], case["rx"], 4, dtype=torch.float16,
                                       device=DEV)
    if kind in ("proposed", "proposal"):
        B = case["bins"]
        s["prop"] = fit.Proposal.create(scene, _mlp(g, 7 + 2 * B, 32, 32, B),
                                        occ_res=(case["occ"],) * 3, n_bins=B, mix=0.6, theta=0.0)
    if kind == "proposal":
        s["o"], s["d"] = _pixels(case, g, n)
        s["grad"] = torch.zeros_like(s["prop"].params)
    if kind == "terms":
        gd, pd, _ = scene.descs(3)
        pd.dtype = ps.F32
        w = ps.table_words(gd) if scene.n_bricks else 0
        gg = scene.grad_buffers()[0]
        gg.view(-1)[w:] = 1e-3 * torch.randn(gg.numel() - w, generator=g, device=DEV)
        s_hat = sdf + 0.002 * torch.randn(sdf.shape, generator=g, device=DEV)
        m = 1e-3 * torch.randn(sdf.shape, generator=g, device=DEV)
        s.update(gd=gd, pd=pd, words=w, gg=gg, s_hat=s_hat, d_hat=torch.zeros_like(s_hat), m=m,
                 v=m * m + 1e-6, probes=scene.probes.float(),
                 gp=1e-3 * torch.randn(scene.probes.shape, generator=g, device=DEV))
    return s


# ---------------------------------------------------------------------------
# One pass
# ---------------------------------------------------------------------------

def _run_step(s):
    case, scene, o, d, params = s["case"], s["scene"], s["o"], s["d"], s["params"]
    n = o.shape[0]
    if case["autograd"]:
        rgb, depth, wsum = ps.render(scene, o, d, params)
        loss = ((rgb - s["target"]) ** 2).sum() / n
        if case["mask_loss"]:
            loss = loss + 0.1 * ((wsum - s["mask"]) ** 2).sum() / n
        grads = torch.autograd.grad(loss, (scene.grid, scene.probes, scene.mlp))
        out = {"rgb": rgb.detach(), "depth": depth.detach(), "wsum": wsum.detach()}
    else:
        for t in s["grads"]:
            t.zero_()
        rgb, depth, wsum, logT, live = ps.render_forward(scene, o, d, params, want_live=True)
        d_rgb = (2.0 / n) * (rgb - s["target"])
        d_wsum = (0.2 / n) * (wsum - s["mask"]) if case["mask_loss"] else None
        grads = ps.render_backward(scene, o, d, params, d_rgb, logT, d_wsum=d_wsum,
                                   grads=s["grads"], n_live=live)
        out = {"rgb": rgb, "depth": depth, "wsum": wsum, "logT": logT, "live": live}
    gg = grads[0].view(-1)
    if scene.n_bricks:  # the records; the brick table in front of them is no gradient
        gg = gg[ps.table_words(scene.descs(3)[0]):]
    return {**out, "d_grid": gg, "d_probes": grads[1], "d_mlp": grads[2]}


def _run_terms(s):
    gd, case = s["gd"], s["case"]
    values = s["scene"].grid
    loss = torch.zeros(5, device=DEV)
    ps.sdf_smooth(gd, s["s_hat"], values)
    ps.grid_regularizers(gd, s["s_hat"], values, s["gg"], s["d_hat"], LAMBDAS["sdf"],
                         LAMBDAS["eik"], LAMBDAS["normal"],
                         LAMBDAS["features"] if case["layout"] == "planes" else 0.0,
                         loss=loss[:4])
    ps.probe_smoothness(s["pd"], s["probes"], s["gp"], LAMBDAS["probes"], loss=loss[4:])
    ps.sdf_smooth_adjoint(gd, s["gg"], s["d_hat"], accumulate=True)
    ps.adam_step(s["s_hat"], s["d_hat"], s["m"], s["v"], 100, 1e-3, 0.9, 0.995)
    sdf = values.view(-1).view(torch.float32)[s["words"]:]
    if case["layout"] in ("nodes", "bricks"):
        sdf = sdf[::4]
    else:
        sdf = sdf[:s["s_hat"].numel()]
    return {"loss": loss, "sdf": sdf, "d_grid": s["gg"].view(-1)[s["words"]:],
            "s_hat": s["s_hat"], "m": s["m"], "v": s["v"], "d_probes": s["gp"]}


def run(state):
    s = state
    kind = s["case"]["kind"]
    if kind == "step":
        return _run_step(s)
    if kind == "view":
        return ps.render_forward(s["scene"], s["o"], s["d"], s["params"])
    if kind == "proposed":
        return fit.render_proposed(s["scene"], s["prop"], s["o"], s["d"], s["case"]["samples"],
                                   s["params"])
    if kind == "two_pass":
        colours = ps.shade_nodes(s["scene"], s["eye"], s["case"]["band"], s["params"],
                                 out=s["colours"])
        return (colours,) + ps.render_colour_field(s["scene"], colours, s["o"], s["d"],
                                                   s["params"])
    if kind == "proposal":
        prop, n = s["prop"], s["o"].shape[0]
        s["grad"].zero_()
        hist = ps.weight_histogram(s["scene"], s["o"], s["d"], s["params"], prop.desc.n_bins)
        grad, loss = ps.proposal_backward(s["scene"], prop.desc, prop.params, prop.occ, s["o"],
                                          s["d"], hist, 1e-3, 1.0 / n, grad=s["grad"])
        return hist, grad, loss
    return _run_terms(s)


# ---------------------------------------------------------------------------
# What a pass cannot do without
# ---------------------------------------------------------------------------

# Share of the samples in the box whose opacity is not zero (the SDF falls
# along the ray): only these need a colour.  Shares of the rays that cross the
# box: a training batch of the object or of the body, a view.
OPAQUE = 0.5
CROSS = dict(object=0.46, sphere=0.46, body=0.63, view=0.26)


def work(case):
    kind, n, N = case["kind"], case["rays"], case["samples"]
    inside = n * N * CROSS["view" if kind in ("view", "proposed", "two_pass") else case["scene"]]
    nodes = case["rx"] * case["ry"] * case["rz"]
    if case["layout"] == "bricks":
        nodes = 4096 * _stored(case)
    per_node = {"nodes": 16, "bf16": 12, "planes": 4 + 9, "bricks": 16}[case["layout"]]
    coeffs = case["px"] * case["py"] * case["pz"] * case["sh_l"] ** 2 * case["n_ang"]
    pb = 2 if case["half"] else 4
    n_in, W, B = 6 + case["n_ang"], case["width"], case["bins"]
    sdf = 8 * 2 * 4 + 30                                         # value, gradient, opacity
    colour = (8 * 2 * 3 + 8 * 2 * case["sh_l"] ** 2 * case["n_ang"] +
              2 * (n_in * W + W * W + 3 * W))                    # features, probes, MLP
    prop = 2 * ((7 + 2 * B) * 32 + 32 * 32 + 32 * B)
    ray = 24 + 24
    if kind == "step":
        return {"bytes": nodes * (per_node + 16) + coeffs * (pb + 4) + n * (ray + 12),
                "flops": inside * (2 * sdf + OPAQUE * 3 * colour)}
    if kind == "view":
        return {"bytes": nodes * per_node + coeffs * pb + n * ray,
                "flops": inside * (sdf + OPAQUE * colour)}
    if kind == "proposed":
        return {"bytes": nodes * per_node + coeffs * pb + n * ray,
                "flops": inside * (sdf + OPAQUE * colour) + n * prop}
    if kind == "two_pass":
        near = min(1.0, 3 * case["band"])
        return {"bytes": nodes * (per_node + 8) + coeffs * pb + n * ray,
                "flops": nodes * near * colour + inside * (sdf + OPAQUE * 48)}
    if kind == "proposal":
        return {"bytes": nodes * 4 + n * (24 + 8 * B + 4), "flops": inside * sdf + n * 3 * prop}
    # raw SDF, moments and their updates; s written; d s in and out; d s_hat
    tex = (nodes * 9) if case["layout"] == "planes" else 0
    return {"bytes": nodes * (4 + 4 + 8 + 24) + 3 * tex + 12 * coeffs,
            "flops": nodes * (30 + 120 + 30 + 12)}


# ---------------------------------------------------------------------------
# The same results in 64 bits, in plain torch.  Sample positions and cell
# fractions are those of the method's FP32 sequence (they choose the integer
# cells, so they are part of its definition); everything after is 64-bit.
# ---------------------------------------------------------------------------

def _r(x):
    """Rounded to 32 bits, held in 64."""
    return x.float().double()


class _Exact:
    """Scene of a case in 64 bits: corner gathers, probes, MLP."""

    def __init__(self, case, s):
        self.case, scene = case, s["scene"]
        self.R = torch.tensor(scene.dims, device=DEV).double()
        self.P = torch.tensor(scene.probe_dims, device=DEV).double()
        lo, hi = _box(case)
        self.lo = torch.tensor(lo, device=DEV).double()
        self.hi = torch.tensor(hi, device=DEV).double()
        self.sc = _r((self.R - 1) / _r(self.hi - self.lo))
        self.psc = _r((self.P - 1) / _r(self.hi - self.lo))
        gd, _, _ = scene.descs(3)
        self.table = self.tex = self.feat = None
        flat = scene.grid.detach()
        nodes = case["rx"] * case["ry"] * case["rz"]
        if scene.n_bricks:
            w = ps.table_words(gd)
            nb = nodes // 4096
            self.table = flat.view(-1)[:nb].view(torch.int32).long()
            rec = flat.view(-1)[w:].view(-1, 4)
            self.sdf, self.feat = rec[:, 0], rec[:, 1:]
        elif scene.feat_layout == ps.FEAT_TRIPLANE:
            off = (nodes + 3) // 4 * 4
            self.sdf = flat.view(-1)[:nodes]
            self.tex = flat.view(-1)[off:].view(-1, 4)[:, :3]
            self.off = off
        elif scene.feat_dtype == ps.BF16:
            off = (nodes * 4 + 15) // 16 * 16
            self.sdf = flat[:nodes * 4].view(torch.float32)
            self.feat = flat[off:].view(torch.bfloat16).view(-1, 4)[:, :3]
        else:
            self.sdf, self.feat = flat[:, 0], flat[:, 1:]
        self.probes = scene.probes.detach().reshape(-1, case["sh_l"] ** 2, case["n_ang"])
        self.mlp = scene.mlp.detach().double()

    def cell(self, x, sc, R):
        u = _r(_r(x - self.lo) * sc)
        i = torch.minimum(u.floor().clamp(min=0.0), R - 2)
        return i.long(), _r(u - i)

    def corners(self, i, R):
        """Linear indices [..., 8] of a cell's corners, x fastest."""
        q = torch.arange(8, device=DEV)
        x, y, z = (i[..., a, None] + ((q >> a) & 1) for a in range(3))
        Rx, Ry = int(R[0]), int(R[1])
        return x, y, z, (z * Ry + y) * Rx + x

    def record(self, x, y, z, lin):
        """Record index of nodes, -1 where the brick is not stored."""
        if self.table is None:
            return lin
        Bx, By = self.case["rx"] // 16, self.case["ry"] // 16
        slot = self.table[((z >> 4) * By + (y >> 4)) * Bx + (x >> 4)]
        return torch.where(slot >= 0, slot * 4096 + ((z & 15) << 8) + ((y & 15) << 4) + (x & 15),
                           slot)

    def node_sdf(self, rec):
        s = self.sdf[rec.clamp(min=0)].double()
        return torch.where(rec >= 0, s, torch.ones_like(s))


def _weights(f):
    """Trilinear weights [..., 8] and their derivatives [..., 3, 8] along the
    cell axes."""
    w, dw = None, [None] * 3
    for a in range(3):
        lin = torch.stack([1 - f[..., a], f[..., a]], -1)
        sgn = torch.tensor([-1.0, 1.0], device=DEV, dtype=f.dtype).expand_as(lin)
        one = [lin if b != a else sgn for b in range(3)]

        def mul(p, v):
            return v if p is None else (p[..., None, :] * v[..., :, None]).flatten(-2)
        w = mul(w, lin)
        for b in range(3):
            dw[b] = mul(dw[b], one[b])
    return w, torch.stack(dw, -2)


def _sh(r, sh_l):
    x, y, z = r.unbind(-1)
    Y = [torch.full_like(x, 0.5 / math.sqrt(math.pi))]
    c = math.sqrt(3 / (4 * math.pi))
    Y += [c * y, c * z, c * x]
    a, b = math.sqrt(15 / (4 * math.pi)), math.sqrt(5 / (16 * math.pi))
    Y += [a * x * y, a * y * z, b * (3 * z * z - 1), a * x * z, a / 2 * (x * x - y * y)]
    if sh_l == 4:
        p = math.pi
        c3, c2 = math.sqrt(35 / (32 * p)), math.sqrt(105 / (4 * p))
        c1, c0 = math.sqrt(21 / (32 * p)), math.sqrt(7 / (16 * p))
        Y += [c3 * y * (3 * x * x - y * y), c2 * x * y * z, c1 * y * (5 * z * z - 1),
              c0 * z * (5 * z * z - 3), c1 * x * (5 * z * z - 1), c2 / 2 * z * (x * x - y * y),
              c3 * x * (x * x - 3 * y * y)]
    return torch.stack(Y, -1)


def _layers(flat, sizes):
    out, at = [], 0
    for fi, fo in zip(sizes[:-1], sizes[1:]):
        out.append((flat[at:at + fo * fi].view(fo, fi), flat[at + fo * fi:at + fo * fi + fo]))
        at += fo * fi + fo
    return out


def _colour(case, mlp, g, v, fs, pv, pw):
    """Colours [m,3]: normal from gradient g, view v, features fs [m,3], probe
    corner coefficients pv [m,8,L,A] with weights pw [m,8]."""
    nrm = g / (g.square().sum(-1, keepdim=True) + 1e-24).sqrt()
    ndv = (nrm * v).sum(-1, keepdim=True)
    r = v if case["view_dir"] else 2 * ndv * nrm - v
    b = torch.einsum("mq,mqla->mla", pw, pv)
    fa = torch.einsum("ml,mla->ma", _sh(r, case["sh_l"]), b)
    om = 1 - ndv
    x = torch.cat([fs, fa, om, om * om, om * om * om], -1)
    W = case["width"]
    (W1, b1), (W2, b2), (W3, b3) = _layers(mlp, (6 + case["n_ang"], W, W, 3))
    h = torch.relu(x @ W1.T + b1)
    h = torch.relu(h @ W2.T + b2)
    return torch.sigmoid(h @ W3.T + b3)


def _texels(E, x):
    """Tri-plane texel indices [m,3,4] and bilinear weights of points x."""
    u = _r(_r(x - E.lo) * E.sc)
    T = torch.tensor(ps.tri_tiles((E.case["rx"], E.case["ry"], E.case["rz"])), device=DEV)
    t = torch.minimum((u / 16).floor().clamp(min=0.0), (T - 1).double())
    tau = _r(_r(u - 16 * t) - 0.5).clamp(0.0, 15.0)
    i = tau.floor().clamp(max=14.0)
    f, i, t = _r(tau - i), i.long(), t.long()
    base = ((t[:, 2] * T[1] + t[:, 1]) * T[0] + t[:, 0]) * 768
    idx, wt = [], []
    for p in range(3):
        a, b = (1 if p == 2 else 2), (1 if p == 0 else 0)
        at = base + p * 256 + i[:, a] * 16 + i[:, b]
        idx.append(torch.stack([at, at + 1, at + 16, at + 17], -1))
        fr, fc = f[:, a], f[:, b]
        wt.append(torch.stack([(1 - fr) * (1 - fc), (1 - fr) * fc, fr * (1 - fc), fr * fc], -1))
    return torch.stack(idx, 1), torch.stack(wt, 1)


def _segment(E, o, d):
    flat = d == 0
    t0 = _r(_r(E.lo - o) / d)
    t1 = _r(_r(E.hi - o) / d)
    inf = torch.full_like(t0, math.inf)
    near = torch.where(flat, -inf, torch.minimum(t0, t1)).amax(-1)
    far = torch.where(flat, inf, torch.maximum(t0, t1)).amin(-1)
    out = (flat & ((o < E.lo) | (o > E.hi))).any(-1)
    tn = near.clamp(min=0.0)
    return tn, far, (far > tn) & ~out


def _distances(E, o, d, N, q):
    """Distances [n, N+1] of the rays' points and which rays hit the box."""
    tn, tf, hit = _segment(E, o, d)
    k = torch.arange(N + 1, device=DEV).double()
    if q is None:
        dt = _r(_r(tf - tn) / N)
        t = _r(k * dt[:, None] + tn[:, None])
    else:  # quantiles of the bin densities
        B = q.shape[1]
        c = q.cumsum(1) - q
        u = (k / N).expand(q.shape[0], -1).contiguous()
        b = (torch.searchsorted(c, u, right=True) - 1).clamp(0, B - 1)
        frac = ((u - c.gather(1, b)) / q.gather(1, b)).clamp(max=1.0)
        t = tn[:, None] + (b + frac) * ((tf - tn) / B)[:, None]
        t = _r(t)
        t[:, 0], t[:, -1] = tn, tf
    return torch.where(hit[:, None], t, torch.zeros_like(t)), hit


def _log_phi(y):
    """log of the logistic function."""
    return -(torch.relu(-y) + torch.log1p(torch.exp(-y.abs())))


def _render(E, o, d, t, hit, leaves=None, colours=None):
    """rgb, depth, wsum, logT of a chunk of rays; `leaves` collects what the
    result depends on, for the gradients."""
    case, tau = E.case, E.case["tau"]
    n, N = t.shape[0], t.shape[1] - 1
    x = _r(t[..., None] * d[:, None] + o[:, None])
    i, f = E.cell(x, E.sc, E.R)
    cx, cy, cz, lin = E.corners(i, E.R)
    rec = E.record(cx, cy, cz, lin)
    v = E.node_sdf(rec)
    if leaves is not None:
        v.requires_grad_(True)
        leaves["v"], leaves["rec"] = v, rec
    w, dw = _weights(f)
    s = (w * v).sum(-1)
    lp = _log_phi(tau * s)
    lam = torch.minimum(lp[:, 1:] - lp[:, :-1], torch.zeros((), device=DEV, dtype=s.dtype))
    lam = lam * hit[:, None]
    alpha = -torch.expm1(lam)
    cum = lam.cumsum(1)
    wgt = torch.exp(cum - lam) * alpha
    on = (alpha.detach() > 1e-13).nonzero(as_tuple=True)  # the others' colours reach no bit
    if colours is not None:
        c = (w[:, :-1][on][..., None] * colours[lin[:, :-1][on]].double()).sum(1)
    else:
        g = (dw[:, :-1][on] * v[:, :-1][on][:, None, :]).sum(-1) * E.sc
        if E.tex is not None:
            ti, tw = _texels(E, x[:, :-1][on])
            tv = E.tex[ti].double()
            if leaves is not None:
                tv.requires_grad_(True)
                leaves["tv"], leaves["ti"] = tv, ti
            fs = (tw[..., None] * tv).sum(2).prod(1)
        else:
            fr = rec[:, :-1][on]
            fv = E.feat[fr.clamp(min=0)].double() * (fr >= 0)[..., None]
            if leaves is not None:
                fv.requires_grad_(True)
                leaves["fv"], leaves["fr"] = fv, fr
            fs = (w[:, :-1][on][..., None] * fv).sum(1)
        pi, pf = E.cell(x[:, :-1][on], E.psc, E.P)
        pw, _ = _weights(pf)
        pr = E.corners(pi, E.P)[3]
        pv = E.probes[pr].double()
        mlp = E.mlp.clone()
        if leaves is not None:
            pv.requires_grad_(True)
            mlp.requires_grad_(True)
            leaves["pv"], leaves["pr"], leaves["mlp"] = pv, pr, mlp
        c = _colour(case, mlp, g, -d[on[0]], fs, pv, pw)
    rgb = torch.zeros(n, 3, dtype=torch.float64, device=DEV)
    rgb = rgb.index_add(0, on[0], wgt[on][:, None] * c)
    return rgb, (wgt * t[:, :-1]).sum(1), wgt.sum(1), cum[:, -1]


def _chunks(case, budget):
    per = max(1, budget // case["samples"])
    return [(i, min(case["rays"], i + per)) for i in range(0, case["rays"], per)]


def _exact_step(case, s):
    E, n = _Exact(case, s), case["rays"]
    L, A = case["sh_l"] ** 2, case["n_ang"]
    gs = torch.zeros(E.sdf.numel(), dtype=torch.float64, device=DEV)
    gf = torch.zeros(E.sdf.numel() if E.tex is None else E.tex.shape[0], 3, dtype=torch.float64,
                     device=DEV)
    gp = torch.zeros(E.probes.shape[0], L * A, dtype=torch.float64, device=DEV)
    gm = torch.zeros_like(E.mlp)
    outs = []
    for i, j in _chunks(case, 1 << 20):
        o, d = s["o"][i:j].double(), s["d"][i:j].double()
        t, hit = _distances(E, o, d, case["samples"], None)
        lv = {}
        rgb, depth, wsum, logT = _render(E, o, d, t, hit, lv)
        loss = ((rgb - s["target"][i:j].double()) ** 2).sum() / n
        if case["mask_loss"]:
            loss = loss + 0.1 * ((wsum - s["mask"][i:j].double()) ** 2).sum() / n
        keys = [k for k in ("v", "fv", "tv", "pv", "mlp") if k in lv]
        got = dict(zip(keys, torch.autograd.grad(loss, [lv[k] for k in keys])))
        rec = lv["rec"].reshape(-1)
        gs.index_add_(0, rec.clamp(min=0), got["v"].reshape(-1) * (rec >= 0))
        at = lv["ti"] if E.tex is not None else lv["fr"]
        val = got["tv"] if E.tex is not None else got["fv"] * (at >= 0)[..., None]
        gf.index_add_(0, at.reshape(-1).clamp(min=0), val.reshape(-1, 3))
        gp.index_add_(0, lv["pr"].reshape(-1), got["pv"].reshape(-1, L * A))
        gm += got["mlp"]
        outs.append([v.detach() for v in (rgb, depth, wsum, logT)])
        del lv, got, loss
    rgb, depth, wsum, logT = (torch.cat(v) for v in zip(*outs))
    if E.tex is not None:
        flat = torch.zeros(E.off + 4 * gf.shape[0], dtype=torch.float64, device=DEV)
        flat[:gs.numel()] = gs
        flat[E.off:].view(-1, 4)[:, :3] = gf
    else:
        flat = torch.cat([gs[:, None], gf], 1).view(-1)
    out = {"rgb": rgb, "depth": depth, "wsum": wsum}
    if not case["autograd"]:
        out.update(logT=logT, live=None)
    return {**out, "d_grid": flat, "d_probes": gp.view(s["scene"].probes.shape), "d_mlp": gm}


def _features(case, s, E, o, d):
    """The proposal's inputs [n, 7 + 2B] of rays (occupancy looked up at FP32
    positions)."""
    prop = s["prop"]
    B, S, res = prop.desc.n_bins, prop.desc.n_sub, case["occ"]
    tn, tf, hit = _segment(E, o, d)
    bits = prop.occ.long() & 0xFFFFFFFF
    seg = _r(_r(tf - tn) / (B * S))
    k = torch.arange(B * S, device=DEV).double() + 0.5
    t = _r(k * seg[:, None] + tn[:, None])
    u = _r(_r(_r(t[..., None] * d[:, None] + o[:, None]) - E.lo) * _r(res / _r(E.hi - E.lo)))
    c = u.clamp(0.0, res - 1.0).nan_to_num().floor().long()
    cell = (c[..., 2] * res + c[..., 1]) * res + c[..., 0]
    occ = ((bits[cell >> 5] >> (cell & 31)) & 1).bool() & hit[:, None]
    first = torch.where(occ.any(1), (occ.int().argmax(1) + 0.5) / (B * S), 1.0).double()
    share = occ.view(-1, B, S).double().mean(-1)
    before = (B * first[:, None] - torch.arange(B, device=DEV)).clamp(0.0, 1.0)
    pos = (o - 0.5 * (E.lo + E.hi)) / (E.hi - E.lo)
    return torch.cat([pos, d, first[:, None], share, before], 1), share


def _logits(flat, x, B):
    (W1, b1), (W2, b2), (W3, b3) = _layers(flat, (7 + 2 * B, 32, 32, B))
    return torch.relu(torch.relu(x @ W1.T + b1) @ W2.T + b2) @ W3.T + b3


def _exact_view(case, s):
    E, outs = _Exact(case, s), []
    if case["kind"] == "two_pass":
        colours = _exact_shade(case, s, E)
    for i, j in _chunks(case, 1 << 22):
        o, d = s["o"][i:j].double(), s["d"][i:j].double()
        q = None
        if case["kind"] == "proposed":
            B, mix = case["bins"], float(s["prop"].desc.mix)
            x, share = _features(case, s, E, o, d)
            p = torch.softmax(_logits(s["prop"].params.double(), x, B), -1)
            on = share > 0
            near = on.clone()
            near[:, 1:] |= on[:, :-1]
            near[:, :-1] |= on[:, 1:]
            cnt = near.sum(1, keepdim=True)
            r = torch.where(cnt > 0, 0.25 / B + 0.75 * near / cnt.clamp(min=1),
                            torch.full_like(p, 1.0 / B))
            q = (1 - mix) * p + mix * r
        t, hit = _distances(E, o, d, case["samples"], q)
        if case["kind"] == "two_pass":
            outs.append(_render(E, o, d, t, hit, colours=colours.view(-1, 4)[:, :3])[:3])
        else:
            outs.append(_render(E, o, d, t, hit))
    outs = tuple(torch.cat(v) for v in zip(*outs))
    return (colours,) + outs if case["kind"] == "two_pass" else outs


def _exact_shade(case, s, E):
    dims = (case["rx"], case["ry"], case["rz"])
    h = (E.hi - E.lo) / (E.R - 1)
    out = torch.zeros(dims[0] * dims[1] * dims[2], 4, dtype=torch.float64, device=DEV)
    eye = torch.tensor(s["eye"], device=DEV).double()

    def at(p):
        lin = (p[:, 2] * dims[1] + p[:, 1]) * dims[0] + p[:, 0]
        return E.record(p[:, 0], p[:, 1], p[:, 2], lin)
    step = 1 << 21
    for b in range(0, out.shape[0], step):
        lin = torch.arange(b, min(out.shape[0], b + step), device=DEV)
        p = torch.stack([lin % dims[0], lin // dims[0] % dims[1], lin // (dims[0] * dims[1])], -1)
        near = E.node_sdf(at(p)).abs() < case["band"]
        p, lin = p[near], lin[near]
        g = []
        for a in range(3):
            up, dn = p.clone(), p.clone()
            up[:, a] = (p[:, a] + 1).clamp(max=dims[a] - 1)
            dn[:, a] = (p[:, a] - 1).clamp(min=0)
            g.append((E.node_sdf(at(up)) - E.node_sdf(at(dn))) / ((up - dn)[:, a] * h[a]))
        x = p * h + E.lo
        v = torch.nn.functional.normalize(eye - x, dim=-1)
        pi, pf = E.cell(_r(x), E.psc, E.P)
        fr = at(p)
        fs = E.feat[fr.clamp(min=0)].double() * (fr >= 0)[:, None]
        out[lin, :3] = _colour(case, E.mlp, torch.stack(g, -1), v, fs,
                               E.probes[E.corners(pi, E.P)[3]].double(), _weights(pf)[0])
    return out.view(dims[2], dims[1], dims[0], 4)


def _exact_proposal(case, s):
    E, B, N = _Exact(case, s), case["bins"], case["samples"]
    flat = s["prop"].params.double().requires_grad_(True)
    grad, hists, losses = torch.zeros_like(flat), [], []
    for i, j in _chunks(case, 1 << 22):
        o, d = s["o"][i:j].double(), s["d"][i:j].double()
        t, hit = _distances(E, o, d, N, None)
        x = _r(t[..., None] * d[:, None] + o[:, None])
        ci, f = E.cell(x, E.sc, E.R)
        v = E.node_sdf(E.record(*E.corners(ci, E.R)))
        lp = _log_phi(case["tau"] * (_weights(f)[0] * v).sum(-1))
        lam = (lp[:, 1:] - lp[:, :-1]).clamp(max=0.0) * hit[:, None]
        w = torch.exp(lam.cumsum(1) - lam) * -torch.expm1(lam)
        hist = w.view(-1, B, N // B).sum(-1)
        valid = hist.sum(1) >= 1e-3
        ce = -(hist * torch.log_softmax(_logits(flat, _features(case, s, E, o, d)[0], B), -1))
        ce = ce.sum(1) * valid
        grad += torch.autograd.grad(ce.sum() / case["rays"], flat)[0]
        hists.append(hist)
        losses.append(ce.detach())
    return torch.cat(hists), grad.detach(), torch.cat(losses)


def _smooth(x):
    w = torch.exp(-0.5 * torch.arange(-2, 3, device=DEV).double() ** 2)
    w = w / w.sum()
    for a in range(3):
        n = x.shape[a]
        i = torch.arange(n, device=DEV)
        x = sum(w[j] * x.index_select(a, (i + j - 2).clamp(0, n - 1)) for j in range(5))
    return x


def _exact_terms(case, s):
    E = _Exact(case, s)
    Rx, Ry, Rz = s["scene"].dims
    h = ((E.hi - E.lo) / (E.R - 1)).tolist()
    if E.table is not None:
        z, y, x = torch.meshgrid(*(torch.arange(r, device=DEV) for r in (Rz, Ry, Rx)),
                                 indexing="ij")
        rec = E.record(x, y, z, None)
        stored = rec >= 0
        del x, y, z

        def spread(v, fill):
            return torch.where(stored, v.reshape(-1)[rec.clamp(min=0)].double(), fill)

        def collect(v):
            out = torch.zeros(E.sdf.numel(), dtype=torch.float64, device=DEV)
            out[rec[stored]] = v[stored]
            return out
    else:
        stored = torch.ones((), dtype=torch.bool, device=DEV)

        def spread(v, fill):
            return v.reshape(Rz, Ry, Rx).double()

        def collect(v):
            return v.reshape(-1)
    s_hat = spread(s["s_hat"], 1.0)
    sm = torch.where(stored, _smooth(s_hat), 1.0).float().double()
    leaf = sm.clone().requires_grad_(True)
    vox = (1 / (1 + 5 * sm.abs())) * stored
    r = leaf - s_hat
    loss = [(r * r * stored).sum()]
    obj = LAMBDAS["sdf"] * (vox * r * r).sum()
    if min(Rx, Ry, Rz) > 2:
        mid = slice(1, -1)
        g = torch.stack([(leaf[mid, mid, 2:] - leaf[mid, mid, :-2]) / (2 * h[0]),
                         (leaf[mid, 2:, mid] - leaf[mid, :-2, mid]) / (2 * h[1]),
                         (leaf[2:, mid, mid] - leaf[:-2, mid, mid]) / (2 * h[2])], -1)
        gg = g.square().sum(-1)
        nrm = g / (gg + 1e-24).sqrt()[..., None]
        e = torch.where(gg > 0, gg.clamp(min=1e-60), 1.0).sqrt() * (gg > 0) - 1
        own = stored[mid, mid, mid] if E.table is not None else stored
        vi = vox[mid, mid, mid]
        loss.append((e * e * own).sum())
        obj = obj + LAMBDAS["eik"] * (vi * e * e).sum()
        l_n = 0.0
        for a in range(3):
            k = 2 - a
            n0, n1 = nrm.narrow(k, 0, nrm.shape[k] - 1), nrm.narrow(k, 1, nrm.shape[k] - 1)
            q = (n1 - n0).square().sum(-1)
            ow = own.narrow(k, 0, nrm.shape[k] - 1) if own.dim() else own
            l_n = l_n + (q * ow).sum()
            obj = obj + LAMBDAS["normal"] * (vi.narrow(k, 0, nrm.shape[k] - 1) * q).sum()
        loss.append(l_n)
    else:
        loss += [torch.zeros_like(loss[0])] * 2
    ds = torch.autograd.grad(obj, leaf)[0] * stored
    direct = -2 * LAMBDAS["sdf"] * vox * (sm - s_hat)
    loss = [v.detach() for v in loss]
    del obj, leaf
    gg = s["gg"].view(-1)[s["words"]:].double()
    l_f = torch.zeros((), dtype=torch.float64, device=DEV)
    if case["layout"] in ("nodes", "bricks", "bf16"):
        gg = gg.view(-1, 4)
        gg[:, 0] += collect(ds)
        slot = gg[:, 0]
    else:
        nodes = Rx * Ry * Rz
        gg[:nodes] += ds.reshape(-1)
        slot = gg[:nodes]
        if case["layout"] == "planes":
            T = E.tex.double().reshape(-1, 16, 16, 3)
            gt = gg[E.off:].view(-1, 16, 16, 4)[..., :3]
            for a in (1, 2):
                df = T.narrow(a, 1, 15) - T.narrow(a, 0, 15)
                l_f = l_f + df.square().sum()
                gt.narrow(a, 1, 15).add_(2 * LAMBDAS["features"] * df)
                gt.narrow(a, 0, 15).sub_(2 * LAMBDAS["features"] * df)
    probe = torch.zeros(torch.Size([1]), device=DEV).double()
    b, gp = s["probes"].double(), s["gp"].double()
    for a in range(3):
        df = b.narrow(a, 1, b.shape[a] - 1) - b.narrow(a, 0, b.shape[a] - 1)
        probe = probe + 2 * df.square().sum()
        gp.narrow(a, 1, b.shape[a] - 1).add_(4 * LAMBDAS["probes"] * df)
        gp.narrow(a, 0, b.shape[a] - 1).sub_(4 * LAMBDAS["probes"] * df)
    z = torch.zeros(Rz, Ry, Rx, dtype=torch.float64, device=DEV, requires_grad=True)
    back = torch.autograd.grad(_smooth(z), z, spread(slot, 0.0))[0]
    d_hat = collect((back + direct) * stored)
    m = 0.9 * s["m"].double().reshape(-1) + 0.1 * d_hat
    v = 0.995 * s["v"].double().reshape(-1) + 0.005 * d_hat * d_hat
    lr = 1e-3 * math.sqrt(1 - 0.995 ** 100) / (1 - 0.9 ** 100)
    new = s["s_hat"].double().reshape(-1) - lr * m / (v.sqrt() +
                                                      1e-8 * math.sqrt(1 - 0.995 ** 100))
    shape = s["s_hat"].shape
    return {"loss": torch.stack(loss + [l_f, probe[0]]), "sdf": collect(sm), "d_grid": gg.view(-1),
            "s_hat": new.view(shape), "m": m.view(shape), "v": v.view(shape), "d_probes": gp}


def exact(case, seed):
    s = prepare(case, seed)
    kind = case["kind"]
    if kind == "step":
        return _exact_step(case, s)
    if kind in ("view", "proposed", "two_pass"):
        return _exact_view(case, s)
    if kind == "proposal":
        return _exact_proposal(case, s)
    return _exact_terms(case, s)
