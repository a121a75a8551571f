"""The work this library is asked to do, as measurable cases.

Every case goes through the public entry points: a ``ctrex.Context`` with its
geometry set (the handle a reconstruction program keeps), the differentiable
``autograd.Projector``, and the convolutions and network of ``unet``.  Inputs
come from a seed: objects are sums of random ellipsoids, measured projections
are their closed-form line integrals, trajectories are circular, perturbed or
helical cone-beam scans with a 32 mm field of view (source-object distance
200 mm, source-detector distance 400 mm, 96 mm detector).

``exact`` restates each path in plain float64 torch.
"""

from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2609_30166_gb300 import autograd, ctrex, inputs, unet

SOD, SDD, FOV, DET = 200.0, 400.0, 32.0, 96.0


def _scan(name, op, n, det, views, dtype="f32", sub=1, traj="perturbed", model="static", iters=1, span=0, zpitch=1.0):
    """n = (nx, ny, nz), det = (nu, nv).  span > 0: the listed views are that
    many of a longer scan (an ordered subset, a part of a helix)."""
    return {"name": name, "op": op, "model": model, "dtype": dtype, "nx": n[0], "ny": n[1], "nz": n[2], "nu": det[0],
            "nv": det[1], "views": views, "sub": sub, "traj": traj, "iters": iters, "span": span, "zpitch": zpitch}


def _conv(name, op, batch, d, h, w, cin, cout):
    return {"name": name, "op": op, "batch": batch, "d": d, "h": h, "w": w, "cin": cin, "cout": cout}


def listed():
    return [
        # the smallest scan: a quick-look reconstruction, where launches and host round trips count
        _scan("sirt_64", "sirt", (64, 64, 64), (96, 96), 90, traj="circular", iters=5),
        # the sparse-view scan that the learned warm start is fed with: five iterations from a rough start
        _scan("sirt_sparse_128", "sirt", (128, 128, 128), (192, 192), 60, traj="circular", iters=5),
        # the full-size reconstruction step: one SIRT iteration of a calibrated 512^3 scan
        _scan("sirt_512", "sirt", (512, 512, 512), (768, 768), 720),
        # the same step where memory is saved by 16-bit storage of volume and projections
        _scan("sirt_bf16_256", "sirt", (256, 256, 256), (384, 384), 360, dtype="bf16"),
        # a forward projection (with row sums) of a ragged volume with unequal pitch onto a ragged detector
        _scan("project_ragged", "project", (301, 243, 187), (403, 317), 90, zpitch=1.25),
        # one subset of an ordered-subset cycle: weighted backprojection of 36 of 720 views
        _scan("backproject_subset", "backproject", (512, 512, 512), (768, 768), 36, span=720),
        # a helical scan with motion blur: four sub-angles a view, 16-bit volume
        _scan("project_helical_s4", "project", (256, 256, 256), (512, 384), 72, dtype="bf16", sub=4, traj="helical",
              span=1440),
        # the classical Joseph projector in the correction step
        _scan("correct_joseph_256", "correct", (256, 256, 256), (384, 384), 360, model="joseph"),
        # event-based 4D scan: initial value, final value and transition time per voxel
        _scan("sirt_event_256", "sirt", (256, 256, 256), (384, 384), 180, model="event"),
        # self-calibration: projection through pose and deformation, gradients for volume, pose and spline
        _scan("calibrate_128", "calibrate", (128, 128, 128), (192, 192), 60, traj="circular", model="motion"),
        # one training pass of the network's widest layer
        _conv("conv_train_128", "conv_train", 2, 128, 128, 128, 16, 16),
        # the network between the rough start and the reconstruction
        _conv("network_128", "network", 1, 128, 128, 128, 16, 16),
    ]


def draw(rng):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    op = rng.choice(["sirt", "sirt", "project", "correct", "backproject", "sirt_event", "joseph", "sub", "calibrate",
                     "conv_train", "network"])
    if op == "conv_train":
        cin, cout = rng.choice([(16, 16), (32, 16), (48, 16), (16, 32), (32, 32), (96, 32), (64, 64), (192, 64),
                                (64, 128), (128, 128)])
        edge = 128 if max(cin, cout) <= 48 else (64 if max(cin, cout) <= 96 else 32)
        d, h, w = (logint(edge // 8, edge) for _ in range(3))
        return _conv("", op, rng.randint(1, 2), d, h, w, cin, cout)
    if op == "network":
        d, h, w = (8 * rng.randint(4, 16) for _ in range(3))
        return _conv("", op, rng.randint(1, 2), d, h, w, 16, 16)
    # a scan: volume edges around one size, detector about 1.5 x as wide, odd sizes as they come
    small = op in ("calibrate",)
    n = logint(32, 128) if small else logint(48, 400)
    dims = tuple(max(16, int(n * rng.uniform(0.7, 1.0))) for _ in range(3))
    det = tuple(max(24, int(1.5 * n * rng.uniform(0.75, 1.1))) for _ in range(2))
    views = logint(16, 60) if small else logint(24, 360)
    kw = {"traj": rng.choice(["circular", "perturbed"]), "zpitch": rng.choice([1.0, 1.0, 1.25])}
    model, dtype = "static", rng.choice(["f32", "f32", "bf16"])
    if op == "sirt":
        kw["iters"] = rng.randint(1, 3) if n <= 160 else 1
    elif op == "sirt_event":
        op, model, dtype = "sirt", "event", "f32"
    elif op == "joseph":
        op, model, dtype = rng.choice(["project", "correct"]), "joseph", "f32"
    elif op == "sub":
        op, kw["sub"], kw["traj"] = rng.choice(["project", "backproject"]), rng.randint(2, 4), "helical"
        kw["span"] = 4 * views
    elif op == "calibrate":
        model, dtype, kw["zpitch"] = "motion", "f32", 1.0
        dims, det = (n,) * 3, (det[0],) * 2
    elif rng.random() < 0.5:
        kw["span"] = views * rng.randint(2, 10)
    return _scan("", op, dims, det, views, dtype=dtype, model=model, **kw)


# -- inputs ------------------------------------------------------------------------------------------------------

def _grid(c):
    """Pitch and origin per axis (x, y, z), mm: the field of view holds the longest edge."""
    p = FOV / max(c["nx"], c["ny"], c["nz"] * c["zpitch"])
    vox = (p, p, p * c["zpitch"])
    org = tuple(-0.5 * (n - 1) * v for n, v in zip((c["nx"], c["ny"], c["nz"]), vox))
    return vox, org


def _matrices(c, seed):
    """P [views, sub, 3, 4]: world mm to homogeneous pixels."""
    rng = np.random.default_rng([seed, 1])
    total = c["span"] or c["views"]
    turns = 2.0 if c["traj"] == "helical" else 1.0
    da = 2.0 * math.pi * turns / total
    S, pitch = c["sub"], DET / c["nu"]
    first = rng.integers(0, total)  # a subset is every (total / views)-th view, a part of a helix its middle
    out = np.zeros((c["views"], S, 3, 4))
    for v in range(c["views"]):
        if c["traj"] == "helical":
            g = (total - c["views"]) // 2 + v
        else:
            g = (first + v * total // c["views"]) % total
        du, dv = rng.uniform(-2, 2, 2)
        tilt, jit = math.radians(rng.uniform(-0.5, 0.5)), rng.uniform(-0.2, 0.2, 3)
        for s in range(S):
            a = g * da + (s + 0.5 - 0.5 * S) * da / S
            z = 36.0 * (a / (math.pi * turns) - 1.0) if c["traj"] == "helical" else 0.0
            ca, sa = math.cos(a), math.sin(a)
            src, ctr = np.array([-SOD * ca, -SOD * sa, z]), np.array([(SDD - SOD) * ca, (SDD - SOD) * sa, z])
            u, w = pitch * np.array([-sa, ca, 0.0]), np.array([0.0, 0.0, pitch])
            if c["traj"] == "perturbed":
                ctr, src = ctr + du * u + dv * w, src + jit
                u, w = math.cos(tilt) * u + math.sin(tilt) * w, math.cos(tilt) * w - math.sin(tilt) * u
            d0 = ctr - 0.5 * (c["nu"] - 1) * u - 0.5 * (c["nv"] - 1) * w
            Mi = np.linalg.inv(np.stack([u, w, d0 - src], axis=1))
            out[v, s] = np.concatenate([Mi, -(Mi @ src)[:, None]], axis=1)
    return out


def _objects(c, seed):
    """Random ellipsoids: centre, semi-axes (mm), density."""
    rng = np.random.default_rng([seed, 2])
    vox, _ = _grid(c)
    half = np.array([0.5 * n * v for n, v in zip((c["nx"], c["ny"], c["nz"]), vox)])
    obj = []
    for _ in range(10):
        semi = half * rng.uniform(0.1, 0.55, 3)
        obj.append((rng.uniform(-1, 1, 3) * (half - semi), semi, rng.uniform(0.1, 1.0)))
    return obj


def _phantom(c, seed):
    vox, org = _grid(c)
    ax = [torch.arange(n, device="cuda", dtype=torch.float32) * v + o
          for n, v, o in zip((c["nx"], c["ny"], c["nz"]), vox, org)]
    vol = torch.zeros(c["nz"], c["ny"], c["nx"], device="cuda")
    for m, semi, dens in _objects(c, seed):
        q = [((x - float(m[i])) / float(semi[i])) ** 2 for i, x in enumerate(ax)]
        r2 = q[2][:, None, None] + (q[1][:, None] + q[0][None, :])[None]
        vol += dens * (r2 <= 1.0)
    return vol


def _lines(P, c):
    """Source (mm) and unit directions [nv, nu, 3] of one 3x4 matrix, float64."""
    M, p4 = P[:, :3], P[:, 3]
    s = 1.0 if P[2, 3] > 0 else -1.0  # the volume centre (the origin) has positive depth
    Mi = np.linalg.inv(s * M)
    src = torch.as_tensor(-(Mi @ (s * p4)), device="cuda")
    Mi = torch.as_tensor(Mi, device="cuda")
    u = torch.arange(c["nu"], device="cuda", dtype=torch.float64)
    v = torch.arange(c["nv"], device="cuda", dtype=torch.float64)
    d = Mi[:, 2] + v[:, None, None] * Mi[:, 1] + u[None, :, None] * Mi[:, 0]
    return src, d / d.norm(dim=-1, keepdim=True)


def _measured(c, seed, P):
    """Closed-form line integrals of the objects (mean over sub-angles), float32 [views, nv, nu]."""
    p = torch.zeros(c["views"], c["nv"], c["nu"], device="cuda")
    obj = _objects(c, seed)
    m = torch.as_tensor(np.stack([o[0] for o in obj]), device="cuda", dtype=torch.float32)
    si = torch.as_tensor(np.stack([1.0 / o[1] for o in obj]), device="cuda", dtype=torch.float32)
    for v in range(c["views"]):
        for s in range(c["sub"]):
            src, d = _lines(P[v, s], c)
            src, d = src.float(), d.float()
            for i, o in enumerate(obj):
                e, f = d * si[i], (src - m[i]) * si[i]
                a, b = (e * e).sum(-1), (e * f).sum(-1)
                # chord 2 sqrt(1 - q^2) / sqrt(a), q the distance of the line from the centre in the unit sphere
                w = f - (b / a)[..., None] * e
                q2 = (w * w).sum(-1)
                p[v] += (2.0 * o[2] / c["sub"]) * torch.sqrt((1.0 - q2).clamp(min=0.0) / a)
    return p


def _gen(seed, k):
    return torch.Generator(device="cuda").manual_seed(seed * 16 + k)


def _motion(c, seed):
    """Pose [views, 15] (rotation, translation, affine), spline [8, 8, 8, 3] (mm) and time scale of each view."""
    rng = np.random.default_rng([seed, 3])
    V = c["views"]
    th = np.zeros((V, 15))
    th[:, :3] = np.radians(rng.uniform(-1, 1, (V, 3)))
    th[:, 3:6] = rng.uniform(-0.5, 0.5, (V, 3))
    th[:, 6:] = np.eye(3).reshape(9) + rng.uniform(-0.01, 0.01, (V, 9))
    co = rng.uniform(-1, 1, (8, 8, 8, 3)) * 2.0 * _grid(c)[0][0]
    t = [torch.as_tensor(a, dtype=torch.float32, device="cuda").contiguous() for a in (th, co, np.arange(V) / (V - 1))]
    return t


MARGIN = 0.5  # mm by which a moving object may leave the box


def _fields(c, seed):
    """Event scene: initial and final values [2, nz, ny, nx], transition times, acquisition times."""
    mu0 = _phantom(c, seed)
    mu1 = mu0 + 0.5 * _phantom(c, seed + 7919)
    z = torch.arange(c["nz"], device="cuda", dtype=torch.float32)[:, None, None] / c["nz"]
    x = torch.arange(c["nx"], device="cuda", dtype=torch.float32)[None, None, :] / c["nx"]
    tau = torch.where(mu1 != mu0, 0.15 + 0.4 * z + 0.3 * x, torch.full_like(mu0, 2.0)).contiguous()
    tv = torch.arange(c["views"], device="cuda", dtype=torch.float32) / (c["views"] - 1)
    return torch.stack([mu0, mu1]), tau, tv


def _conv_inputs(c, seed):
    g = _gen(seed, 0)
    shape = (c["batch"], c["d"], c["h"], c["w"])
    x = torch.randn(shape + (c["cin"],), generator=g, device="cuda").relu().to(torch.bfloat16)  # as after a ReLU
    w = torch.randn(c["cout"], 27, c["cin"], generator=g, device="cuda") * math.sqrt(2.0 / (27 * c["cin"]))
    b = 0.1 * torch.randn(c["cout"], generator=g, device="cuda")
    dy = torch.randn(shape + (c["cout"],), generator=g, device="cuda").to(torch.bfloat16)
    return x, w, b, dy


def _network(seed):
    m = unet.UNet3D(seed=seed % 1000)
    g = torch.Generator().manual_seed(seed)
    with torch.no_grad():  # a head as after training: the fresh one is zero
        m.head_w.copy_(0.1 * torch.randn(m.head_w.shape, generator=g))
    return m.cuda()


def _dtype(c):
    return torch.bfloat16 if c["dtype"] == "bf16" else torch.float32


def _scan_inputs(c, seed):
    """Everything random of a scan: matrices and the tensors of its operation."""
    P, t, dt = _matrices(c, seed), {}, _dtype(c)
    if c["op"] == "backproject":
        t["r"] = torch.randn(c["views"], c["nv"], c["nu"], generator=_gen(seed, 1), device="cuda").to(dt)
        # correction images are smooth against a pixel: a 5 x 5 mean of noise
        t["r"] = F.avg_pool2d(t["r"].float(), 5, 1, 2).to(dt).contiguous()
        t["x0"] = _phantom(c, seed).to(dt)
        t["w"] = torch.rand(c["nz"], c["ny"], c["nx"], generator=_gen(seed, 2), device="cuda") * 0.5 + 0.5
        return P, t
    if c["model"] == "event":
        fields, t["tau"], t["tv"] = _fields(c, seed)
        t["x0"] = (0.8 * fields).to(dt).contiguous()
    else:
        t["x0"] = (0.8 * _phantom(c, seed)).to(dt)
    if c["op"] in ("sirt", "correct"):
        t["p"] = _measured(c, seed, P).to(dt)
    if c["op"] == "calibrate":
        t["theta"], t["coef"], t["sv"] = _motion(c, seed)
        t["g"] = torch.rand(c["views"], c["nv"], c["nu"], generator=_gen(seed, 3), device="cuda") + 0.5
    return P, t


def prepare(case, seed):
    c, st = case, {"case": case}
    if c["op"] == "conv_train":
        x, w, b, dy = _conv_inputs(c, seed)
        st["layer"] = unet.Conv3(c["cin"], c["cout"]).cuda()
        with torch.no_grad():
            st["layer"].w.copy_(w)
            st["layer"].b.copy_(b)
        st["x"], st["dy"] = x.requires_grad_(True), dy
        return st
    if c["op"] == "network":
        st["net"] = _network(seed)
        st["x"] = torch.rand(c["batch"], c["d"], c["h"], c["w"], generator=_gen(seed, 0), device="cuda")
        return st
    P, t = _scan_inputs(c, seed)
    vox, org = _grid(c)
    if c["op"] == "calibrate":
        cfg = inputs.Config("calibrate", n=c["nx"], nu=c["nu"], nv=c["nv"], n_views=c["views"], motion=True,
                            margin=MARGIN)
        st["projector"] = autograd.Projector(cfg, P=P, s_view=t["sv"])
        st.update({k: t[k].requires_grad_(True) for k in ("x0", "theta", "coef")}, g=t["g"])
        return st
    ctx = ctrex.Context()
    ctx.set_geometry(P, (c["nz"], c["ny"], c["nx"]), vox, org, (c["nu"], c["nv"]))
    if c["model"] == "event":
        ctx.set_dyrect(t["tau"], t["tv"])
    elif c["model"] == "joseph":
        ctx.set_projector("joseph")
    st.update(t, ctx=ctx)
    return st


def run(st):
    c = st["case"]
    if c["op"] == "conv_train":
        y = st["layer"](st["x"])
        dx, dw, db = torch.autograd.grad(y, [st["x"], st["layer"].w, st["layer"].b], st["dy"])
        return {"y": y.detach(), "dx": dx, "dw": dw, "db": db}
    if c["op"] == "network":
        with torch.no_grad():
            return {"x": st["net"](st["x"])}
    if c["op"] == "calibrate":
        proj = st["projector"](st["x0"], st["theta"], st["coef"])
        gx, gt, gc = torch.autograd.grad(proj, [st["x0"], st["theta"], st["coef"]], st["g"])
        return {"proj": proj.detach(), "gx": gx, "gtheta": gt, "gcoef": gc}
    ctx = st["ctx"]
    if c["op"] == "project":
        rowsum = torch.empty((c["views"], c["nv"], c["nu"]), device="cuda")
        return {"proj": ctx.fwd_project(st["x0"], rowsum=rowsum), "rowsum": rowsum}
    if c["op"] == "correct":
        r, sums = ctx.fwd_correct(st["x0"], st["p"])
        return {"r": r, "sums": sums}
    if c["op"] == "backproject":
        return {"x": ctx.back_project(st["r"], vol=st["x0"].clone(), w=st["w"], alpha=0.9)}
    x, hist, _ = ctx.sirt_iterate(st["x0"].clone(), st["p"], c["iters"])
    return {"x": x, "residual": hist}


# -- what a pass cannot do without -------------------------------------------------------------------------------

def work(case):
    c = case
    if c["op"] == "conv_train":
        vox = c["batch"] * c["d"] * c["h"] * c["w"]
        # x and dy read, y and dx written (16 bit); filter and its gradient (32 bit); three convolutions
        byts = 2 * vox * (2 * c["cin"] + 2 * c["cout"]) + 2 * 4 * 27 * c["cin"] * c["cout"]
        return {"bytes": byts, "flops": 3 * 2 * vox * 27 * c["cin"] * c["cout"]}
    if c["op"] == "network":
        vox = c["batch"] * c["d"] * c["h"] * c["w"]
        layers = [(0, 16, 16), (0, 16, 16), (1, 16, 32), (1, 32, 32), (2, 32, 64), (2, 64, 64), (3, 64, 128),
                  (3, 128, 128), (2, 192, 64), (2, 64, 64), (1, 96, 32), (1, 32, 32), (0, 48, 16), (0, 16, 16)]
        return {"bytes": 8 * vox + sum(4 * 27 * a * b for _, a, b in layers),
                "flops": sum(2 * (vox >> (3 * lv)) * 27 * a * b for lv, a, b in layers)}
    vox, _ = _grid(c)
    n = (c["nx"], c["ny"], c["nz"])
    nvox, pix = n[0] * n[1] * n[2], c["views"] * c["nv"] * c["nu"]
    b = 2 if c["dtype"] == "bf16" else 4
    fields = 2 if c["model"] == "event" else 1
    # samples: the box's volume over (pixel area at the object x step), twice as many slices as voxels along a ray
    area = (DET / c["nu"] * SOD / SDD) ** 2
    box = n[0] * vox[0] * n[1] * vox[1] * n[2] * vox[2]
    if c["traj"] == "helical":
        box *= min(1.0, 0.5 * c["nv"] * DET / c["nu"] / (n[2] * vox[2]))
    step = 0.5 * min(vox)
    if c["model"] == "joseph":
        step = 1.11 * vox[0]  # one crossing a slice of the principal axis
    samples = c["views"] * c["sub"] * box / (area * step)
    updates = float(nvox) * c["views"] * c["sub"]
    tap = 16 if c["model"] != "joseph" else 8  # multiply-adds of the taps
    if c["op"] == "project":
        return {"bytes": b * nvox + b * pix + 4 * pix, "flops": tap * samples}
    if c["op"] == "correct":
        return {"bytes": b * nvox + 2 * b * pix, "flops": tap * samples}
    if c["op"] == "backproject":
        return {"bytes": 2 * b * nvox + 4 * nvox + b * pix, "flops": 8 * updates}
    if c["op"] == "calibrate":
        # volume and detector weights read, projections and gradient written; spline value, its derivatives, taps
        return {"bytes": 2 * 4 * nvox + 2 * 4 * pix, "flops": samples * (3 * 252 * 2 + 2 * 576 + 3 * 16)}
    k = c["iters"]
    return {"bytes": k * (fields * 2 * b * nvox + 2 * b * pix) + (4 * nvox if fields == 2 else 0),
            "flops": k * (tap * samples + 8 * updates)}


# -- the same in 64 bits -----------------------------------------------------------------------------------------

def _axis_weight(g, n):
    """Summed weight of the taps inside [0, n - 1] at index coordinate g."""
    return torch.minimum(torch.minimum(g + 1.0, n - g), torch.ones_like(g)).clamp(min=0.0)


def _trilinear(vol, g):
    """vol [nz, ny, nx] at index coordinates g [..., 3] (x, y, z); zero outside."""
    n = torch.tensor([vol.shape[2], vol.shape[1], vol.shape[0]], device=g.device, dtype=g.dtype)
    q = 2.0 * g / (n - 1.0) - 1.0
    return F.grid_sample(vol[None, None], q.reshape(1, 1, 1, -1, 3), align_corners=True).reshape(g.shape[:-1])


def _clip(src, d, lo, hi):
    t0 = torch.zeros(d.shape[:-1], device="cuda", dtype=torch.float64)
    t1 = torch.full_like(t0, math.inf)
    for a in range(3):
        ta, tb = (lo[a] - src[a]) / d[..., a], (hi[a] - src[a]) / d[..., a]
        t0, t1 = torch.maximum(t0, torch.minimum(ta, tb)), torch.minimum(t1, torch.maximum(ta, tb))
    return t0, t1


def _march(c, P, chunk=1 << 23):
    """Samples of one view's sub-angle: yields (ray indices, index coordinates [k, rays, 3], weights [k, rays])."""
    vox, org = (torch.tensor(a, device="cuda", dtype=torch.float64) for a in _grid(c))
    n = torch.tensor([c["nx"], c["ny"], c["nz"]], device="cuda", dtype=torch.float64)
    m = MARGIN if c["model"] == "motion" else 0.0
    src, d = _lines(P, c)
    d = d.reshape(-1, 3)
    t0, t1 = _clip(src, d, org - 0.5 * vox - m, org + (n - 0.5) * vox + m)
    live = (t1 > t0).nonzero()[:, 0]
    if not len(live):
        return
    d, t0, t1 = d[live], t0[live], t1[live]
    step = 0.5 * float(vox.min())
    K = int(torch.ceil((t1 - t0).max() / step))
    per = max(1, chunk // len(live))
    for k0 in range(0, K, per):
        k = torch.arange(k0, min(K, k0 + per), device="cuda", dtype=torch.float64)[:, None]
        a = t0 + k * step
        b = torch.minimum(a + step, t1)
        w = (b - a).clamp(min=0.0)
        x = src + (0.5 * (a + b))[..., None] * d
        g = (x - org) / vox
        yield live, g, w


def _forward64(c, P, vol):
    """Projections and row sums, [views, nv, nu] float64.  vol: a volume, or a function of the view."""
    proj = torch.zeros(c["views"], c["nv"] * c["nu"], device="cuda", dtype=torch.float64)
    rows = torch.zeros_like(proj)
    n = (c["nx"], c["ny"], c["nz"])
    for v in range(c["views"]):
        x = vol(v) if callable(vol) else vol
        for s in range(c["sub"]):
            for live, g, w in (_joseph(c, P[v, s]) if c["model"] == "joseph" else _march(c, P[v, s])):
                proj[v, live] += (w * _trilinear(x, g)).sum(0) / c["sub"]
                inr = _axis_weight(g[..., 0], n[0]) * _axis_weight(g[..., 1], n[1]) * _axis_weight(g[..., 2], n[2])
                rows[v, live] += (w * inr).sum(0) / c["sub"]
    shape = (c["views"], c["nv"], c["nu"])
    return proj.view(shape), rows.view(shape)


def _joseph(c, P, chunk=1 << 23):
    """Slice crossings of each ray's principal axis, as _march yields samples."""
    vox, org = (torch.tensor(a, device="cuda", dtype=torch.float64) for a in _grid(c))
    n = (c["nx"], c["ny"], c["nz"])
    src, d = _lines(P, c)
    dg = d.reshape(-1, 3) / vox
    gs = (src - org) / vox
    axis = dg.abs().argmax(1)
    for m in range(3):
        live = (axis == m).nonzero()[:, 0]
        if not len(live):
            continue
        e = dg[live]
        per = max(1, chunk // len(live))
        for k0 in range(0, n[m], per):
            k = torch.arange(k0, min(n[m], k0 + per), device="cuda", dtype=torch.float64)[:, None]
            t = (k - gs[m]) / e[:, m]
            g = gs + t[..., None] * e
            g[..., m] = k
            yield live, g, (1.0 / e[:, m].abs()) * (t >= 0)


def _back64(c, P, r, take=None):
    """Backprojection sums b and c [nz, ny, nx] of images r (float64) over the views in take."""
    vox, org = _grid(c)
    ax = [torch.arange(n, device="cuda", dtype=torch.float64) * v + o
          for n, v, o in zip((c["nx"], c["ny"], c["nz"]), vox, org)]
    b = torch.zeros(c["nz"], c["ny"], c["nx"], device="cuda", dtype=torch.float64)
    cs = torch.zeros_like(b)
    size = torch.tensor([c["nu"] - 1.0, c["nv"] - 1.0], device="cuda", dtype=torch.float64)
    slab = max(1, (1 << 24) // (c["nx"] * c["ny"]))
    for v in range(c["views"]):
        for s in range(c["sub"]):
            p = P[v, s] * (1.0 if P[v, s][2, 3] > 0 else -1.0)
            for z0 in range(0, c["nz"], slab):
                z = ax[2][z0:z0 + slab]
                h = [p[i, 0] * ax[0] + (p[i, 1] * ax[1])[:, None] + (p[i, 2] * z + p[i, 3])[:, None, None]
                     for i in range(3)]
                q = torch.stack([h[0] / h[2], h[1] / h[2]], dim=-1)
                inr = _axis_weight(q[..., 0], c["nu"]) * _axis_weight(q[..., 1], c["nv"]) * (h[2] > 0)
                val = F.grid_sample(r[v][None, None], (2.0 * q / size - 1.0).view(1, 1, -1, 2), align_corners=True)
                on = 1.0 if take is None else take(v)[z0:z0 + slab]
                b[z0:z0 + slab] += on * (val.view(inr.shape) * (h[2] > 0)) / c["sub"]
                cs[z0:z0 + slab] += on * inr / c["sub"]
    return b, cs


def _warp64(x, th, coef, sv):
    """World points x [N, 3] through one view's pose and deformation."""
    W = x.new_zeros(3, 3)
    W[0, 1], W[0, 2], W[1, 0], W[1, 2], W[2, 0], W[2, 1] = -th[2], th[1], th[2], -th[0], -th[1], th[0]
    R = torch.linalg.matrix_exp(W)
    xp = (x @ R.T + th[3:6]) @ th[6:].view(3, 3).T
    xi = ((xp + 0.5 * FOV) * (5.0 / FOV) + 1.0).clamp(1.0, 6.0)
    w = []
    for a in range(3):  # cubic B-spline weights over the eight control points
        t = (xi[:, a, None] - torch.arange(8, device=x.device, dtype=x.dtype)).abs()
        w.append(torch.where(t < 1, 2 / 3 - t ** 2 + 0.5 * t ** 3, (2 - t).clamp(min=0.0) ** 3 / 6))
    zy = (w[2][:, :, None] * w[1][:, None, :]).reshape(-1, 64)
    u = (zy @ coef.reshape(64, 24)).view(-1, 8, 3)
    return xp + sv * (u * w[0][:, :, None]).sum(1)


def _calibrate64(c, P, t):
    vox, org = _grid(c)
    x, th, co = (t[k].detach().double().requires_grad_(True) for k in ("x0", "theta", "coef"))
    g = t["g"].double().view(c["views"], -1)
    proj = torch.zeros_like(g)
    vx, og = vox[0], org[0]
    for v in range(c["views"]):
        for live, gi, w in _march(c, P[v, 0], chunk=1 << 21):
            y = _warp64(gi.reshape(-1, 3) * vx + og, th[v], co, float(t["sv"][v]))
            val = w * _trilinear(x, ((y - og) / vx).view(gi.shape))
            proj[v, live] += val.detach().sum(0)
            (val.sum(0) * g[v, live]).sum().backward()
    return {"proj": proj.view(c["views"], c["nv"], c["nu"]), "gx": x.grad, "gtheta": th.grad, "gcoef": co.grad}


def _conv64(x, w):
    """3x3x3 'same' convolution, channels last: a sum of shifted matrix products."""
    p = F.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    d, h, ww = x.shape[1:4]
    y = 0
    for k in range(27):
        a, b, e = k // 9, k // 3 % 3, k % 3
        y = y + p[:, a:a + d, b:b + h, e:e + ww] @ w[:, k].T
    return y


def _conv_train64(c, seed):
    x, w, b, dy = _conv_inputs(c, seed)
    x, w, dy = x.double(), w.to(torch.bfloat16).double(), dy.double()
    y = (_conv64(x, w) + b.double()).relu()
    dy = dy * (y > 0)
    dx = _conv64(dy, w.flip(1).transpose(0, 2))
    p = F.pad(x, (0, 0, 1, 1, 1, 1, 1, 1))
    d, h, ww = x.shape[1:4]
    f = dy.reshape(-1, c["cout"])
    dw = torch.stack([f.T @ p[:, k // 9:k // 9 + d, k // 3 % 3:k // 3 % 3 + h, k % 3:k % 3 + ww]
                      .reshape(-1, c["cin"]) for k in range(27)], dim=1)
    return {"y": y, "dx": dx, "dw": dw, "db": f.sum(0)}


def _network64(c, seed):
    m = _network(seed).double()
    x = torch.rand(c["batch"], c["d"], c["h"], c["w"], generator=_gen(seed, 0), device="cuda").double()

    def block(layers, v):
        for layer in layers:
            v = (_conv64(v, layer.w.detach()) + layer.b.detach()).relu()
        return v

    def pool(v):
        return F.max_pool3d(v.permute(0, 4, 1, 2, 3), 2).permute(0, 2, 3, 4, 1)

    def up(v, skip):
        return torch.cat([F.interpolate(v.permute(0, 4, 1, 2, 3), scale_factor=2).permute(0, 2, 3, 4, 1), skip], -1)

    s1 = block(m.e1, F.pad(x[..., None], (0, 15)))
    s2 = block(m.e2, pool(s1))
    s3 = block(m.e3, pool(s2))
    u3 = block(m.d3, up(block(m.e4, pool(s3)), s3))
    u1 = block(m.d1, up(block(m.d2, up(u3, s2)), s1))
    return {"x": x + (u1 * m.head_w.detach()).sum(-1) + m.head_b.detach()}


def exact(case, seed):
    c = case
    if c["op"] == "conv_train":
        return _conv_train64(c, seed)
    if c["op"] == "network":
        return _network64(c, seed)
    w = work(c)
    if w["flops"] > (6e11 if c["op"] != "calibrate" else 3e12):
        return None  # minutes in 64 bits
    P, t = _scan_inputs(c, seed)
    if c["op"] == "calibrate":
        return _calibrate64(c, P, t)
    x0 = t["x0"].double()
    if c["op"] == "backproject":
        b, cs = _back64(c, P, t["r"].double())
        return {"x": x0 + 0.9 * t["w"].double() * torch.where(cs > 1e-6, b / cs, 0.0 * b)}
    event = c["model"] == "event"

    def at(x):  # what a view sees
        return (lambda v: torch.where(t["tv"][v] < t["tau"], x[0], x[1])) if event else x

    if c["op"] == "project":
        proj, rows = _forward64(c, P, x0)
        return {"proj": proj, "rowsum": rows}
    p = t["p"].double()
    eps = 1e-6 * min(_grid(c)[0])

    def correct(x):
        q, rows = _forward64(c, P, at(x))
        e = p - q
        r = torch.where(rows > eps, e / rows.clamp(min=eps), 0.0 * e)
        return r, torch.stack([(e * e).sum(), (p * p).sum()])

    if c["op"] == "correct":
        r, sums = correct(x0)
        return {"r": r, "sums": sums}
    x, hist = x0, []
    for _ in range(c["iters"]):
        r, sums = correct(x)
        hist.append(math.sqrt(float(sums[0] / sums[1])))
        if event:
            parts = []
            for k in range(2):
                b, cs = _back64(c, P, r, lambda v, k=k: ((t["tv"][v] < t["tau"]) == (k == 0)).double())
                parts.append(torch.where(cs > 1e-6, b / cs, 0.0 * b))
            x = x + torch.stack(parts)
        else:
            b, cs = _back64(c, P, r)
            x = x + torch.where(cs > 1e-6, b / cs, 0.0 * b)
    return {"x": x, "residual": np.array(hist)}
