"""The work that is timed: what users of the library have it do, through its
public entry points, over the sizes they have it do it at.

A case is a dict of plain values; its "kind" names the call:

  request     a new target end to end, as a serving request brings it: surfel
              radii, the eight aggregation views, their fusion, the sweep
  sweep       a monostatic RCS sweep of a target whose geometry is resident
  geometry    GFBs of the aggregation views and their fusion into splats
  attributes  surfel radii and PCA normals of a point cloud
  gfb         incidence screens of a point cloud, surfels or ray tubes
  trace       the bounces of a batch of screens, every ray's record returned
  field       the physical-optics sum of traced records over a band
  forward     the completion network on a batch of coarse depth maps
  gradient    its training step up to the gradients of every parameter
  layers      the layers of one of its blocks, forward and backward

Targets are the shapes of the repository's workloads (dihedral, sphere, OctAR
plates, the noisy composite), sampled on the GPU from the seed alone.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2408_15583_gb300 import api, learned, learned_train, pipeline

C0 = 299_792_458.0
DEV = "cuda:0"
WIDTHS, BLOCKS = (32, 64, 128, 256), (2, 2, 2, 2)
HEADS = (("depth", 1), ("normal", 3), ("mask", 1))


def listed():
    return [
        # a small target served once: 10k points, 128^2 rays, an azimuth cut;
        # every launch of the path counts
        dict(name="request dihedral", kind="request", target="dihedral", n=10_000, view=512,
             W=128, angles=91, freqs=1, bounces=2),
        # the band sweep of a smooth target (two batches of angles)
        dict(name="sweep sphere", kind="sweep", target="sphere", n=200_000, view=512, W=1024,
             angles=128, freqs=64, bounces=2),
        # the large scene: a million noisy points, five bounces, one frequency
        dict(name="sweep composite", kind="sweep", target="composite", n=1_000_000, view=512,
             W=2048, angles=24, freqs=1, bounces=5),
        # the geometry a new target needs before its first sweep
        dict(name="geometry sphere", kind="geometry", target="sphere", n=200_000, view=512,
             edge=0),
        # radii and normals of a million-point scan that brings neither
        dict(name="attributes composite", kind="attributes", target="composite", n=1_000_000,
             k_r=8, k_n=16, normal=True),
        # the smallest call: one screen of a small target
        dict(name="gfb dihedral", kind="gfb", target="dihedral", n=10_000, W=128, views=1,
             tube=False),
        # multi-bounce records of the OctAR plates (eight of its angles)
        dict(name="trace octar", kind="trace", target="octar", n=50_000, view=512, W=480, views=8,
             bounces=3),
        # the field of written records over an uneven frequency list
        dict(name="field sphere", kind="field", target="sphere", n=100_000, view=256, W=509,
             views=4, freqs=33, uniform=False),
        # inference on one target's sixteen views
        dict(name="forward 16x256", kind="forward", batch=16, H=256, W=256),
        # a training batch
        dict(name="gradient 32x256", kind="gradient", batch=32, H=256, W=256),
        # the layers of a block at the second level of a training batch
        dict(name="layers 64ch", kind="layers", batch=32, H=128, W=128, C=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["request", "sweep", "geometry", "attributes", "gfb", "trace", "field",
                       "forward", "gradient", "layers"])
    target = rng.choice(["dihedral", "sphere", "octar", "composite"])
    view = rng.choice([128, 256, 384, 512])
    if kind == "request":
        return dict(kind=kind, target=target, n=_log(rng, 10_000, 300_000), view=view,
                    W=_log(rng, 64, 400), angles=_log(rng, 1, 91), freqs=_log(rng, 1, 16),
                    bounces=rng.randint(1, 5))
    if kind == "sweep":
        W = _log(rng, 128, 1500)
        rays = (1 << 26) // (W * W)              # at most half the listed sweep's rays
        return dict(kind=kind, target=target, n=_log(rng, 10_000, 500_000), view=view, W=W,
                    angles=_log(rng, 1, max(1, min(180, rays))), freqs=_log(rng, 1, 64),
                    bounces=rng.randint(1, 4))
    if kind == "geometry":
        return dict(kind=kind, target=target, n=_log(rng, 10_000, 1_000_000), view=_log(rng, 96, 512),
                    edge=rng.choice([0, 0, 0, 1]))
    if kind == "attributes":
        return dict(kind=kind, target=target, n=_log(rng, 1_000, 1_000_000), k_r=8,
                    k_n=rng.choice([12, 16, 24]), normal=rng.random() < 0.6)
    if kind == "gfb":
        return dict(kind=kind, target=target, n=_log(rng, 2_000, 1_000_000), W=_log(rng, 64, 1024),
                    views=_log(rng, 1, 16), tube=rng.random() < 0.4)
    if kind == "trace":
        return dict(kind=kind, target=target, n=_log(rng, 10_000, 200_000), view=view,
                    W=_log(rng, 64, 600), views=_log(rng, 1, 8), bounces=rng.randint(1, 5))
    if kind == "field":
        return dict(kind=kind, target=target, n=_log(rng, 10_000, 100_000), view=256,
                    W=_log(rng, 64, 600), views=_log(rng, 1, 6), freqs=_log(rng, 1, 64),
                    uniform=rng.random() < 0.6)
    H, W = 8 * _log(rng, 4, 32), 8 * _log(rng, 4, 32)
    most = max(1, (1 << 20) // (H * W))
    if kind == "forward":
        return dict(kind=kind, batch=_log(rng, 1, most), H=H, W=W)
    if kind == "gradient":
        return dict(kind=kind, batch=_log(rng, 1, 2 * most), H=H, W=W)
    C = rng.choice([32, 64, 128, 256])
    return dict(kind=kind, batch=_log(rng, 1, max(1, min(64, (1 << 25) // (C * H * W)))), H=H, W=W,
                C=C)


# ---- inputs -----------------------------------------------------------------

def _points(target, n, seed):
    """(pos, exact nrm) float32 [n, 3] of the target, uniform samples."""
    g = torch.Generator(device=DEV).manual_seed(seed)
    rnd = lambda *s: torch.rand(*s, generator=g, device=DEV, dtype=torch.float64)

    def face(axis, m, size, lo):
        p = torch.zeros(m, 3, device=DEV, dtype=torch.float64)
        o = [k for k in range(3) if k != axis]
        p[:, o] = rnd(m, 2) * size + lo
        q = torch.zeros_like(p)
        q[:, axis] = 1.0
        return p, q

    if target == "dihedral":
        parts = [face(1, n - n // 2, 0.5, 0.0), face(0, n // 2, 0.5, 0.0)]
    elif target == "octar":
        parts = [face(a, n // 3 + (n % 3 if a == 0 else 0), 20.0, -10.0) for a in range(3)]
    elif target == "sphere":                    # golden-angle lattice, turned by the seed
        i = torch.arange(n, device=DEV, dtype=torch.float64)
        z = 1.0 - (2.0 * i + 1.0) / n
        r = torch.sqrt(1.0 - z * z)
        t = i * (math.pi * (3.0 - math.sqrt(5.0)))
        p = torch.stack([r * torch.cos(t), r * torch.sin(t), z], 1)
        q, _ = torch.linalg.qr(torch.randn(3, 3, generator=g, device=DEV, dtype=torch.float64).cpu())
        p = p @ q.to(DEV)
        return p.float().contiguous(), p.float().contiguous()
    else:                                       # trihedral, plate and cylinder, by area
        a_tri, a_pl, a_cy = 1.08, 1.0, 2 * math.pi * 0.3
        n_tri = int(n * a_tri / (a_tri + a_pl + a_cy)) // 3
        n_pl = int(n * a_pl / (a_tri + a_pl + a_cy))
        n_cy = n - 3 * n_tri - n_pl
        parts = [face(a, n_tri, 0.6, 0.0) for a in range(3)]
        p, q = face(0, n_pl, 1.0, -0.5)
        parts.append((p + torch.tensor([-1.5, 0.0, 0.0], device=DEV, dtype=torch.float64), q))
        ph = rnd(n_cy) * (2 * math.pi)
        q = torch.stack([torch.cos(ph), torch.sin(ph), torch.zeros_like(ph)], 1)
        parts.append((torch.stack([0.3 * q[:, 0], 0.3 * q[:, 1] - 1.5, rnd(n_cy) - 0.5], 1), q))
    p = torch.cat([a for a, _ in parts])
    q = torch.cat([b for _, b in parts])
    if target == "composite":                   # position noise of lambda / 50 at 10 GHz
        p = p + torch.randn(p.shape, generator=g, device=DEV, dtype=torch.float64) * (C0 / 10e9 / 50)
    return p.float().contiguous(), q.float().contiguous()


def _target(case, seed):
    """Points, normals, radii and the bounding sphere of the case's target."""
    pos, nrm = _points(case["target"], case["n"], seed)
    rad, pca = api.point_attributes(pos, 8, 16, nrm, radius=True,
                                    normal=case["target"] == "composite")
    if pca is not None:                         # a scan's normals come from its points
        nrm = pca
    lo, hi = pos.amin(0).double(), pos.amax(0).double()
    centre = (lo + hi) / 2
    r = float((pos.double() - centre).norm(dim=1).max())
    return dict(pos=pos, nrm=nrm, rad=rad, centre=centre.tolist(), extent=1.02 * r,
                corners=torch.stack([lo, hi]).float().cpu().numpy())


def _views(t, W):
    return pipeline.views_from_angles([60.0] * 4 + [120.0] * 4, [45.0, 135.0, 225.0, 315.0] * 2,
                                      t["centre"], t["extent"], W, W)


def _freqs(case):
    """8-12 GHz for the metre-sized targets, 0.4-0.6 GHz for the 20 m plates."""
    lo, hi = (0.4e9, 0.6e9) if case["target"] == "octar" else (8e9, 12e9)
    nf = case["freqs"]
    if nf == 1:
        return np.array([0.5 * (lo + hi)])
    x = np.arange(nf) / (nf - 1.0)
    return lo + (hi - lo) * x if case.get("uniform", True) else lo * (hi / lo) ** x


def _sweep_args(case, t):
    a = case["angles"]
    th = np.full(a, 90.0 if case["target"] in ("dihedral", "sphere") else 60.0)
    span = 90.0 if case["target"] == "dihedral" else 360.0
    return api.SweepArgs(th, np.arange(a) * (span / a), case["W"], case["W"], t["centre"],
                         t["extent"], _freqs(case), case["bounces"])


def _screens(case, t):
    n = case["views"]
    th = 75.0 if case["target"] != "sphere" else 90.0
    return pipeline.views_from_angles([th] * n, [20.0 + 360.0 * k / n for k in range(n)],
                                      t["centre"], t["extent"], case["W"], case["W"])


def _net(seed):
    """Seeded initial parameters of the completion network."""
    rng = np.random.Generator(np.random.PCG64(seed))
    p = {}

    def put(name, shape, fan_in, scale=1.0):
        p[name + ".w"] = (scale / math.sqrt(fan_in) * rng.standard_normal(shape)).astype(np.float32)
        p[name + ".b"] = (0.1 * rng.standard_normal(shape[-1] if name.endswith(".dw") else shape[0])
                          ).astype(np.float32)

    def block(name, c):
        put(name + ".dw", (7, 7, c), 49)
        p[name + ".ln.g"] = (1.0 + 0.1 * rng.standard_normal(c)).astype(np.float32)
        p[name + ".ln.b"] = (0.1 * rng.standard_normal(c)).astype(np.float32)
        put(name + ".pw1", (4 * c, c), c)
        put(name + ".pw2", (c, 4 * c), 4 * c, 0.1)

    c = WIDTHS
    put("stem", (c[0], 3, 3, 1), 9)
    for lvl in range(4):
        if lvl:
            put(f"down{lvl}", (c[lvl], c[lvl - 1]), c[lvl - 1])
        for k in range(BLOCKS[lvl]):
            block(f"enc{lvl}.{k}", c[lvl])
    for head, nout in HEADS:
        for lvl in (2, 1, 0):
            put(f"{head}.up{lvl}", (4 * c[lvl], 3, 3, c[lvl + 1]), 9 * c[lvl + 1])
            put(f"{head}.fuse{lvl}", (c[lvl], 2 * c[lvl]), 2 * c[lvl])
            block(f"{head}.blk{lvl}", c[lvl])
        put(f"{head}.head", (nout, c[0]), c[0])
    p["normal.head.b"] = np.array([0.0, 0.0, 1.0], np.float32)   # toward the view, as trained
    return p


def _maps(case, seed):
    """Depth maps as the coarse splat leaves them: smooth where a surface
    was hit, zero elsewhere and in the holes between sparse points; with the
    dense targets of the same surface."""
    B, H, W = case["batch"], case["H"], case["W"]
    g = torch.Generator(device=DEV).manual_seed(seed)
    coarse = torch.randn(B, 2, 6, 6, generator=g, device=DEV)
    f = F.interpolate(coarse, size=(H, W), mode="bicubic", align_corners=True)
    d = 0.5 + 0.12 * f[:, 0]
    hit = f[:, 1] > -0.2
    du = F.pad(d[:, :, 2:] - d[:, :, :-2], (1, 1)) * (W / 8)
    dv = F.pad(d[:, 2:] - d[:, :-2], (0, 0, 1, 1)) * (H / 8)
    n = F.normalize(torch.stack([du, dv, torch.ones_like(du)], -1), dim=-1)
    seen = hit & (torch.rand(B, H, W, generator=g, device=DEV) < 0.6)
    x = torch.where(seen, d, torch.zeros_like(d)).to(torch.bfloat16).reshape(-1)
    m = hit.float()
    return (x, (d * m).reshape(-1).contiguous(), (n * m[..., None]).reshape(-1, 3).contiguous(),
            m.reshape(-1).contiguous())


def _layer_inputs(case, seed):
    """Activations, gradients and parameters of one block's layers."""
    B, H, W, C = case["batch"], case["H"], case["W"], case["C"]
    P = B * H * W
    g = torch.Generator(device=DEV).manual_seed(seed)
    rnd = lambda *s: torch.randn(*s, generator=g, device=DEV)
    act = lambda c, s=1.0: (s * rnd(P, c)).to(torch.bfloat16)
    return dict(x=act(C), a=act(C), bn=act(C), h=F.gelu(act(4 * C).float()).to(torch.bfloat16),
                z=act(4 * C), dy=act(C, 0.1), dz=act(4 * C, 0.1), dn=act(C, 0.1), da=act(C, 0.1),
                mean=0.1 * rnd(P), rstd=1.0 + 0.1 * torch.rand(P, generator=g, device=DEV),
                dw_w=rnd(7, 7, C) / 7, dw_b=0.1 * rnd(C), ln_g=1.0 + 0.1 * rnd(C),
                ln_b=0.1 * rnd(C), w1=(rnd(4 * C, C) / math.sqrt(C)).to(torch.bfloat16),
                b1=0.1 * rnd(4 * C), w2=(rnd(C, 4 * C) / math.sqrt(4 * C)).to(torch.bfloat16),
                b2=0.1 * rnd(C))


def prepare(case, seed):
    kind = case["kind"]
    s = dict(case=case)
    if kind == "forward" or kind == "gradient":
        s["net"] = learned.UNet(_net(seed), WIDTHS, BLOCKS, DEV)
        s["x"], s["d"], s["n"], s["m"] = _maps(case, seed)
        return s
    if kind == "layers":
        s["ops"] = learned.Ops(DEV)
        s["t"] = _layer_inputs(case, seed)
        return s
    if kind == "attributes":
        s["pos"], s["ref"] = _points(case["target"], case["n"], seed)
        return s
    t = s["t"] = _target(case, seed)
    if kind == "gfb":
        s["views"] = _screens(case, t)
        s["delta"] = 2.0 * s["views"][0].pitch
        return s
    gv = s["gviews"] = _views(t, case["view"])
    s["prm"] = pipeline.default_params(t["corners"], gv, edge_mode=case.get("edge", 0))
    if kind == "request" or kind == "sweep":
        s["args"] = _sweep_args(case, t)
    if kind == "geometry" or kind == "request":
        return s
    s["geom"], _ = pipeline.build_geometry(t["pos"], t["nrm"], t["rad"], gv, s["prm"])
    if kind == "sweep":                         # kept over the sweeps of one target
        s["args"].set_point_order(api.order_points(t["pos"]))
        s["ws"] = api.workspace(s["args"].workspace_bytes(), DEV)
        return s
    s["views"] = _screens(case, t)
    s["keys"] = api.build_gfb(s["views"], t["pos"], t["nrm"], t["rad"], 0, outputs=("keys",))["keys"]
    mb = case.get("bounces", 2)
    s["hits"] = api.alloc_hits(len(s["views"]) * case["W"] ** 2, mb, DEV)
    if kind == "field":
        api.trace_bounces(s["views"], s["keys"], t["nrm"], s["geom"], mb, s["prm"], hits=s["hits"])
        s["ks"] = np.array([[-c for c in v.d] for v in s["views"]], np.float32)
        s["freqs"] = _freqs(case)
    return s


# ---- one pass ---------------------------------------------------------------

def _run_request(s):
    t, c = s["t"], s["case"]
    rad, _ = api.point_attributes(t["pos"], 8, 16, None, radius=True, normal=False)
    geom, _ = pipeline.build_geometry(t["pos"], t["nrm"], rad, s["gviews"], s["prm"])
    E, sigma = api.rcs_sweep(s["args"], t["pos"], t["nrm"], rad, geom, s["prm"])
    return {"rad": rad, "E": E, "sigma": sigma}


def _run_layers(s):
    o, t, c = s["ops"], s["t"], s["case"]
    B, H, W, C = c["batch"], c["H"], c["W"], c["C"]
    P = B * H * W
    bf = lambda *n: torch.empty(*n, dtype=torch.bfloat16, device=DEV)
    f32 = lambda *n: torch.empty(*n, dtype=torch.float32, device=DEV)
    conv, norm, mean, rstd = bf(P, C), bf(P, C), f32(P), f32(P)
    o.dw(t["x"], t["dw_w"], t["dw_b"], B, H, W, C, conv)
    o.ln(t["a"], t["ln_g"], t["ln_b"], P, C, norm, mean, rstd)
    z, h, y = bf(P, 4 * C), bf(P, 4 * C), bf(P, C)
    o.linear(t["bn"], C, t["w1"], t["b1"], h, 4 * C, Z=z, gelu=True)
    o.linear(t["h"], 4 * C, t["w2"], t["b2"], y, C, R=t["x"], ldr=C)
    dz, dw2, db2 = bf(P, 4 * C), f32(C, 4 * C), f32(C)
    o.linear_bwd(t["dy"], t["h"], 4 * C, t["w2"], dz, 4 * C, dw2, db2, gelu_z=t["z"])
    dbn, dw1, db1 = bf(P, C), f32(4 * C, C), f32(4 * C)
    o.linear_bwd(t["dz"], t["bn"], C, t["w1"], dbn, C, dw1, db1)
    da, dg, dbeta = bf(P, C), f32(C), f32(C)
    o.ln_bwd(t["dn"], t["a"], t["ln_g"], t["mean"], t["rstd"], P, C, da, dg, dbeta)
    dx, dww, dwb = bf(P, C), f32(7, 7, C), f32(C)
    o.dw_bwd(t["x"], t["da"], t["dw_w"], B, H, W, C, dx, dww, dwb)
    return dict(conv=conv, norm=norm, mean=mean, rstd=rstd, z=z, h=h, y=y, dz=dz, dw2=dw2, db2=db2,
                dbn=dbn, dw1=dw1, db1=db1, da=da, dg=dg, dbeta=dbeta, dx=dx, dww=dww, dwb=dwb)


def run(state):
    s, c = state, state["case"]
    kind = c["kind"]
    if kind == "forward":
        return s["net"].forward(s["x"], c["batch"], c["H"], c["W"])[0]
    if kind == "gradient":
        net, B, H, W = s["net"], c["batch"], c["H"], c["W"]
        outs, tape = net.forward(s["x"], B, H, W)
        loss, grads = net.losses(outs, s["d"], s["n"], s["m"], B, H, W)
        net.backward(tape, grads)
        return {"loss": loss, "grad": net.grad, "outs": outs}
    if kind == "layers":
        return _run_layers(s)
    if kind == "attributes":
        rad, nrm = api.point_attributes(s["pos"], c["k_r"], c["k_n"], s["ref"],
                                        normal=c["normal"])
        return {"rad": rad, "nrm": nrm}
    if kind == "request":
        return _run_request(s)
    t = s["t"]
    if kind == "gfb":
        if c["tube"]:
            return api.build_gfb(s["views"], t["pos"], None, None, 1, s["delta"], outputs=("keys",))
        return api.build_gfb(s["views"], t["pos"], t["nrm"], t["rad"], 0, outputs=("nd", "keys"))
    if kind == "geometry":
        geom, gfb = pipeline.build_geometry(t["pos"], t["nrm"], t["rad"], s["gviews"], s["prm"])
        cr, nf = geom.planes()
        return {"centre": cr, "normal": nf, "mask": gfb["mask"]}
    if kind == "sweep":
        E, sigma = api.rcs_sweep(s["args"], t["pos"], t["nrm"], t["rad"], s["geom"], s["prm"],
                                 ws=s["ws"])
        return {"E": E, "sigma": sigma}
    if kind == "trace":
        h = api.trace_bounces(s["views"], s["keys"], t["nrm"], s["geom"], c["bounces"], s["prm"],
                              hits=s["hits"])
        return dict(p=h.p, n=h.n, k=h.k, u=h.u, v=h.v, path=h.path, M=h.M, psi=h.psi, ids=h.ids)
    return api.po_field(s["hits"], len(s["views"]), c["W"] ** 2, s["ks"], s["freqs"])


# ---- what a pass cannot do without ------------------------------------------

def work(case):
    """Inputs read once and outputs written once; a bounce query at least
    reads its ray's key and writes its count, a field term is 64 operations
    on about half of the rays (those that hit the target)."""
    kind = case["kind"]
    if kind in ("forward", "gradient"):
        B, H, W = case["batch"], case["H"], case["W"]
        px = B * H * W
        fl = B * learned_train.forward_flops(WIDTHS, BLOCKS, H, W)
        weights = 4 * 3.2e6
        if kind == "forward":
            return {"bytes": px * (2 + 20) + weights, "flops": fl}
        return {"bytes": px * (2 + 20 + 20) + 2 * weights, "flops": 3 * fl}
    if kind == "layers":
        px, C = case["batch"] * case["H"] * case["W"], case["C"]
        # read x a bn h z dy dz dn da, written conv norm z h y dz dbn da dx; weights small
        return {"bytes": px * C * 2.0 * (7 + 12 + 6 + 12) + 16.0 * px,
                "flops": px * C * (2.0 * 49 * 3 + 6 * 2 * 4 * C)}
    n = case["n"]
    if kind == "attributes":
        return {"bytes": n * (12 + 12 + 4 + (12 if case["normal"] else 0)), "flops": n * 16 * 8.0}
    if kind == "gfb":
        px = case["views"] * case["W"] ** 2
        return {"bytes": n * (12 if case["tube"] else 28) + px * (8 if case["tube"] else 24),
                "flops": n * case["views"] * 30.0}
    vp = 8 * case["view"] ** 2
    if kind == "geometry":
        return {"bytes": 28 * n + vp * (17 + 32), "flops": (n * 8 + vp) * 30.0}
    rays = case["W"] ** 2 * (case.get("views") or case["angles"])
    if kind == "trace":
        return {"bytes": rays * (8 + 85 + 4 * case["bounces"]), "flops": rays * case["bounces"] * 100.0}
    if kind == "field":
        return {"bytes": rays * 73.0, "flops": 0.5 * rays * case["freqs"] * 64}
    geo = 28 * n + (vp * (17 + 32) if kind == "request" else vp * 32)
    return {"bytes": geo + rays * (16 + 5 * case["bounces"]) + 256.0 * case["angles"] * case["freqs"],
            "flops": rays * (100.0 * case["bounces"] + 0.5 * 64 * case["freqs"])}


# ---- the same in 64 bits ----------------------------------------------------

def _field64(s):
    """Eq. 14 over the state's records."""
    h, ks = s["hits"], torch.tensor(s["ks"], device=DEV, dtype=torch.float64)
    per = s["case"]["W"] ** 2
    out = []
    for g in range(len(s["views"])):
        sl = slice(g * per, (g + 1) * per)
        ok = (h.M[sl] >= 1) & (h.psi[sl] != 0)
        p, n, k, u, v = (getattr(h, q)[sl][ok].double() for q in "pnkuv")
        q = k - ks[g]
        dot = lambda a, b: (a * b).sum(-1, keepdim=True)
        nk = dot(n, k)
        up, vp = u - k * (dot(n, u) / nk), v - k * (dot(n, v) / nk)
        area = torch.linalg.cross(up, vp).norm(dim=1)
        sinc = lambda x: torch.sinc(x / math.pi)
        au, av = 0.5 * dot(q, up)[:, 0], 0.5 * dot(q, vp)[:, 0]
        delta = h.path[sl][ok] - (p @ ks[g])
        kg = ks[g].expand_as(n)
        vec = [torch.linalg.cross(torch.linalg.cross(torch.linalg.cross(n, e), kg), kg)
               for e in (-v / v.norm(dim=1, keepdim=True), u / u.norm(dim=1, keepdim=True))]
        rows = []
        for f in s["freqs"]:
            kf = 2 * math.pi * float(f) / C0
            a = area * sinc(kf * au) * sinc(kf * av)
            re, im = a * torch.cos(kf * delta), -a * torch.sin(kf * delta)
            rows.append(torch.stack([torch.stack([re @ w, im @ w], -1) for w in vec]))
        out.append(torch.stack(rows))
    return torch.stack(out)


def _attributes64(s, c):
    pos = s["pos"].double()
    n = pos.shape[0]
    rad, nrm = [], []
    K = max(c["k_r"] + 1, c["k_n"])
    ctr = pos.mean(0)
    q = pos - ctr
    sq = (q * q).sum(1)
    step = max(1, (1 << 27) // n)
    for i in range(0, n, step):
        b = q[i:i + step]
        d2 = sq[None] - 2.0 * (b @ q.T)
        idx = d2.topk(K + 4, largest=False).indices
        d2 = (q[idx] - b[:, None]).square().sum(-1)
        d2, o = d2.sort(1)
        idx = idx.gather(1, o)
        rad.append(d2[:, 1:c["k_r"] + 1].sqrt().mean(1))
        if c["normal"]:
            nb = q[idx[:, :c["k_n"]]]
            nb = nb - nb.mean(1, keepdim=True)
            cov = nb.transpose(1, 2) @ nb
            w = torch.linalg.eigh(cov.cpu())[1][:, :, 0].to(DEV)
            r = s["ref"][i:i + step].double()
            nrm.append(torch.where((w * r).sum(1, keepdim=True) < 0, -w, w))
    return {"rad": torch.cat(rad), "nrm": torch.cat(nrm) if c["normal"] else None}


def _dw64(x, w, flip=False):
    """Depthwise 7x7 of NHWC x, as 49 shifted products."""
    B, H, W, C = x.shape
    xp = F.pad(x, (0, 0, 3, 3, 3, 3))
    y = torch.zeros_like(x)
    for i in range(7):
        for j in range(7):
            wv = w[6 - i, 6 - j] if flip else w[i, j]
            y += wv * xp[:, i:i + H, j:j + W]
    return y


def _layers64(s, c):
    t = {k: v.double() for k, v in s["t"].items()}
    B, H, W, C = c["batch"], c["H"], c["W"], c["C"]
    img = lambda a: a.view(B, H, W, C)
    flat = lambda a: a.reshape(-1, C)
    mean = t["a"].mean(1)
    rstd = (t["a"].var(1, unbiased=False) + learned.LN_EPS).rsqrt()
    z = t["bn"] @ t["w1"].T + t["b1"]
    gg = 0.5 * (1 + torch.erf(t["z"] / math.sqrt(2))) + t["z"] * torch.exp(
        -0.5 * t["z"] ** 2) / math.sqrt(2 * math.pi)
    xh = (t["a"] - t["mean"][:, None]) * t["rstd"][:, None]
    gy = t["dn"] * t["ln_g"]
    da = t["rstd"][:, None] * (gy - gy.mean(1, keepdim=True) - xh * (gy * xh).mean(1, keepdim=True))
    xp, g = F.pad(img(t["x"]), (0, 0, 3, 3, 3, 3)), img(t["da"])
    dww = torch.stack([torch.stack([(xp[:, i:i + H, j:j + W] * g).sum((0, 1, 2)) for j in range(7)])
                       for i in range(7)])
    return dict(conv=flat(_dw64(img(t["x"]), t["dw_w"]) + t["dw_b"]),
                norm=(t["a"] - mean[:, None]) * rstd[:, None] * t["ln_g"] + t["ln_b"], mean=mean,
                rstd=rstd, z=z, h=F.gelu(z), y=t["h"] @ t["w2"].T + t["b2"] + t["x"],
                dz=(t["dy"] @ t["w2"]) * gg, dw2=t["dy"].T @ t["h"], db2=t["dy"].sum(0),
                dbn=t["dz"] @ t["w1"], dw1=t["dz"].T @ t["bn"], db1=t["dz"].sum(0), da=da,
                dg=(t["dn"] * xh).sum(0), dbeta=t["dn"].sum(0),
                dx=flat(_dw64(img(t["da"]), t["dw_w"], flip=True)), dww=dww, dwb=t["da"].sum(0))


def _forward64(net, x, B, H, W):
    """The network's outputs from its FP32 parameters."""
    P = {k: net.pf(k).double() for k in net.slots}
    c1 = lambda y, n: F.conv2d(y, P[n + ".w"][:, :, None, None], P[n + ".b"])

    def c3(y, n):
        return F.conv2d(y, P[n + ".w"].permute(0, 3, 1, 2), P[n + ".b"], padding=1)

    def block(y, n):
        a = _dw64(y.permute(0, 2, 3, 1).contiguous(), P[n + ".dw.w"]) + P[n + ".dw.b"]
        a = F.layer_norm(a, (a.shape[-1],), P[n + ".ln.g"], P[n + ".ln.b"], learned.LN_EPS)
        a = F.gelu(F.linear(a, P[n + ".pw1.w"], P[n + ".pw1.b"]))
        return y + F.linear(a, P[n + ".pw2.w"], P[n + ".pw2.b"]).permute(0, 3, 1, 2)

    x = x.double().view(B, 1, H, W)
    y, skips = c3(x, "stem"), []
    for lvl in range(4):
        if lvl:
            y = c1(F.max_pool2d(y, 2), f"down{lvl}")
        for k in range(BLOCKS[lvl]):
            y = block(y, f"enc{lvl}.{k}")
        skips.append(y)
    out = {}
    for head, nout in HEADS:
        u = skips[-1]
        for lvl in (2, 1, 0):
            u = F.pixel_shuffle(c3(u, f"{head}.up{lvl}"), 2)
            u = block(c1(torch.cat([u, skips[lvl]], 1), f"{head}.fuse{lvl}"), f"{head}.blk{lvl}")
        u = c1(u, f"{head}.head")
        u = u + x if head == "depth" else u
        out[head] = u.permute(0, 2, 3, 1).reshape(-1, nout) if nout > 1 else u.reshape(-1)
    return out


def exact(case, seed):
    kind = case["kind"]
    if kind == "field":
        return _field64(prepare(case, seed))
    if kind == "attributes" and case["n"] <= 100_000:
        return _attributes64(prepare(case, seed), case)
    if kind == "layers":
        return _layers64(prepare(case, seed), case)
    if kind in ("forward", "gradient") and case["batch"] * case["H"] * case["W"] <= 1 << 20:
        s = prepare(case, seed)
        with torch.no_grad():
            outs = _forward64(s["net"], s["x"], case["batch"], case["H"], case["W"])
        if kind == "forward":
            return outs
        return {"loss": None, "grad": None, "outs": outs}
    return None                                 # traced paths: indices and counts are compared
