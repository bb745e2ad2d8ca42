"""The work that users of this library have it do, as cases that can be timed.

A case is one pass through public entry points at one size: whole optimisation
steps (`pipeline.ShadingPipeline`), whole render requests
(`serving.ServingEngine`), and single parts through the calls a program of its
own would make (`mcdi.ShadeMC`, `mcdi.Denoise`, `mcdi.Bvh`,
`mcdi.bilateral_fwd`, `mcdi.image_loss`, `mcdi.shadow_edge_grad`, ...).
Inputs have the shapes of the repository's own workloads: marching-tetrahedra
meshes of sphere and box unions, value-noise textures, log-normal probes with
sun lobes, orbit cameras, Xavier-initialised denoisers.  They are made on the
GPU from the seed alone.
"""
from __future__ import annotations

import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2206_03380_gb300 import mcdi, scenes
from paper_2206_03380_gb300.pipeline import ShadingPipeline
from paper_2206_03380_gb300.scenes import RenderRequest, Scene, split_spp
from paper_2206_03380_gb300.serving import ServingEngine

DEV = "cuda"
UVMAP = np.array([-1.0, -1.0, 0.5], np.float32)
UNET_FLOPS = 2 * 9 * (9 * 32 + 32 * 32 + 80 * 32 + 32 * 32 + 32 * 3 + (32 * 48 + 48 * 48 + 112 * 48 + 48 * 48) / 4 +
                      (48 * 64 + 64 * 64 + 160 * 64 + 64 * 64) / 16 + (64 * 96 + 96 * 96) / 64)  # per full-size pixel
SAMPLE_FLOPS = 300.0  # drawing, weighing and shading one sample, its shadow ray's traversal not counted


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # the smallest request a serving loop gets: 128 x 128 at 4 samples, where launches and latency count
        dict(name="render-128", kind="render", res=128, spp=4, grid=64, boxes=0, tex=512, env=256),
        # its largest: 1024 x 1024 at 64 samples against a mesh of about half a million triangles
        dict(name="render-1024", kind="render", res=1024, spp=64, grid=192, boxes=0, tex=512, env=1024),
        # the optimisation step at its usual size: one 512 x 512 view, 16 samples, about 200k triangles, BF16 U-Net
        dict(name="step-512", kind="step", views=1, height=512, width=512, spp=16, grid=128, boxes=0, tex=1024,
             env=512, denoiser="bf16"),
        # the largest: eight 800 x 800 views of a million triangles at 32 samples
        dict(name="step-batch", kind="step", views=8, height=800, width=800, spp=32, grid=256, boxes=32, tex=2048,
             env=1024, denoiser="bf16"),
        # the estimator alone as an autograd function, forward and adjoint, with the forward's visibility kept
        dict(name="shade-512", kind="shade", views=1, height=512, width=512, spp=16, grid=128, boxes=0, env=512,
             mask=True, workspace=True, decorrelate=False),
        # the same at ragged sizes, without scratch memory and with the adjoint's own samples (App. D)
        dict(name="shade-ragged", kind="shade", views=3, height=155, width=203, spp=11, grid=96, boxes=8, env=256,
             mask=False, workspace=False, decorrelate=True),
        # the denoiser on the two terms of a view, forward and input gradient, in both precisions
        dict(name="denoise-512", kind="denoise", images=2, height=512, width=512, precision="bf16", train=False),
        dict(name="denoise-e4m3", kind="denoise", images=4, height=264, width=344, precision="e4m3", train=False),
        # the live-trained denoiser: forward, input gradient and weight gradient
        dict(name="denoise-train", kind="denoise", images=2, height=256, width=256, precision="bf16", train=True),
        # a new mesh of a million triangles and its G-buffer by ray casting
        dict(name="cast-1m", kind="cast", height=512, width=512, grid=256, boxes=32, tex=512, refit=False),
        # the denoiser without a network: cross-bilateral filter, image loss and its gradient back through the filter
        dict(name="bilateral-512", kind="bilateral", views=1, height=512, width=512, grid=128, boxes=0, sigma=2.0),
        # shadow-visibility gradients: the edge table of a new topology and the edge samples of a view
        dict(name="edges-512", kind="edges", height=512, width=512, grid=128, boxes=0, env=512, samples=16),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _by8(v, lo=16):
    return max(lo, (v + 4) // 8 * 8)


def draw(rng):
    kind = rng.choice(["render", "step", "step", "shade", "shade", "denoise", "denoise", "cast", "bilateral", "edges"])
    grid, boxes = _log(rng, 24, 256), rng.choice([0, 0, 8, 32])
    if kind == "render":
        return dict(kind=kind, res=32 * rng.randint(4, 32), spp=rng.choice([4, 8, 16, 32, 64]), grid=grid, boxes=0,
                    tex=rng.choice([256, 512, 1024]), env=rng.choice([256, 512, 1024]))
    height, width = _log(rng, 64, 800), _log(rng, 64, 800)
    if kind == "step":
        return dict(kind=kind, views=_log(rng, 1, 6), height=_by8(height), width=_by8(width), spp=rng.randint(4, 32),
                    grid=grid, boxes=boxes, tex=rng.choice([500, 1024, 2048]), env=rng.choice([254, 512, 1024]),
                    denoiser=rng.choice(["bf16", "bf16", "e4m3", "bilateral", "none"]))
    if kind == "shade":
        return dict(kind=kind, views=_log(rng, 1, 4), height=height, width=width, spp=rng.randint(3, 40), grid=grid,
                    boxes=boxes, env=rng.choice([32, 254, 512, 1024]), mask=rng.random() < 0.7,
                    workspace=rng.random() < 0.7, decorrelate=rng.random() < 0.3)
    if kind == "denoise":
        return dict(kind=kind, images=_log(rng, 1, 8), height=_by8(height), width=_by8(width),
                    precision=rng.choice(["bf16", "bf16", "e4m3"]), train=rng.random() < 0.4)
    if kind == "cast":
        return dict(kind=kind, height=height, width=width, grid=grid, boxes=boxes, tex=rng.choice([256, 500, 1024]),
                    refit=rng.random() < 0.5)
    if kind == "bilateral":
        return dict(kind=kind, views=_log(rng, 1, 4), height=height, width=width, grid=grid, boxes=boxes,
                    sigma=round(rng.uniform(0.6, 4.0), 2))
    return dict(kind=kind, height=height, width=width, grid=grid, boxes=boxes, env=rng.choice([128, 512]),
                samples=rng.randint(1, 24))


# ------------------------------------------------------------------ inputs
def _primitives(rng, boxes):
    """32 spheres (radii 0.05-0.3) and some axis-aligned boxes: (centre, radius) and (centre, half extents)."""
    return (rng.uniform(-0.62, 0.62, (32, 3)), rng.uniform(0.05, 0.3, 32), rng.uniform(-0.62, 0.62, (boxes, 3)),
            rng.uniform(0.04, 0.22, (boxes, 3)))


def _distance(p, prim, k):
    """Signed distance of points p (..., 3) to primitive k, and the direction it grows in."""
    sc, sr, bc, bh = prim
    if k < len(sr):
        v = p - sc[k]
        l = v.norm(dim=-1)
        return l - sr[k], v / l.clamp_min(1e-12)[..., None]
    v = p - bc[k - len(sr)]
    q = v.abs() - bh[k - len(sr)]
    out = q.clamp_min(0)
    lo = out.norm(dim=-1)
    face = F.one_hot(q.argmax(-1), 3).to(p.dtype)
    n = torch.where((lo > 0)[..., None], out / lo.clamp_min(1e-12)[..., None], face) * v.sign()
    return lo + q.amax(-1).clamp_max(0), n


def _mesh(grid, boxes, seed):
    """Marching tetrahedra (Kuhn split) of the union's distance field on a grid^3 lattice over [-1.35, 1.35]^3:
    float32 vertices and unit normals, int32 triangles, vertices on shared lattice edges welded."""
    n, ext = grid, 1.35
    prim = [torch.tensor(a, device=DEV, dtype=torch.float64) for a in _primitives(np.random.default_rng(seed), boxes)]
    n_prim = len(prim[1]) + boxes
    lin = torch.linspace(-ext, ext, n, device=DEV, dtype=torch.float64)
    sdf = torch.empty((n, n, n), device=DEV, dtype=torch.float64)  # [z, y, x]
    for z0 in range(0, n, 32):
        Z, Y, X = torch.meshgrid(lin[z0:z0 + 32], lin, lin, indexing="ij")
        p = torch.stack([X, Y, Z], -1).float()
        d = torch.full(p.shape[:-1], 1e9, device=DEV)
        for k in range(n_prim):
            d = torch.minimum(d, _distance(p, [a.float() for a in prim], k)[0])
        sdf[z0:z0 + 32] = d
    inside = sdf < 0
    corners = [(c & 1, c >> 1 & 1, c >> 2 & 1) for c in range(8)]
    cells = [inside[dz:dz + n - 1, dy:dy + n - 1, dx:dx + n - 1] for dx, dy, dz in corners]
    hit = torch.zeros_like(cells[0])
    for c in cells[1:]:
        hit |= c != cells[0]
    cz, cy, cx = hit.nonzero(as_tuple=True)
    gid = torch.stack([(cx + dx) + n * ((cy + dy) + n * (cz + dz)) for dx, dy, dz in corners], 1)
    flat, keys = sdf.reshape(-1), []
    tets = [[0, 1, 3, 7], [0, 1, 5, 7], [0, 2, 3, 7], [0, 2, 6, 7], [0, 4, 5, 7], [0, 4, 6, 7]]
    for tet in tets:
        g = gid[:, tet]
        mask = ((flat[g] < 0).long() * torch.tensor([1, 2, 4, 8], device=DEV)).sum(1)
        for m in range(1, 15):
            ins, out = [k for k in range(4) if m >> k & 1], [k for k in range(4) if not m >> k & 1]
            if len(ins) == 2:
                (a, b), (c, d) = ins, out
                tris = [[(a, c), (a, d), (b, d)], [(a, c), (b, d), (b, c)]]
            else:
                a = (ins if len(ins) == 1 else out)[0]
                o = [k for k in range(4) if k != a]
                tris = [[(a, o[0]), (a, o[1]), (a, o[2])]]
            s = g[mask == m]
            for tri in tris:
                keys.append(torch.stack([torch.minimum(s[:, a], s[:, b]) * n ** 3 + torch.maximum(s[:, a], s[:, b])
                                         for a, b in tri], 1))
    keys = torch.cat(keys)
    uniq, inv = torch.unique(keys, return_inverse=True)
    ga, gb = uniq // n ** 3, uniq % n ** 3
    fa, fb = flat[ga], flat[gb]
    at = lambda g: torch.stack([lin[g % n], lin[(g // n) % n], lin[g // (n * n)]], 1)
    pa, pb = at(ga), at(gb)
    verts = pa + (fa / (fa - fb))[:, None] * (pb - pa)
    best, nrm = torch.full((len(verts),), 1e9, device=DEV, dtype=torch.float64), torch.zeros_like(verts)
    for k in range(n_prim):
        d, g = _distance(verts, prim, k)
        near = d < best
        best, nrm = torch.where(near, d, best), torch.where(near[:, None], g, nrm)
    nrm = F.normalize(nrm, dim=1)
    return verts.float().contiguous(), nrm.float().contiguous(), inv.reshape(-1, 3).int().contiguous()


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _noise(S, channels, gen):
    """Smooth value noise in [0, 1], (S, S, channels)."""
    acc = 0.0
    for k, L in enumerate((4, 8, 16, 32)):
        lat = torch.rand((1, channels, L, L), generator=gen, device=DEV)
        acc = acc + 0.5 ** k * F.interpolate(lat, size=(S, S), mode="bilinear", align_corners=True)
    lo, hi = acc.amin((2, 3), keepdim=True), acc.amax((2, 3), keepdim=True)
    return ((acc - lo) / (hi - lo))[0].permute(1, 2, 0)


def _textures(S, gen):
    """k_d in [0, 1]; roughness in [0.08, 1], metallic blended toward {0, 1}."""
    kd, korm = (torch.zeros((S, S, 4), device=DEV) for _ in range(2))
    kd[..., :3] = _noise(S, 3, gen)
    korm[..., :3] = _noise(S, 3, gen)
    korm[..., 1] = 0.08 + 0.92 * korm[..., 1]
    x = ((korm[..., 2] - 0.42) / 0.16).clamp(0, 1)
    korm[..., 2] = x * x * (3 - 2 * x)
    return kd, korm


def _probe(W, gen):
    """Log-normal texels and three Gaussian lobes of peak 1e3 in the upper hemisphere, (W / 2, W, 4)."""
    H = W // 2
    env = torch.zeros((H, W, 4), device=DEV)
    env[..., :3] = torch.randn((H, W, 3), generator=gen, device=DEV).exp()
    th = math.pi * (torch.arange(H, device=DEV) + 0.5) / H
    ph = 2 * math.pi * (torch.arange(W, device=DEV) + 0.5) / W
    T, P = torch.meshgrid(th, ph, indexing="ij")
    dirs = torch.stack([T.sin() * P.cos(), T.cos(), T.sin() * P.sin()], -1)
    r = torch.rand((3, 6), generator=gen, device=DEV).tolist()
    for a, b, c, *tint in r:
        z, p = 0.15 + 0.8 * a, 2 * math.pi * b
        s = math.sqrt(1 - z * z)
        d = torch.tensor([s * math.cos(p), z, s * math.sin(p)], device=DEV)
        ang = (dirs @ d).clamp(-1, 1).acos()
        sig = math.radians(1 + 3 * c)
        env[..., :3] += 1e3 * torch.exp(-0.5 * (ang / sig) ** 2)[..., None] * (0.8 + 0.2 * torch.tensor(tint, device=DEV))
    return env


def _cameras(views, height, width, seed):
    return scenes.orbit_cameras(200, list(range(views)), 2.4, 45.0, width / height, np.random.default_rng(seed))


def _unet(seed):
    return mcdi.flatten_unet_params(scenes.unet_xavier_weights(seed))


def _radiance(shape, gen):
    """Positive, long-tailed pixel values with w = 0."""
    t = torch.zeros((*shape, 4), device=DEV)
    t[..., :3] = torch.randn((*shape, 3), generator=gen, device=DEV).exp()
    return t


def _gradient(shape, gen, scale=1.0):
    t = torch.zeros((*shape, 4), device=DEV)
    t[..., :3] = torch.randn((*shape, 3), generator=gen, device=DEV) * scale
    return t


def _gbuffer(case, seed, views, mesh, gen):
    verts, vnrm, tris = mesh
    H, W = case["height"], case["width"]
    kd, korm = _textures(512, gen)
    cams = torch.from_numpy(_cameras(views, H, W, seed)).to(DEV)
    gb = mcdi.GBuffer.allocate(views, H, W)
    ws = mcdi._empty_bytes(mcdi.raster_workspace_size(views, H, W), DEV)
    mcdi.raster_gbuffer(verts, vnrm, tris, cams, H, W, kd, korm, UVMAP, gb, ws)
    return gb, cams


# ------------------------------------------------------------------ prepare
def prepare(case, seed):
    state = globals()["_prepare_" + case["kind"]](case, int(seed), _gen(seed))
    state["kind"] = case["kind"]
    return state


def _prepare_render(case, seed, gen):
    verts, vnrm, tris = _mesh(case["grid"], case["boxes"], seed)
    kd, korm = _textures(case["tex"], gen)
    c = lambda t: t.cpu().numpy()
    scene = dict(verts=c(verts), vnrm=c(vnrm), tris=c(tris), tex_kd=c(kd), tex_korm=c(korm),
                 cams=_cameras(4, 1, 1, seed), uvmap=UVMAP)
    engine = ServingEngine([scene], [c(_probe(case["env"], gen))], _unet(seed), n_slots=1, sides=(case["res"],),
                           max_spp=case["spp"])
    return dict(engine=engine, request=RenderRequest(0, 0.0, 0, 0, case["res"], case["spp"], seed % 4, seed + 1))


def _prepare_step(case, seed, gen):
    verts, vnrm, tris = _mesh(case["grid"], case["boxes"], seed)
    kd, korm = _textures(case["tex"], gen)
    c = lambda t: t.cpu().numpy()
    n, h, w = case["views"], case["height"], case["width"]
    scene = Scene("step", c(verts), c(vnrm), c(tris), c(_probe(case["env"], gen)), c(kd), c(korm), UVMAP,
                  _cameras(n, h, w, seed), w, h, *split_spp(case["spp"]), seed + 1)
    d = case["denoiser"]
    pipe = ShadingPipeline(scene, device=DEV, denoiser_params=_unet(seed) if d in ("bf16", "e4m3") else None,
                           denoiser_precision=mcdi.E4M3 if d == "e4m3" else mcdi.BF16,
                           bilateral_sigma=2.0 if d == "bilateral" else None)
    ref = _radiance((n, h, w), gen)
    pipe.capture_loss_step(ref)
    return dict(pipe=pipe, ref=ref)


def _prepare_shade(case, seed, gen):
    mesh = _mesh(case["grid"], case["boxes"], seed)
    n, h, w = case["views"], case["height"], case["width"]
    gb, cams = _gbuffer(case, seed, n, mesh, gen)
    env = _probe(case["env"], gen)
    prm = mcdi.make_params(*split_spp(case["spp"]), seed=seed + 1, decorrelate_bwd=case["decorrelate"])
    ws = mcdi._empty_bytes(mcdi.shade_workspace_size(n, h, w, prm), DEV) if case["workspace"] else None
    return dict(bvh=mcdi.Bvh.allocate(mesh[2].shape[0]).build(mesh[0], mesh[2]), probe=mcdi.Probe.allocate(env).build(),
                leaves=[t.requires_grad_() for t in (gb.kd, gb.korm, gb.nrm, env)], pos=gb.pos, cams=cams, params=prm,
                mask=case["mask"], workspace=ws, grads=[_gradient((n, h, w), gen) for _ in range(3)])


def _prepare_denoise(case, seed, gen):
    n, h, w = case["images"], case["height"], case["width"]
    den = mcdi.Denoiser(_unet(seed), n, h, w, precision=mcdi.E4M3 if case["precision"] == "e4m3" else mcdi.BF16)
    aux = max(1, n // 2) if n % 2 == 0 else n
    kd = torch.zeros((aux, h, w, 4), device=DEV)
    kd[..., :3] = torch.rand((aux, h, w, 3), generator=gen, device=DEV)
    nrm = torch.zeros((aux, h, w, 4), device=DEV)
    nrm[..., :3] = F.normalize(torch.randn((aux, h, w, 3), generator=gen, device=DEV), dim=-1)
    return dict(denoiser=den, term=_radiance((n, h, w), gen).requires_grad_(), kd=kd, nrm=nrm,
                gy=_gradient((n, h, w), gen), train=case["train"])


def _prepare_cast(case, seed, gen):
    verts, vnrm, tris = _mesh(case["grid"], case["boxes"], seed)
    bvh = mcdi.Bvh.allocate(tris.shape[0])
    if case["refit"]:  # a fixed topology whose vertices moved since the last build
        bvh.build(verts, tris)
        verts = verts + 0.01 * torch.sin(7.0 * verts.roll(1, 1))
    kd, korm = _textures(case["tex"], gen)
    h, w = case["height"], case["width"]
    return dict(bvh=bvh, mesh=(verts.contiguous(), vnrm, tris), cams=torch.from_numpy(_cameras(1, h, w, seed)).to(DEV),
                tex=(kd, korm), gb=mcdi.GBuffer.allocate(1, h, w), size=(h, w), refit=case["refit"])


def _prepare_bilateral(case, seed, gen):
    n, h, w = case["views"], case["height"], case["width"]
    gb, cams = _gbuffer(case, seed, n, _mesh(case["grid"], case["boxes"], seed), gen)
    z = lambda *s, dtype=torch.float32: torch.zeros(s, device=DEV, dtype=dtype)
    return dict(gb=gb, cams=cams, sigma=case["sigma"], terms=_radiance((2 * n, h, w), gen), ref=_radiance((n, h, w), gen),
                den=z(2 * n, h, w, 4), wsum=z(n, h, w), color=z(n, h, w, 4), loss=z(3, dtype=torch.float64),
                g_kd=z(n, h, w, 4), g_den=z(2 * n, h, w, 4), g_terms=z(2 * n, h, w, 4),
                ws=mcdi._empty_bytes(mcdi.image_loss_workspace_size(n * h * w), DEV))


def _prepare_edges(case, seed, gen):
    # one shape whose triangle list starts elsewhere for each seed, so that the table's capacity is the same
    verts, vnrm, tris = _mesh(case["grid"], case["boxes"], 1)
    tris = tris.roll(7919 * (seed % 1009), 0).contiguous()
    h, w = case["height"], case["width"]
    gb, cams = _gbuffer(case, seed, 1, (verts, vnrm, tris), gen)
    n = tris.shape[0]
    edges = mcdi.EdgeTable(torch.zeros((3 * n, 4), dtype=torch.int32, device=DEV),
                           torch.zeros(1, dtype=torch.int32, device=DEV),
                           mcdi._empty_bytes(mcdi.edge_table_workspace_size(n), DEV))
    return dict(bvh=mcdi.Bvh.allocate(n).build(verts, tris), verts=verts, tris=tris, edges=edges, gb=gb, cams=cams,
                probe=mcdi.Probe.allocate(_probe(case["env"], gen)).build(),
                params=mcdi.make_params(8, 4, 4, seed=seed + 1), samples=case["samples"],
                g_cd=_gradient((1, h, w), gen), g_cs=_gradient((1, h, w), gen), g_verts=torch.zeros_like(verts))


# ------------------------------------------------------------------ run
def run(state):
    return globals()["_run_" + state["kind"]](state)


def _run_render(s):
    return s["engine"].render_one(s["request"])


def _run_step(s):
    p = s["pipe"]
    p.replay()
    return dict(loss=p.loss, color=p.color, kd_out=p.kd_out, c_d=p.c_d, c_s=p.c_s, g_kd=p.g_kd, g_korm=p.g_korm,
                g_nrm=p.g_nrm, g_env=p.g_env)


def _run_shade(s):
    out = mcdi.ShadeMC.apply(*s["leaves"], s["pos"], s["bvh"], s["probe"], s["cams"], s["params"], s["mask"],
                             s["workspace"])
    return dict(out=[t.detach() for t in out], grads=torch.autograd.grad(out, s["leaves"], s["grads"]))


def _run_denoise(s):
    y = mcdi.Denoise.apply(s["term"], s["kd"], s["nrm"], s["denoiser"])
    gx, = torch.autograd.grad(y, s["term"], s["gy"])
    return dict(y=y.detach(), gx=gx, gw=s["denoiser"].weight_grad() if s["train"] else None)


def _run_cast(s):
    verts, vnrm, tris = s["mesh"]
    (s["bvh"].refit if s["refit"] else s["bvh"].build)(verts, tris)
    gb = s["gb"]
    mcdi.primary_cast(s["bvh"], verts, vnrm, tris, s["cams"], *s["size"], *s["tex"], UVMAP, gb)
    return [gb.pos, gb.nrm, gb.kd, gb.korm]


def _run_bilateral(s):
    gb, n = s["gb"], s["gb"].pos.shape[0]
    mcdi.bilateral_fwd(gb.pos, gb.nrm, s["cams"], s["terms"], s["sigma"], s["den"], s["wsum"])
    mcdi.image_loss(gb.kd, s["den"][:n], s["den"][n:], s["ref"], s["loss"], s["g_kd"], s["g_den"][:n], s["g_den"][n:],
                    s["ws"], 0.15, s["color"])
    mcdi.bilateral_bwd(gb.pos, gb.nrm, s["cams"], s["wsum"], s["g_den"], s["sigma"], s["g_terms"])
    return dict(den=s["den"], wsum=s["wsum"], color=s["color"], loss=s["loss"], g_kd=s["g_kd"], g_terms=s["g_terms"])


def _run_edges(s):
    s["edges"].build(s["tris"])
    s["g_verts"].zero_()
    mcdi.shadow_edge_grad(s["bvh"], s["verts"], s["edges"], s["probe"], s["gb"], s["cams"], s["params"], s["samples"],
                          s["g_cd"], s["g_cs"], s["g_verts"])
    return dict(records=s["edges"].records, count=s["edges"].count, g_verts=s["g_verts"])


# ------------------------------------------------------------------ work
def _mesh_bytes(case):
    """Vertices with normals and index triples of about 11.7 grid^2 triangles (half as many vertices)."""
    t = 11.7 * case["grid"] ** 2 * (1.6 if case["boxes"] > 8 else 1.0)
    return t * (12 + 0.5 * 24)


def work(case):
    kind = case["kind"]
    if kind == "denoise":
        px = case["images"] * case["height"] * case["width"]
        passes = 3 if case["train"] else 2
        return {"bytes": px * (4 * 16 + 16), "flops": passes * UNET_FLOPS * px}
    px = case.get("views", 1) * case.get("height", case.get("res")) * case.get("width", case.get("res"))
    env = case.get("env", 0) ** 2 / 2 * 16
    if kind == "render":
        return {"bytes": _mesh_bytes(case) + 32 * case["tex"] ** 2 + env + 16 * px,
                "flops": px * (case["spp"] * SAMPLE_FLOPS + 2 * UNET_FLOPS)}
    if kind == "step":
        net = {"bf16": 4 * UNET_FLOPS, "e4m3": 4 * UNET_FLOPS, "bilateral": 4 * 81 * 20, "none": 0}[case["denoiser"]]
        return {"bytes": _mesh_bytes(case) + 32 * case["tex"] ** 2 + 2 * env + 16 * px * 8,
                "flops": px * (case["spp"] * 2.5 * SAMPLE_FLOPS + net)}
    if kind == "shade":  # a G-buffer, three gradients in; three terms, three gradients out
        return {"bytes": 16 * px * (4 + 3 + 3 + 3) + 2 * env, "flops": px * case["spp"] * 2.5 * SAMPLE_FLOPS}
    if kind == "cast":
        return {"bytes": _mesh_bytes(case) + 32 * case["tex"] ** 2 + 64 * px, "flops": px * 20 * 52}
    if kind == "bilateral":
        taps = (2 * math.ceil(2 * case["sigma"]) + 1) ** 2
        return {"bytes": 16 * px * (3 + 2 + 1 + 2 + 1 + 1 + 2), "flops": px * taps * 2 * 40}
    return {"bytes": 2 * _mesh_bytes(case) + 11.7 * case["grid"] ** 2 * 1.5 * 16 + 16 * px * 6 + env,
            "flops": px * case["samples"] * 60}


# ------------------------------------------------------------------ exact
def exact(case, seed):
    """In 64 bits, where plain tensor code gives it: the network's forward in BF16 (the gradients and E4M3 lie too
    far from an unquantised network to say anything) and the bilateral filter with its loss and gradients.  The
    Monte Carlo cases take discrete decisions (texels, shadow rays against every triangle) that 64 bits takes
    differently, or that would take minutes by testing all pairs."""
    if case["kind"] == "denoise" and case["precision"] == "bf16":
        s = prepare(case, seed)
        return dict(y=_exact_unet(s, _unet(int(seed))), gx=None, gw=None)
    if case["kind"] == "bilateral":
        return _exact_bilateral(prepare(case, seed))
    return None


def _exact_unet(s, flat):
    w = {k: (torch.as_tensor(a, device=DEV).double(), torch.as_tensor(b, device=DEV).double())
         for k, (a, b) in mcdi.unflatten_unet_params(flat).items()}
    conv = lambda k, x, relu=True: F.relu(F.conv2d(x, *w[k], padding=1)) if relu else F.conv2d(x, *w[k], padding=1)
    up = lambda x: F.interpolate(x, scale_factor=2, mode="nearest")
    out = []
    term, kd, nrm = s["term"].detach(), s["kd"], s["nrm"]
    for i in range(term.shape[0]):
        a = i % kd.shape[0]
        x = torch.cat([term[i, ..., :3], kd[a, ..., :3], nrm[a, ..., :3]], -1).double().permute(2, 0, 1)[None]
        e1 = conv("enc1b", conv("enc1a", x))
        e2 = conv("enc2b", conv("enc2a", F.max_pool2d(e1, 2)))
        e3 = conv("enc3b", conv("enc3a", F.max_pool2d(e2, 2)))
        b = conv("bot_b", conv("bot_a", F.max_pool2d(e3, 2)))
        d = conv("dec3b", conv("dec3a", torch.cat([up(b), e3], 1)))
        d = conv("dec2b", conv("dec2a", torch.cat([up(d), e2], 1)))
        d = conv("dec1b", conv("dec1a", torch.cat([up(d), e1], 1)))
        out.append(F.pad(conv("out", d, False)[0].permute(1, 2, 0), (0, 1)))
    return torch.stack(out)


def _shift(t, dy, dx, fill=0.0):
    """t[..., y + dy, x + dx], `fill` outside; t is (N, H, W)."""
    r = max(abs(dy), abs(dx))
    p = F.pad(t, (r, r, r, r), value=fill)
    return p[:, r + dy:r + dy + t.shape[1], r + dx:r + dx + t.shape[2]]


def _exact_bilateral(s):
    gb, sigma = s["gb"], s["sigma"]
    n, h, w = gb.pos.shape[:3]
    cams = s["cams"].double()
    pos, nrm = gb.pos.double(), F.normalize(gb.nrm[..., :3].double(), dim=-1)
    cov = gb.pos[..., 3] > 0
    z = ((pos[..., :3] - cams[:, None, None, 0:3]) * cams[:, None, None, 9:12]).sum(-1)
    c1 = cov.double()

    def slope(dy, dx):
        zp, zm = _shift(z, dy, dx), _shift(z, -dy, -dx)
        cp, cm = _shift(c1, dy, dx) > 0, _shift(c1, -dy, -dx) > 0
        one = torch.where(cp, zp - z, torch.where(cm, z - zm, torch.zeros_like(z)))
        return torch.where(cp & cm, 0.5 * (zp - zm), one)

    gx, gy, R = slope(0, 1), slope(1, 0), math.ceil(2 * sigma)
    planes = s["terms"][..., :3].double().requires_grad_()
    src = planes.reshape(2, n, h, w, 3)
    acc, wsum = torch.zeros_like(src), torch.zeros_like(z)
    for dy in range(-R, R + 1):
        for dx in range(-R, R + 1):
            both = cov & (_shift(c1, dy, dx) > 0)
            nn = sum(nrm[..., k] * _shift(nrm[..., k], dy, dx) for k in range(3)).clamp_min(0)
            den = (gx * dx + gy * dy).abs() + 1e-3 * z.abs()
            wt = math.exp(-(dx * dx + dy * dy) / (2 * sigma * sigma)) * nn ** 128
            wt = wt * torch.exp(-(z - _shift(z, dy, dx)).abs() / torch.where(both, den, torch.ones_like(den)))
            wt = torch.where(both, wt, torch.zeros_like(wt))
            wsum = wsum + wt
            moved = torch.stack([_shift(src[..., k].reshape(2 * n, h, w), dy, dx) for k in range(3)], -1)
            acc = acc + wt[None, ..., None] * moved.reshape_as(src)
    safe = torch.where(cov, wsum, torch.ones_like(wsum))[None, ..., None]
    den = torch.where(cov[None, ..., None], acc / safe, src)
    kd = gb.kd[..., :3].double().requires_grad_()
    ref = s["ref"][..., :3].double()

    def tone(x):
        y = torch.log1p(x.clamp_min(0))
        return torch.where(y <= 0.0031308, 12.92 * y, 1.055 * y.clamp_min(0.0031308) ** (1 / 2.4) - 0.055)

    color = kd * den[0] + den[1]
    img = (tone(color) - tone(ref)).abs().mean()
    light = (tone(den[0] + den[1]).mean(-1) - tone(ref).amax(-1)).abs().mean()
    loss = img + 0.15 * light
    g_kd, g_terms = torch.autograd.grad(loss, [kd, planes])
    four = lambda t: F.pad(t.detach(), (0, 1))
    return dict(den=four(den.reshape(2 * n, h, w, 3)), wsum=wsum, color=four(color),
                loss=torch.stack([loss, img, light]).detach(), g_kd=four(g_kd), g_terms=four(g_terms))
