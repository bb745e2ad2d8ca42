"""Shadow rays from origins far outside the mesh, where the rounding of slab
distances outgrows the margin of the four-wide nodes' quantised boxes, and
against meshes whose bounds are infinite: decided as the oracle decides them,
respectively as without the infinite triangle, by every kernel that traces."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes
from tests import parity_util as PU
from tests.test_gpu_shadow_grad import ETA, _parity_case

pytestmark = pytest.mark.gpu


def _pipe(sc, planes, wavefront):
    from paper_2206_03380_gb300.pipeline import ShadingPipeline

    pipe = ShadingPipeline(sc, wavefront=wavefront)
    for dst, src in zip((pipe.gb.pos, pipe.gb.nrm, pipe.gb.kd, pipe.gb.korm), planes):
        dst.copy_(torch.from_numpy(src))
    pipe.build_probe()
    pipe.build_bvh()
    pipe.forward()
    torch.cuda.synchronize()
    return pipe


def _retraced_gradients(mcdi, pipe, mask, g):
    out = [torch.zeros_like(pipe.gb.pos) for _ in range(3)]
    mcdi.shade_mc_bwd(pipe.bvh, pipe.probe, pipe.gb, pipe.cams, pipe.params, *g, mask, *out, torch.zeros_like(pipe.env))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("dist,env_w", [(8.0, 32), (100.0, 256), (2000.0, 4096)])
def test_distant_pixels_match_oracle(cuda_lib, orc, dist, env_w):
    """A patch of 18,432 small triangles, pixels `dist` away from it, a probe lit in the one texel behind it."""
    n, H, W = 96, 24, 32
    rng = np.random.default_rng(int(dist))
    u = np.linspace(-1, 1, n + 1)
    X, Y = np.meshgrid(u, u)
    a = np.array([0.48, 0.6, 0.64])  # the patch's normal, no axis of it small
    b1 = np.cross(a, [0, 0, 1.0])
    b1 /= np.linalg.norm(b1)
    b2 = np.cross(a, b1)
    verts = (X[..., None] * b1 + Y[..., None] * b2 + rng.uniform(-0.02, 0.02, X.shape)[..., None] * a).reshape(-1, 3)
    k = (np.arange(n)[:, None] * (n + 1) + np.arange(n)).reshape(-1)
    tris = np.concatenate([np.stack([k, k + 1, k + n + 2], 1), np.stack([k, k + n + 2, k + n + 1], 1)]).astype(np.int32)
    env = np.zeros((env_w // 2, env_w, 4), np.float32)
    j, i = int(np.arccos(-a[1]) / np.pi * (env_w // 2)), int(np.arctan2(-a[2], -a[0]) / (2 * np.pi) % 1 * env_w)
    env[j, i, :3] = 1.0
    th, ph = np.pi * (j + 0.5) / (env_w // 2), 2 * np.pi * (i + 0.5) / env_w
    d = np.array([np.sin(th) * np.cos(ph), np.cos(th), np.sin(th) * np.sin(ph)])  # towards the lit texel
    base = scenes.parity_scene()
    sc = scenes.Scene(**{**base.__dict__, "verts": verts.astype(np.float32), "vnrm": np.ones_like(verts, np.float32),
                         "tris": tris, "env": env, "width": W, "height": H, "n_light": 4, "n_cos": 0, "n_ggx": 0})
    planes = [np.zeros((1, H, W, 4), np.float32) for _ in range(4)]
    planes[0][..., :3] = -dist * d + rng.uniform(-0.3, 0.3, (1, H, W, 3))
    planes[0][..., 3] = 1
    planes[1][..., :3] = d
    planes[2][..., :3] = 0.5
    planes[3][..., 1] = 0.5
    rows = np.concatenate(planes, -1).reshape(-1, 16)
    _, vis, recs = PU.oracle_shade(orc, sc, rows, np.arange(H * W), 0)
    want = PU.mask_bits(vis, 4)
    assert 0.1 < want.mean() < 0.99 and (recs["active"] != 0).all()
    pipes = [_pipe(sc, planes, wavefront) for wavefront in (True, False)]
    for pipe in pipes:
        got = PU.mask_bits(pipe.mask.cpu().numpy().reshape(H * W, -1), 4)
        # rays that pass the patch's rim within the rounding of their coordinates go either way
        assert (got != want).mean() <= 0.005, (got != want).mean()
    g = [torch.randn(planes[0].shape, device="cuda") for _ in range(3)]
    fed, traced = (_retraced_gradients(cuda_lib, pipes[0], m, g) for m in (pipes[0].mask, None))
    assert all(torch.equal(x, y) for x, y in zip(fed, traced))
    st = torch.zeros(5, dtype=torch.int64, device="cuda")
    cuda_lib.shadow_ray_stats(pipes[0].bvh, 1, H, W, pipes[0].params, pipes[0].workspace, st)
    assert int(st[0]) == H * W * 4 and int(st[4]) == 0


def _with_infinite(verts, tris, bad):
    far = np.array([[5.0, 5.0, 9.0], [5.0, 6.0, 9.0], bad], np.float32)
    extra = np.array([[len(verts), len(verts) + 1, len(verts) + 2]], np.int32)
    return np.concatenate([verts, far]).astype(np.float32), np.concatenate([tris, extra]).astype(np.int32)


@pytest.mark.parametrize("n", [3, 600])
@pytest.mark.parametrize("bad", [(np.inf, 0.0, 0.0), (0.0, -np.inf, 3e38)])
def test_an_infinite_vertex_hides_no_triangle(cuda_lib, n, bad):
    H, W = 12, 20
    rng = np.random.default_rng(n)
    verts = (rng.uniform(-0.8, 0.8, (n, 1, 3)) + rng.normal(0, 0.2, (n, 3, 3))).reshape(-1, 3).astype(np.float32)
    tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    planes = [rng.uniform(lo, 0.9, (1, H, W, 4)).astype(np.float32) for lo in (-0.9, -1, 0.1, 0.1)]
    planes[0][..., 3] = 1
    base = scenes.parity_scene()
    kw = {"width": W, "height": H, "n_light": 8, "n_cos": 4, "n_ggx": 4}
    sc = [scenes.Scene(**{**base.__dict__, **kw, "verts": v, "vnrm": np.ones_like(v), "tris": t})
          for v, t in ((verts, tris), _with_infinite(verts, tris, bad))]
    g = [torch.randn((1, H, W, 4), device="cuda") for _ in range(3)]
    for wavefront in (True, False):
        plain, both = (_pipe(s, planes, wavefront) for s in sc)
        assert (plain.mask != 0).any()
        assert torch.equal(both.mask, plain.mask)
    fed, traced = (_retraced_gradients(cuda_lib, p, m, g) for p, m in ((plain, plain.mask), (both, None)))
    assert all(torch.equal(x, y) for x, y in zip(fed, traced))


@pytest.mark.parametrize("bad", [(np.inf, 0.0, 0.0)])
def test_an_infinite_vertex_opens_no_edge_sample(cuda_lib, orc, bad):
    mcdi = cuda_lib
    sc, pipe, rows, prm = _parity_case(mcdi, orc, 0.7)
    W, H, M = sc.width, sc.height, 16
    verts, tris = _with_infinite(sc.verts, sc.tris, bad)
    edges = orc.edge_table(sc.tris)
    et = mcdi.EdgeTable.allocate(len(sc.tris), "cuda")
    et.records[:len(edges)].copy_(torch.from_numpy(edges.astype(np.int32)))
    et.count.fill_(len(edges))
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    gen = torch.Generator(device="cuda").manual_seed(3)
    gc = [torch.randn((1, H, W, 4), generator=gen, device="cuda") for _ in range(2)]
    out = []
    for v, tr in ((sc.verts, sc.tris), (verts, tris)):
        bvh = mcdi.Bvh.allocate(len(tr)).build(t(v), t(tr))
        w = torch.full((H * W, M), float("nan"), device="cuda")
        mcdi.shadow_edge_grad(bvh, t(v), et, pipe.probe, pipe.gb, pipe.cams, prm, M, *gc,
                              torch.zeros((len(v), 3), device="cuda"), w, eta=ETA)
        out.append(w)
    torch.cuda.synchronize()
    assert (out[0] != 0).any() and torch.equal(out[0], out[1])
