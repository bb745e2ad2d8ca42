"""The wavefront's shadow-ray tracer at the sizes where its bookkeeping can go
wrong: meshes of a few triangles, meshes whose boxes all overlap (every child
of every node is hit, so a lane's node stack outgrows its 20 entries and its
leaf queue of 8 fills), many rays per lane and fewer rays than lanes.  A ray is
blocked or not by the OR of its triangle tests, so the visibility masks must
equal, bit for bit, those of the kernel without scratch memory (which traces
its pixels' rays in chunks of 16 samples) and of the counting re-trace; and the
adjoint that traces the rays again must equal, bit for bit, the one given the
forward's mask.  The tallest probe makes those kernels ask for more than the
default shared memory."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu


def slivers(n, rng):
    """n long thin triangles across the cube [-1, 1]^3: overlapping boxes, few hits."""
    a, b = rng.uniform(-1, 1, (n, 3)), rng.uniform(-1, 1, (n, 3))
    v = np.stack([a, a + rng.normal(0, 2e-4, (n, 3)), b], 1).reshape(-1, 3)
    return v.astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


def soup(n, rng):
    c = rng.uniform(-1, 1, (n, 1, 3))
    v = (c + rng.normal(0, 0.08, (n, 3, 3))).reshape(-1, 3)
    return v.astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(-1, 3)


def tall_probe(rng):
    env = np.exp(rng.normal(size=(4096, 8, 4))).astype(np.float32)
    env[..., 3] = 0
    return env


@pytest.mark.parametrize("kind,n,size,split", [
    ("slivers", 1, (5, 3), (1, 1, 1)), ("slivers", 2, (33, 7), (4, 2, 2)), ("slivers", 5, (16, 16), (8, 4, 4)),
    ("slivers", 4000, (37, 23), (8, 4, 4)), ("slivers", 20000, (9, 2), (3, 1, 1)),
    ("soup", 17, (37, 23), (20, 10, 9)), ("soup", 3000, (131, 77), (8, 4, 4)), ("soup", 3000, (64, 64), (1, 0, 0)),
    ("soup tall probe", 300, (33, 5), (9, 4, 4)),
])
def test_tracer_equals_fused_kernel(cuda_lib, kind, n, size, split):
    from paper_2206_03380_gb300.pipeline import ShadingPipeline

    rng = np.random.default_rng(n + size[0])
    v, t = (slivers if kind == "slivers" else soup)(n, rng)
    tall = "tall" in kind
    base = scenes.parity_scene()
    W, H = size
    sc = scenes.Scene(**{**base.__dict__, "verts": v, "vnrm": np.zeros_like(v), "tris": t, "width": W, "height": H,
                         "n_light": split[0], "n_cos": split[1], "n_ggx": split[2]})
    if tall:
        sc.env = tall_probe(rng)
    masks, rays = [], None
    pos = rng.uniform(-0.9, 0.9, (1, H, W, 4)).astype(np.float32)
    pos[..., 3] = rng.random((1, H, W)) < 0.8  # some uncovered pixels
    nrm = rng.normal(size=(1, H, W, 4)).astype(np.float32)
    mat = rng.uniform(0.1, 0.9, (2, 1, H, W, 4)).astype(np.float32)
    for wavefront in (True, False):
        pipe = ShadingPipeline(sc, wavefront=wavefront)
        for dst, src in zip((pipe.gb.pos, pipe.gb.nrm, pipe.gb.kd, pipe.gb.korm), (pos, nrm, mat[0], mat[1])):
            dst.copy_(torch.from_numpy(src))
        pipe.build_probe()
        pipe.build_bvh()
        pipe.forward()
        torch.cuda.synchronize()
        masks.append(pipe.mask.clone())
        if wavefront:
            st = torch.zeros(5, dtype=torch.int64, device="cuda")
            cuda_lib.shadow_ray_stats(pipe.bvh, 1, H, W, pipe.params, pipe.workspace, st)
            rays = [int(x) for x in st]
            g = [torch.randn_like(pipe.gb.pos) for _ in range(3)]
            got = []
            for m in (pipe.mask, None):
                out = [torch.zeros_like(pipe.gb.pos) for _ in range(3)]
                cuda_lib.shade_mc_bwd(pipe.bvh, pipe.probe, pipe.gb, pipe.cams, pipe.params, *g, m, *out,
                                      torch.zeros_like(pipe.env))
                got.append(out)
            assert all(torch.equal(a, b) for a, b in zip(*got))
    assert torch.equal(masks[0], masks[1])
    assert rays[0] > 0 and rays[4] == 0
