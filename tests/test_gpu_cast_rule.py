"""Where the ray cast may use the four-wide nodes' quantised boxes: cameras just
inside and outside the distance up to which their margin covers the rounding,
and meshes whose bounds are infinite or too large for their steps."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu

H, W = 24, 32


def _cast(mcdi, sc, verts, tris, cam):
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pad = lambda a: t(np.concatenate([a, np.zeros(a.shape[:2] + (1,), np.float32)], -1)) if a.shape[-1] == 3 else t(a)
    vnrm = np.tile(np.array([[0, 0, 1]], np.float32), (len(verts), 1))
    bvh = mcdi.Bvh.allocate(len(tris)).build(t(verts), t(tris))
    gb = mcdi.GBuffer.allocate(1, H, W)
    for p in (gb.pos, gb.nrm, gb.kd, gb.korm):
        p.fill_(float("nan"))
    mcdi.primary_cast(bvh, t(verts), t(vnrm), t(tris), t(cam[None]), H, W, pad(sc.tex_kd), pad(sc.tex_korm), sc.uvmap,
                      gb)
    torch.cuda.synchronize()
    return np.concatenate([x.cpu().numpy() for x in (gb.pos, gb.nrm, gb.kd, gb.korm)], -1).reshape(-1, 16)


@pytest.mark.parametrize("n", [2, 7, 1500])
@pytest.mark.parametrize("bad", [(np.inf, 0.0, 0.0), (0.0, -np.inf, 3e38), (3e38, -3e38, 3e38), (1e20, 0.0, 1e20)])
def test_one_far_vertex_hides_nothing(cuda_lib, n, bad):
    """A triangle with an infinite or very far vertex, pointing away from the view, leaves the others' pixels as they
    are without it."""
    rng = np.random.default_rng(n)
    sc = scenes.parity_scene()
    verts = (rng.uniform(-0.6, 0.6, (n, 1, 3)) + rng.normal(0, 0.25, (n, 3, 3))).reshape(-1, 3).astype(np.float32)
    tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    cam = scenes.look_at((0.1, 0.4, 3.2), (0, 0, 0), (0, 1, 0), 30.0, W / H).astype(np.float32)
    plain = _cast(cuda_lib, sc, verts, tris, cam)
    assert (plain[:, 3] > 0).any()
    far = np.array([[5.0, 5.0, 9.0], [5.0, 6.0, 9.0], bad], np.float32)  # behind the camera but for the last vertex
    both = _cast(cuda_lib, sc, np.concatenate([verts, far]), np.concatenate([tris, [[3 * n, 3 * n + 1, 3 * n + 2]]]).astype(np.int32), cam)
    seen = (plain[:, 3] > 0) & (both[:, 3] > 0) & (np.abs(both[:, :3]).max(1) < 10)
    assert seen.sum() >= 0.9 * (plain[:, 3] > 0).sum()
    # (equal distances on shared edges may be met in another order)
    assert (np.abs(both[seen] - plain[seen]).max(1) > 1e-5).sum() <= 1


@pytest.mark.parametrize("far", [10.0, 10.99, 11.01, 15.9, 16.1, 60.0])
def test_cameras_around_the_distance_line(cuda_lib, orc, far):
    """far: the largest coordinate of the eye, in units of the mesh's."""
    sc = scenes.parity_scene()
    m = float(np.abs(sc.verts).max())
    eye = np.array([0.2, 0.62, 1.0]) * far * m
    cam = scenes.look_at(tuple(eye), (0, -0.2, 0), (0, 1, 0), np.degrees(2.4 / np.linalg.norm(eye)), W / H).astype(np.float32)
    g = _cast(cuda_lib, sc, sc.verts, sc.tris, cam)
    o = orc.primary_cast(sc.verts, np.tile(np.array([[0, 0, 1]], np.float32), (len(sc.verts), 1)), sc.tris, cam, W, H,
                         np.arange(H * W), sc.tex_kd, sc.tex_korm, sc.uvmap)
    # a hit's distance comes from differences of coordinates as large as the eye's, a few ulps of it, and moves the
    # point by that over the cosine of the angle it is seen under; the triangles' edges by as much
    both = (g[:, 3] > 0) & (o[:, 3] > 0)
    assert ((g[:, 3] > 0) != (o[:, 3] > 0)).sum() <= 3 and both.sum() > H * W // 2
    tol = 64 * 2.0 ** -24 * np.linalg.norm(eye)
    off = np.abs(g[:, :3] - o[:, :3]).max(1) > 10 * tol
    assert (both & off).sum() <= 0.02 * both.sum() + 3


def test_far_cameras_of_large_and_small_images(cuda_lib):
    """A ray per lane in one tile per CTA (few pixels) and in two (many), with an odd number of tiles per view: the
    same pixels, all of them."""
    sc = scenes.parity_scene()
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pad = lambda a: t(np.concatenate([a, np.zeros(a.shape[:2] + (1,), np.float32)], -1)) if a.shape[-1] == 3 else t(a)
    eye = np.array([0.2, 0.62, 1.0]) * 20 * float(np.abs(sc.verts).max())
    verts, vnrm, tris, kd, korm = t(sc.verts), t(sc.vnrm), t(sc.tris), pad(sc.tex_kd), pad(sc.tex_korm)
    bvh = cuda_lib.Bvh.allocate(len(sc.tris)).build(verts, tris)
    cam = scenes.look_at(tuple(eye), (0, -0.2, 0), (0, 1, 0), np.degrees(2.4 / np.linalg.norm(eye)), 1.0).astype(np.float32)

    def cast(views, h, w):
        gb = cuda_lib.GBuffer.allocate(views, h, w)
        for p in (gb.pos, gb.nrm, gb.kd, gb.korm):
            p.fill_(float("nan"))
        cuda_lib.primary_cast(bvh, verts, vnrm, tris, t(np.stack([cam] * views)), h, w, kd, korm, sc.uvmap, gb)
        torch.cuda.synchronize()
        return torch.cat([gb.pos, gb.nrm, gb.kd, gb.korm], -1)

    one = cast(1, 99, 71)  # 13 x 9 tiles of 8 x 8
    many = cast(41, 99, 71)  # the same view, in enough CTAs to join tiles
    assert torch.isfinite(one).all() and (one[..., 3] > 0).float().mean() > 0.5
    assert torch.equal(many, one.expand_as(many))
