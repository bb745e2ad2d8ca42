"""The ray-cast G-buffer at the edges of its tiles and of its rules, against the
oracle: images narrower or lower than a warp's pixels, one triangle, a camera too
far away for the four-wide nodes' quantised boxes (the two-child tree decides),
and a tree so deep and overlapping that a ray has more pending nodes than its
row of shared memory holds."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu


def _deep_mesh():
    """Four wide triangles at each of 30 heights whose Morton codes have one bit each: the tree is a chain of
    30 overlapping nodes with an inner sibling at every level; all of them in front of the camera."""
    v, t = [], []
    for j in range(30):
        c = np.zeros(3)
        c[j % 3] = 2.0 ** -(1 + j // 3)
        for k in range(4):
            z = c[2] + 1e-5 * (4 * j + k)
            # centroid (c.x, c.y, z), all corners at height z
            base = np.array([[-9.0, -6.0], [9.0, -6.0], [0.0, 12.0]]) + c[:2]
            t.append([len(v), len(v) + 1, len(v) + 2])
            v.extend([[x, y, z] for x, y in base])
    # two small triangles that pin the centroid bounds to [0, 1]^3, out of sight
    for c in ((0.0, 0.0, 0.0), (1.0, 1.0, 1.0)):
        t.append([len(v), len(v) + 1, len(v) + 2])
        v.extend([[c[0] + dx, c[1] + dy, c[2]] for dx, dy in ((-1e-4, -1e-4), (1e-4, -1e-4), (0, 2e-4))])
    return np.array(v, np.float32), np.array(t, np.int32)


@pytest.mark.parametrize("kind,H,W", [("mesh", 1, 1), ("mesh", 1, 40), ("mesh", 40, 1), ("mesh", 2, 37), ("mesh", 37, 3),
                                      ("mesh", 9, 9), ("mesh", 33, 65), ("far", 24, 24), ("single", 9, 17),
                                      ("deep", 16, 24)])
def test_matches_oracle(cuda_lib, orc, kind, H, W):
    mcdi = cuda_lib
    sc = scenes.parity_scene()
    verts, vnrm, tris = sc.verts, sc.vnrm, sc.tris
    eye, target, up, fov = (0.1, 0.4, 3.2), (0, 0, 0), (0, 1, 0), 40.0 * H / max(H, W)
    tol = 2e-5
    if kind == "far":  # beyond 16 times the largest coordinate (8)
        eye, fov = (20.0, 90.0, 140.0), 1.0
    elif kind == "single":
        verts = np.array([[-1, -1, 0], [1, -1, 0.2], [0, 1, -0.3]], np.float32)
        tris = np.array([[0, 1, 2]], np.int32)
    elif kind == "deep":
        verts, tris = _deep_mesh()
        eye, target, fov = (0.3, 0.2, -4.0), (0.3, 0.2, 0.0), 50.0  # the chain is nearest, its siblings pending
    if kind in ("single", "deep"):
        vnrm = np.tile(np.array([[0, 0, 1]], np.float32), (len(verts), 1))
    cam = scenes.look_at(eye, target, up, fov, W / H).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pad = lambda a: t(np.concatenate([a, np.zeros(a.shape[:2] + (1,), np.float32)], -1)) if a.shape[-1] == 3 else t(a)
    bvh = mcdi.Bvh.allocate(len(tris)).build(t(verts), t(tris))
    gb = mcdi.GBuffer.allocate(1, H, W)
    for p in (gb.pos, gb.nrm, gb.kd, gb.korm):
        p.fill_(float("nan"))
    mcdi.primary_cast(bvh, t(verts), t(vnrm), t(tris), t(cam[None]), H, W, pad(sc.tex_kd), pad(sc.tex_korm), sc.uvmap,
                      gb)
    torch.cuda.synchronize()
    g = np.concatenate([x.cpu().numpy() for x in (gb.pos, gb.nrm, gb.kd, gb.korm)], -1).reshape(-1, 16)
    o = orc.primary_cast(verts, vnrm, tris, cam, W, H, np.arange(H * W), sc.tex_kd, sc.tex_korm, sc.uvmap)
    assert np.isfinite(g).all()
    cov = (g[:, 3] > 0) != (o[:, 3] > 0)
    both = (g[:, 3] > 0) & (o[:, 3] > 0)
    if kind == "far":
        # the hit's distance comes from differences of coordinates as large as the origin's, a few ulps of it,
        # and moves the point by that over the cosine of the angle it is seen under
        d = o[:, :3] - np.array(eye)
        cos = np.abs((o[:, 4:7] * d).sum(1)) / np.linalg.norm(d, axis=1)
        tol = (16 * 2.0 ** -24 * np.linalg.norm(eye) / np.maximum(cos, 1e-2))[:, None]
    else:
        tol = np.full((H * W, 1), tol)
    off = (np.abs(g[:, :3] - o[:, :3]) > 5 * tol).any(1)
    assert cov.sum() <= 3 and (both & off).sum() <= 3, (cov.sum(), (both & off).sum())
    ok = both & ~off
    assert ok.sum() >= (1 if H * W == 1 else H * W // 8)
    assert np.all(np.abs(g[ok, :3] - o[ok, :3]) <= tol[ok])
    if kind != "far":
        np.testing.assert_allclose(g[ok, 4:7], o[ok, 4:7], atol=2e-5)
    assert np.all(g[g[:, 3] == 0] == 0)
