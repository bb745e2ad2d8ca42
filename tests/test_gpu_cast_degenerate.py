"""Cameras whose rays are not finite see nothing: a basis of zeros (its direction
is 0 / 0), NaN or infinite entries, a basis so short that its square is zero.
Meshes of a few triangles, whose four-wide nodes have empty slots, and one with
many nodes; the view beside it in the same launch is not disturbed."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu


def cameras():
    """(name, camera): origin, right, up, forward, aspect, tan."""
    ok = scenes.look_at((0.1, 0.4, 3.2), (0, 0, 0), (0, 1, 0), 40.0, 1.25).astype(np.float32)
    out = []
    for name, at, value in (("zero basis", slice(3, 12), 0.0), ("nan forward", slice(9, 12), np.nan),
                            ("nan right.x", slice(3, 4), np.nan), ("nan origin", slice(0, 3), np.nan),
                            ("nan origin.y", slice(1, 2), np.nan), ("infinite origin", slice(0, 3), -np.inf),
                            ("infinite forward.z", slice(11, 12), np.inf), ("tiny basis", slice(3, 12), 1e-30)):
        c = ok.copy()
        c[at] = value
        out.append((name, c))
    return ok, out


@pytest.mark.parametrize("n", [1, 2, 3, 5, 200])
def test_a_camera_without_finite_rays_sees_nothing(cuda_lib, orc, n):
    mcdi = cuda_lib
    sc = scenes.parity_scene()
    rng = np.random.default_rng(n)
    centre = rng.uniform(-0.5, 0.5, (n, 1, 3))
    verts = (centre + rng.normal(0, 0.4, (n, 3, 3))).reshape(-1, 3).astype(np.float32)
    tris = np.arange(3 * n, dtype=np.int32).reshape(-1, 3)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pad = lambda a: t(np.concatenate([a, np.zeros(a.shape[:2] + (1,), np.float32)], -1)) if a.shape[-1] == 3 else t(a)
    bvh = mcdi.Bvh.allocate(n).build(t(verts), t(tris))
    H, W = 16, 20
    good, bad = cameras()

    def cast(cams):
        gb = mcdi.GBuffer.allocate(len(cams), H, W)
        for p in (gb.pos, gb.nrm, gb.kd, gb.korm):
            p.fill_(7.0)
        mcdi.primary_cast(bvh, t(verts), t(np.ones_like(verts)), t(tris), t(np.stack(cams)), H, W, pad(sc.tex_kd),
                          pad(sc.tex_korm), sc.uvmap, gb)
        torch.cuda.synchronize()
        return torch.cat([gb.pos, gb.nrm, gb.kd, gb.korm], -1)

    alone = cast([good])[0]
    seen = orc.primary_cast(verts, np.ones_like(verts), tris, good, W, H, np.arange(H * W), sc.tex_kd, sc.tex_korm,
                            sc.uvmap)[:, 3] > 0
    assert ((alone[..., 3].cpu().numpy().reshape(-1) > 0) != seen).sum() <= 1
    for name, c in bad:
        both = cast([c, good])
        assert (both[0] == 0).all(), name
        assert torch.equal(both[1], alone), name
