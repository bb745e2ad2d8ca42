"""Sample generation is compiled for small and for large grids: a pixel's terms
and visibility bits are the same in either.  A pixel's samples depend on its index
in its view, so the first rows of a tall image are those of a low one."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,low,tall,spp", [(160, 16, 1200, (3, 2, 2)), (333, 5, 640, (8, 4, 4))])
def test_low_and_tall_images_agree(cuda_lib, orc, W, low, tall, spp):
    mcdi = cuda_lib
    sc = scenes.parity_scene()
    rows = orc.primary_cast(sc.verts, sc.vnrm, sc.tris, sc.cams[0], sc.width, sc.height,
                            np.arange(sc.width * sc.height), sc.tex_kd, sc.tex_korm, sc.uvmap).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    bvh = mcdi.Bvh.allocate(len(sc.tris)).build(t(sc.verts), t(sc.tris))
    env = t(np.concatenate([sc.env, np.zeros(sc.env.shape[:2] + (1,), np.float32)], -1) if sc.env.shape[-1] == 3 else sc.env)
    probe = mcdi.Probe.allocate(env).build()
    prm = mcdi.make_params(*spp, seed=5, tau=0.6)
    out = []
    for H in (low, tall):
        g = t(rows[np.arange(H * W) * 7 % len(rows)]).reshape(1, H, W, 16)
        gb = mcdi.GBuffer(*(g[..., 4 * k:4 * k + 4].contiguous() for k in range(4)))
        cd, kd, cs = (torch.full((1, H, W, 4), float("nan"), device="cuda") for _ in range(3))
        mask = torch.full((1, H, W, 1), -1, dtype=torch.int32, device="cuda")
        ws = mcdi._empty_bytes(mcdi.shade_workspace_size(1, H, W, prm), "cuda")
        mcdi.shade_mc_fwd(bvh, probe, gb, t(sc.cams[:1]), prm, cd, kd, cs, mask, ws)
        torch.cuda.synchronize()
        out.append([x[:, :low].cpu().numpy() for x in (cd, kd, cs, mask)])
    for a, b in zip(*out):
        assert np.array_equal(a, b)
    assert np.isfinite(out[0][0]).all() and (out[0][0] > 0).any() and (out[0][3] != 0).any()
