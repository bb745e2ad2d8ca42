"""G-buffer pixels whose positions are infinite or NaN: their shadow rays meet
every box of a tree, empty slots among them, and no triangle."""
import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu

W, H = 24, 12
VALUES = [(-np.inf,) * 3, (np.inf,) * 3, (np.nan,) * 3, (np.inf, -np.inf, 0.5), (0.1, -np.inf, 0.2), (np.nan, 0, 0)]
BAD_ROWS = [2 * k for k in range(len(VALUES))]


def _shade(n, wavefront, bad):
    """The pipeline after a forward pass over n random triangles, every second row of pixels at one of VALUES."""
    from paper_2206_03380_gb300.pipeline import ShadingPipeline

    rng = np.random.default_rng(50 + n)
    verts = (rng.uniform(-0.5, 0.5, (n, 1, 3)) + rng.normal(0, 0.4, (n, 3, 3))).reshape(-1, 3).astype(np.float32)
    base = scenes.parity_scene()
    sc = scenes.Scene(**{**base.__dict__, "verts": verts, "vnrm": np.ones_like(verts), "width": W, "height": H,
                         "tris": np.arange(3 * n, dtype=np.int32).reshape(-1, 3), "n_light": 6, "n_cos": 3, "n_ggx": 2})
    pos = rng.uniform(-0.9, 0.9, (1, H, W, 4)).astype(np.float32)
    pos[..., 3] = 1
    nrm, kd, korm = (rng.uniform(lo, 1, (1, H, W, 4)).astype(np.float32) for lo in (-1, 0, 0.1))
    if bad:
        for y, v in zip(BAD_ROWS, VALUES):
            pos[0, y, :, :3] = v
    pipe = ShadingPipeline(sc, wavefront=wavefront)
    for dst, src in zip((pipe.gb.pos, pipe.gb.nrm, pipe.gb.kd, pipe.gb.korm), (pos, nrm, kd, korm)):
        dst.copy_(torch.from_numpy(src))
    pipe.build_probe()
    pipe.build_bvh()
    pipe.forward()
    torch.cuda.synchronize()
    return pipe


@pytest.mark.parametrize("n", [1, 2, 3, 5, 40])
def test_counting_retrace_tests_no_empty_slot(cuda_lib, n):
    pipe = _shade(n, True, True)
    st = torch.zeros(5, dtype=torch.int64, device="cuda")
    cuda_lib.shadow_ray_stats(pipe.bvh, 1, H, W, pipe.params, pipe.workspace, st)
    rays, _, tests, _, differ = (int(x) for x in st)
    assert rays > 0 and differ == 0
    assert tests <= rays * n  # a ray tests each triangle at most once
