"""The bilateral filter's tiles at their edges against the oracle: image sizes
around the 32-pixel tile and its rows, radii on both sides of the wider CTA's
line, one to four images per view, and values that must not leak: infinities in
uncovered pixels and outside every covered pixel's footprint."""
import numpy as np
import pytest
import torch

from oracle import bilateral_ref as B
from tests.test_gpu_bilateral import guides  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,H,W,K,radius,sigma", [(1, 1, 1, 1, 0, 1.0), (1, 9, 33, 2, 8, 4.0), (2, 17, 31, 3, 7, 3.5),
                                                  (1, 8, 48, 4, 6, 3.0), (2, 35, 37, 1, 3, 1.5), (1, 16, 32, 4, 8, 4.0)])
def test_tiles_match_oracle(cuda_lib, guides, n, H, W, K, radius, sigma):
    mcdi = cuda_lib
    y0, x0 = (40 - H) // 2, (48 - W) // 2
    pos, nrm = (np.ascontiguousarray(a[:n, y0:y0 + H, x0:x0 + W]) for a in guides[:2])
    cams = guides[2][:n]
    rng = np.random.default_rng(100 * H + W)
    y, x = np.meshgrid(np.arange(H), np.arange(W), indexing="ij")
    covered = pos[..., 3] > 0
    c = rng.lognormal(0, 1, size=(K * n, H, W, 4)).astype(np.float32)
    g = rng.normal(size=(K * n, H, W, 4)).astype(np.float32)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()

    def run(c, g):
        out, gin = (torch.full((K * n, H, W, 4), float("nan"), device="cuda") for _ in range(2))
        wsum = torch.full((n, H, W), float("nan"), device="cuda")
        mcdi.bilateral_fwd(t(pos), t(nrm), t(cams), t(c), sigma, out, wsum, radius=radius)
        mcdi.bilateral_bwd(t(pos), t(nrm), t(cams), wsum, t(g), sigma, gin, radius=radius)
        torch.cuda.synchronize()
        return out.cpu().numpy(), gin.cpu().numpy(), wsum.cpu().numpy()

    out, gin, wsum = run(c, g)
    o_out, o_w = B.filter_forward(c[..., :3], pos, nrm, cams, sigma, radius)
    o_g = B.filter_backward(g[..., :3], pos, nrm, cams, sigma, radius)
    np.testing.assert_allclose(wsum, o_w, rtol=1e-4, atol=1e-6)  # the parity test's tolerances and scene
    np.testing.assert_allclose(out[..., :3], o_out, rtol=1e-4, atol=1e-5 * np.abs(o_out).max())
    # signed terms: the same relative error of each weight, against the sum of the terms' magnitudes
    mag = B.filter_backward(np.abs(g[..., :3]), pos, nrm, cams, sigma, radius)
    assert np.all(np.abs(gin[..., :3] - o_g) <= 1e-4 * mag + 1e-6), np.abs(gin[..., :3] - o_g).max()
    assert np.all(out[..., 3] == 0) and np.all(gin[..., 3] == 0)
    # an uncovered pixel's infinity stays there
    tile = np.tile(covered, (K, 1, 1))
    c2, g2 = c.copy(), g.copy()
    c2[~tile], g2[~tile] = np.inf, np.inf
    out2, gin2, _ = run(c2, g2)
    assert np.array_equal(out2[tile], out[tile]) and np.array_equal(gin2[tile], gin[tile])
    assert np.all(np.isinf(out2[~tile][:, :3])) and np.all(np.isinf(gin2[~tile][:, :3]))
    # and a covered one's reaches exactly its footprint (where its weight is not zero)
    yy, xx = H // 2, W // 2
    if covered[0, yy, xx]:
        c2 = c.copy()
        c2[0, yy, xx, :3] = np.inf
        out2 = run(c2, g)[0]
        far = (np.abs(y - yy) > radius) | (np.abs(x - xx) > radius)
        assert np.array_equal(out2[0][far], out[0][far]) and not np.isfinite(out2[0, yy, xx, 0])
        assert np.array_equal(out2[1:], out[1:])
