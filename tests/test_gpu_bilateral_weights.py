"""The bilateral filter's backward is the transpose of its forward with the same
weights, bit for bit: with one pixel of every footprint set to one, the
forward's w(p, q) 1 / W(p) and the backward's 1 / W(p) w(p, q) are the same two
roundings.  Every pair (p, q) of a view whose footprints hold them, at radii on
both sides of each rule that chooses a kernel, with one to four images a view."""
import numpy as np
import pytest
import torch

from tests.test_gpu_bilateral import guides  # noqa: F401 (fixture)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("radius,K,sigma,scale", [(0, 2, 0.7, 1.0), (1, 1, 0.5, 1.0), (1, 4, 0.5, 1.0), (2, 2, 1.0, 1.0),
                                                  (2, 3, 0.6, 1.0), (4, 4, 2.0, 1.0), (6, 1, 3.0, 1.0), (7, 2, 3.5, 1.0),
                                                  (8, 4, 4.0, 1.0), (3, 2, 1.4, 2.0 ** -45), (3, 2, 1.4, 2.0 ** 45)])
def test_backward_has_the_forwards_weights(cuda_lib, guides, radius, K, sigma, scale):
    """scale: of the scene, so that its depths lie outside the range whose divisions take no branch."""
    mcdi, S = cuda_lib, 2 * radius + 1
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pos, nrm, cams = (t(a[:1].copy()) for a in guides)
    H, W = pos.shape[1:3]
    pos[..., :3] *= scale
    cams[:, :3] *= scale
    y, x = torch.meshgrid(torch.arange(H, device="cuda"), torch.arange(W, device="cuda"), indexing="ij")
    label = (y % S) * S + x % S  # a footprint holds each label once
    ones = lambda a: torch.stack([(label == k).float()[..., None].expand(H, W, 4) for k in a]).contiguous()
    fwd, bwd = (torch.zeros((S * S, H, W), device="cuda") for _ in range(2))
    out, wsum = torch.empty((K, H, W, 4), device="cuda"), torch.empty((1, H, W), device="cuda")
    for k0 in range(0, S * S, K):
        a = [min(k, S * S - 1) for k in range(k0, k0 + K)]
        mcdi.bilateral_fwd(pos, nrm, cams, ones(a), sigma, out, wsum, radius=radius)
        fwd[a] = out[..., 0]  # [label of q][p]
        mcdi.bilateral_bwd(pos, nrm, cams, wsum, ones(a), sigma, out, radius=radius)
        bwd[a] = out[..., 0]  # [label of p][q]
    torch.cuda.synchronize()
    pairs = 0
    cov = pos[0, ..., 3] > 0
    for dy in range(-radius, radius + 1):
        for dx in range(-radius, radius + 1):  # q = p + (dx, dy)
            ps = (slice(max(0, -dy), H - max(0, dy)), slice(max(0, -dx), W - max(0, dx)))
            qs = (slice(max(0, dy), H - max(0, -dy)), slice(max(0, dx), W - max(0, -dx)))
            both = cov[ps] & cov[qs]
            f = fwd[:, ps[0], ps[1]].gather(0, label[qs][None])[0]
            b = bwd[:, qs[0], qs[1]].gather(0, label[ps][None])[0]
            assert torch.isfinite(f[both]).all()
            assert torch.equal(f[both], b[both]), (dx, dy, (f - b)[both].abs().max())
            pairs += int((both & (f > 0)).sum())
    assert pairs > int(cov.sum()) * (1 if radius == 0 else 3) * 0.9


@pytest.mark.parametrize("radius,K", [(0, 1), (1, 2), (1, 4)])
def test_small_radii_on_both_sides_of_the_size_line(cuda_lib, guides, radius, K):
    """A large image, and a piece of it that is small enough for the kernel of one pixel per thread: the same bits
    wherever the piece holds the footprints and their slopes' neighbours."""
    mcdi, n = cuda_lib, 17
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    cams = t(guides[2][:1].copy())
    pos, nrm = (t(np.tile(a[:1], (1, n, n, 1))) for a in guides[:2])  # 680 x 816 pixels
    H, W = pos.shape[1:3]
    gen = torch.Generator(device="cuda").manual_seed(radius + K)
    g = torch.randn((K, H, W, 4), generator=gen, device="cuda")
    out, wsum = torch.empty_like(g), torch.empty((1, H, W), device="cuda")
    mcdi.bilateral_fwd(pos, nrm, cams, g, 0.5, out, wsum, radius=radius)
    mcdi.bilateral_bwd(pos, nrm, cams, wsum, g, 0.5, out, radius=radius)
    ys, xs, m = slice(200, 333), slice(311, 400), radius + 1
    cut = lambda a: a[:, ys, xs].contiguous()
    piece = torch.empty_like(cut(g))
    mcdi.bilateral_bwd(cut(pos), cut(nrm), cams, cut(wsum), cut(g), 0.5, piece, radius=radius)
    torch.cuda.synchronize()
    assert torch.equal(piece[:, m:-m, m:-m], cut(out)[:, m:-m, m:-m])
    assert (piece != cut(g)).any()
