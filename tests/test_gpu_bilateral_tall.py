"""Images with more rows of tiles than a grid's second axis holds: the forward
takes up to 16 x 65,535 rows, and the backward as many, in both of its forms."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("H,W,radius", [(524288, 4, 2), (524281, 3, 4), (1048560, 2, 3), (1048560, 1, 0)])
def test_tall_images(cuda_lib, H, W, radius):
    mcdi = cuda_lib
    gen = torch.Generator(device="cuda").manual_seed(radius)
    rand = lambda *s: torch.rand(s, generator=gen, device="cuda")
    pos, nrm, g = rand(1, H, W, 4), rand(1, H, W, 4) + 0.5, rand(1, H, W, 4)
    pos[..., 2] -= 3
    pos[..., 3] = (pos[..., 3] > 0.2).float()
    cams = torch.tensor([[0, 0, 0, 1, 0, 0, 0, 1, 0, 0, 0, -1, 0.4, W / H]], device="cuda", dtype=torch.float32)

    def run(pos, nrm, g):
        out, gin = (torch.full_like(g, float("nan")) for _ in range(2))
        wsum = torch.full(g.shape[:3], float("nan"), device="cuda")
        mcdi.bilateral_fwd(pos, nrm, cams, g, 1.0, out, wsum, radius=radius)
        mcdi.bilateral_bwd(pos, nrm, cams, wsum, g, 1.0, gin, radius=radius)
        torch.cuda.synchronize()
        return out, gin, wsum

    whole = run(pos, nrm, g)
    assert all(torch.isfinite(a).all() for a in whole)
    m = 2 * radius + 2  # rows whose weights, or whose neighbours' weight sums, the cut touches
    for y0, y1 in ((0, 700), (H // 2 - 350, H // 2 + 350), (H - 700, H)):
        piece = run(*(a[:, y0:y1].contiguous() for a in (pos, nrm, g)))
        lo, hi = (0 if y0 == 0 else m), (y1 - y0 if y1 == H else y1 - y0 - m)
        for a, b in zip(whole, piece):
            assert torch.equal(a[:, y0 + lo:y0 + hi], b[:, lo:hi])
