"""The denoiser's elementwise kernels over planes: more planes than a grid has
rows (thousands of the smallest images), pixel counts around a block, and the
published maxima of E4M3 tensors.  Images do not see each other in BF16, so a
large batch gives each image the bits a small one does; in E4M3 a batch of
copies has the maxima, and so the bits, of one."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _run(mcdi, flat, term, kd, nrm, gy, precision):
    n, H, W = term.shape[:3]
    den = mcdi.Denoiser(flat, n, H, W, precision=precision)
    y, gx = torch.full_like(term, float("nan")), torch.full_like(term, float("nan"))
    den.forward(term, kd, nrm, y)
    den.backward(gy, gx)
    torch.cuda.synchronize()
    assert den.err.item() == 0
    return y, gx


def _inputs(n, H, W, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    r = lambda: torch.randn((n, H, W, 4), generator=g, device="cuda")
    t = r().abs()
    t[..., 3] = 0
    return t, r().abs(), r(), r()


@pytest.mark.parametrize("n,H,W,precision", [(7000, 8, 8, "bf16"), (3, 16, 24, "bf16"), (2, 136, 120, "bf16"),
                                             (6600, 8, 8, "e4m3"), (4, 24, 40, "e4m3"), (3, 128, 136, "e4m3")])
def test_images_of_a_batch_do_not_see_each_other(cuda_lib, n, H, W, precision):
    mcdi = cuda_lib
    flat = np.random.default_rng(1).normal(0, 0.08, sum(co * ci * 9 + co for _, ci, co in mcdi.UNET_PLAN)).astype(
        np.float32)
    prec = mcdi.E4M3 if precision == "e4m3" else mcdi.BF16
    term, kd, nrm, gy = _inputs(n if precision == "bf16" else 1, H, W, n)
    pick = [0, n // 2, n - 1] if precision == "bf16" else [0]
    small = _run(mcdi, flat, *(a[pick].contiguous() for a in (term, kd, nrm, gy)), prec)
    if precision == "e4m3":
        term, kd, nrm, gy = (a.expand(n, -1, -1, -1).contiguous() for a in (term, kd, nrm, gy))
        pick = [0, n // 2, n - 1]
    big = _run(mcdi, flat, term, kd, nrm, gy, prec)
    for b, s in zip(big, small):
        assert torch.isfinite(s).all() and s.abs().max() > 0
        assert torch.equal(b[pick], s.expand(len(pick), -1, -1, -1))
