"""The U-Net's weight gradient does not depend on how its convolutions share
launches: with scratch from the least it accepts (the largest convolution's
partial sums, one or a few convolutions per launch) to what the library asks for
(one group), the results are the same bits, whatever the scratch held before."""
import numpy as np
import pytest
import torch

from tests.test_gpu_wgrad import make_inputs

pytestmark = pytest.mark.gpu

# (channels of the input and of the gradient, level) of each convolution
CONVS = [(16, 32, 0), (32, 32, 0), (32, 48, 1), (48, 48, 1), (48, 64, 2), (64, 64, 2), (64, 96, 3), (96, 96, 3),
         (160, 64, 2), (64, 64, 2), (112, 48, 1), (48, 48, 1), (80, 32, 0), (32, 32, 0), (32, 16, 0)]


@pytest.mark.parametrize("H,W", [(8, 8), (16, 24), (48, 136), (200, 264)])
def test_groups_do_not_change_the_bits(cuda_lib, H, W):
    mcdi = cuda_lib
    rng = np.random.default_rng(H * W)
    term, kd, nrm = make_inputs(rng, H, W)
    n_par = sum(co * ci * 9 + co for _, ci, co in mcdi.UNET_PLAN)
    den = mcdi.Denoiser(rng.normal(0, 0.05, n_par).astype(np.float32), 2, H, W)
    t = lambda a: torch.from_numpy(a).cuda().contiguous()
    y, gx = torch.zeros(term.shape, device="cuda"), torch.zeros(term.shape, device="cuda")
    den.forward(t(term), t(kd), t(nrm), y)
    den.backward(t(rng.normal(size=term.shape).astype(np.float32)), gx)
    least = max(mcdi.conv3x3_wgrad_bytes(2, H >> l, W >> l, ci, co) for ci, co, l in CONVS)
    full = mcdi.denoise_wgrad_bytes(2, H, W)
    assert full >= least
    out = []
    for n in sorted({least, (least + full) // 2, full, full + 4096}):
        scratch = torch.full((n,), 0xFF, dtype=torch.uint8, device="cuda")  # NaNs
        gw = torch.full((n_par,), float("nan"), device="cuda")
        mcdi.denoise_wgrad(den.acts, den.grad_ws, gw, scratch, den.err, 2, H, W)
        out.append(gw.clone())
    torch.cuda.synchronize()
    assert den.err.item() == 0 and torch.isfinite(out[0]).all() and out[0].abs().max() > 0
    for o in out[1:]:
        assert torch.equal(o, out[0])
    with pytest.raises(Exception, match="scratch too small"):
        mcdi.denoise_wgrad(den.acts, den.grad_ws, out[0], torch.empty(least - 1, dtype=torch.uint8, device="cuda"),
                           den.err, 2, H, W)
