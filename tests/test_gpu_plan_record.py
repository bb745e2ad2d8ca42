"""The recorded launch plan names the form each convolution runs in: row tiles
from 48 pixels wide, halo tiles below."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["BF16", "E4M3"])
@pytest.mark.parametrize("W", [24, 64, 200])
def test_forms_are_told_apart(cuda_lib, precision, W):
    mcdi, H = cuda_lib, 32
    n_par = sum(co * ci * 9 + co for _, ci, co in mcdi.UNET_PLAN)
    den = mcdi.Denoiser(np.random.default_rng(2).normal(0, 0.05, n_par).astype(np.float32), 2, H, W,
                        precision=getattr(mcdi, precision))
    term, kd, nrm = (torch.rand((2, H, W, 4), device="cuda") for _ in range(3))
    y, gx = torch.empty_like(term), torch.empty_like(term)
    with mcdi.denoise_plan_recorder() as rec:
        den.forward(term, kd, nrm, y)
        den.backward(term, gx)
    torch.cuda.synchronize()
    assert len(rec.records) == 30
    for r in rec.records:
        assert r["rows_form"] == (1 if W >> r["level"] >= 48 else 2), r
        assert (r["rows"] > 0) == (r["rows_form"] == 1), r
