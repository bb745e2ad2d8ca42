"""Calls that encode tensor maps work as a host thread's first use of the GPU:
the driver's encoder needs a context that is current in the calling thread."""
import threading

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _in_fresh_thread(call):
    failed = []

    def work():
        try:
            call()
        except Exception as e:  # noqa: BLE001 (reported below)
            failed.append(e)

    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not failed, failed


@pytest.mark.parametrize("what", ["denoise_fwd", "conv3x3_wgrad"])
@pytest.mark.parametrize("W", [24, 128])
def test_first_call_of_a_thread(cuda_lib, what, W):
    mcdi, H = cuda_lib, 16
    stream = torch.cuda.current_stream()
    if what == "denoise_fwd":
        n_par = sum(co * ci * 9 + co for _, ci, co in mcdi.UNET_PLAN)
        den = mcdi.Denoiser(np.random.default_rng(1).normal(0, 0.05, n_par).astype(np.float32), 2, H, W)
        term, kd, nrm = (torch.rand((2, H, W, 4), device="cuda") for _ in range(3))
        want, got = torch.zeros_like(term), torch.zeros_like(term)
        den.forward(term, kd, nrm, want)
        torch.cuda.synchronize()
        _in_fresh_thread(lambda: den.forward(term, kd, nrm, got, stream))
    else:
        x, g = (torch.randn((1, c // 8, H, W, 8), device="cuda").bfloat16() for c in (16, 32))
        want, got = (torch.zeros(32 * 16 * 9 + 32, device="cuda") for _ in range(2))
        err = torch.zeros(1, dtype=torch.int32, device="cuda")
        scratch = torch.empty(mcdi.conv3x3_wgrad_bytes(1, H, W, 16, 32), dtype=torch.uint8, device="cuda")
        mcdi.conv3x3_wgrad(x, g, 16, 32, want, scratch, err)
        torch.cuda.synchronize()
        _in_fresh_thread(lambda: mcdi.conv3x3_wgrad(x, g, 16, 32, got, scratch, err, stream))
    assert torch.equal(got, want) and want.abs().max() > 0
