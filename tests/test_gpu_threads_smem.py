"""Host threads that call the same kernel with different needs of shared memory
beyond the default limit do not take it from each other: probes of different
heights without scratch memory, weight gradients of different widths, bilateral
filters with different numbers of images and tile sizes."""
import threading

import numpy as np
import pytest
import torch

from paper_2206_03380_gb300 import scenes

pytestmark = pytest.mark.gpu

CALLS = 4000


def _rand(*shape):
    return torch.rand(shape, device="cuda") + 0.1


def _forward(mcdi, rows):
    from paper_2206_03380_gb300.pipeline import ShadingPipeline

    base = scenes.parity_scene()
    env = np.ones((rows, 4, 4), np.float32)
    pipe = ShadingPipeline(scenes.Scene(**{**base.__dict__, "env": env, "width": 4, "height": 4, "n_light": 1,
                                           "n_cos": 0, "n_ggx": 0}), wavefront=False)
    pipe.build_probe()
    pipe.build_bvh()
    pipe.primary()
    return pipe.forward


def _wgrad(mcdi, cout):
    x, g = (torch.zeros((1, c // 8, 4, 128, 8), dtype=torch.bfloat16, device="cuda") for c in (16, cout))
    gw, err = torch.empty(cout * 16 * 9 + cout, device="cuda"), torch.zeros(1, dtype=torch.int32, device="cuda")
    scratch = torch.empty(mcdi.conv3x3_wgrad_bytes(1, 4, 128, 16, cout), dtype=torch.uint8, device="cuda")
    return lambda stream: mcdi.conv3x3_wgrad(x, g, 16, cout, gw, scratch, err, stream)


def _bilateral(mcdi, K, H, backward):
    pos, nrm, src, out = _rand(1, H, 24, 4), _rand(1, H, 24, 4), _rand(K, H, 24, 4), _rand(K, H, 24, 4)
    wsum, cams = _rand(1, H, 24), torch.from_numpy(scenes.parity_scene().cams[:1].astype(np.float32)).cuda()
    if backward:
        return lambda stream: mcdi.bilateral_bwd(pos, nrm, cams, wsum, src, 4.0, out, stream=stream)
    return lambda stream: mcdi.bilateral_fwd(pos, nrm, cams, src, 4.0, out, wsum, stream=stream)


@pytest.mark.parametrize("make,a,b", [(_forward, (4096,), (2420,)), (_wgrad, (16,), (32,)),
                                      (_bilateral, (4, 8, False), (2, 8, False)), (_bilateral, (4, 8, True), (4, 1300, True))])
def test_two_threads(cuda_lib, make, a, b):
    calls = [make(cuda_lib, *args) for args in (a, b)]
    torch.cuda.synchronize()
    start, failed = threading.Barrier(2), []

    def work(call):
        stream = torch.cuda.Stream()
        start.wait()
        try:
            for k in range(CALLS):
                call(stream)
                if k % 100 == 99:
                    stream.synchronize()
        except Exception as e:  # noqa: BLE001 (reported below)
            failed.append(e)
        stream.synchronize()

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed, failed
