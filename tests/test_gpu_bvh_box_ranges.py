"""Node boxes that span more than 32 runs of leaves, formed from whole runs, whole
32s and single leaves at both ends: unions of their leaf boxes to the bit."""
import numpy as np
import pytest
import torch

from tests.test_gpu_bvh_boxes import _check, _mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["soup", "equal", "chain"])
@pytest.mark.parametrize("n", [16385, 20000, 40007])
def test_boxes_over_many_runs(cuda_lib, n, kind):
    verts, tris = _mesh(n, kind, n)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    bvh = cuda_lib.Bvh.allocate(n)
    bvh.scratch.fill_(0xFF)
    bvh.build(t(verts), t(tris))
    torch.cuda.synchronize()
    _check(bvh, verts, tris, n)
