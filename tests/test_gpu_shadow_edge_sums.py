"""The edge gradient's vertex sums where its list of outer rays fills many times in
a run and where short lists are traced in parts: every sample reaches both ends
of its edge, once.  Against the oracle's sums, at every vertex, with each sample's
own tolerance and the whole of the marginal samples that touch it."""
import numpy as np
import pytest
import torch

from tests import parity_util as PU
from tests.test_gpu_shadow_grad import ETA, _parity_case, weight_tol

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("keep,M", [(1, 1), (1, 32), (40, 32), (0, 5)])
def test_vertex_sums_match_oracle(cuda_lib, orc, keep, M):
    """keep: every keep-th edge loses its second face, so that it always counts as a silhouette (0: none)."""
    mcdi, tau = cuda_lib, 0.7
    sc, pipe, rows, prm = _parity_case(mcdi, orc, tau)
    W, H, V = sc.width, sc.height, len(sc.verts)
    edges = orc.edge_table(sc.tris).copy()
    if keep:
        edges[::keep, 3] = -1
    et = mcdi.EdgeTable.allocate(len(sc.tris), "cuda")
    et.records[:len(edges)].copy_(torch.from_numpy(edges.astype(np.int32)))
    et.count.fill_(len(edges))
    rng = np.random.default_rng(29)
    gcd, gcs = (rng.normal(size=(H * W, 3)).astype(np.float32) for _ in range(2))
    pad = lambda a: torch.from_numpy(np.concatenate([a, np.zeros((len(a), 1), np.float32)], 1)).cuda().reshape(
        1, H, W, 4)
    g = torch.zeros(V, 3, device="cuda")
    w = torch.full((H * W, M), float("nan"), device="cuda")
    mcdi.shadow_edge_grad(pipe.bvh, pipe.verts, et, pipe.probe, pipe.gb, pipe.cams, prm, M, pad(gcd), pad(gcs), g, w,
                          eta=ETA)
    torch.cuda.synchronize()
    pix = np.arange(W * H)
    cam = np.tile(sc.cams[0, :3].astype(np.float64), (len(pix), 1))
    ctr = np.stack([pix, np.zeros_like(pix)], 1).astype(np.uint32)
    g_orc, rec = orc.shadow_edge_grad(sc.verts, sc.tris, edges, sc.env, rows, cam, ctr, gcd, gcs, n_samples=M,
                                      seed=sc.seed, stream=2, tau=tau, ray_eps=1e-4, eta=ETA)
    w_orc, margin, w_gpu = rec[..., 0], rec[..., 1], w.cpu().numpy().astype(np.float64)
    safe = margin >= PU.MARGIN
    # what a sample may move each of its ends by: its weight's tolerance (and that of its direction, of the same
    # order), or all of it where its decision is marginal; and FP32 sums of up to thousands of terms
    may = np.where(safe, (2 * weight_tol(np.maximum(margin, PU.MARGIN)) + 1e-4) * np.abs(w_orc),
                   np.abs(w_gpu) + np.abs(w_orc))
    ends = edges[rec[..., 2].astype(np.int64)][..., :2]
    tol = np.zeros(V)
    np.add.at(tol, ends.reshape(-1, 2), may.reshape(-1, 1))
    got = g.cpu().numpy().astype(np.float64)
    assert np.all(np.abs(got - g_orc).max(1) <= tol + 1e-12)
    # the bound tells a sample that reaches one end only, or twice: most of the sums are far above it
    size = np.abs(g_orc).max(1)
    assert (size > 20 * tol).sum() >= 0.3 * (size > 0).sum() > 0
