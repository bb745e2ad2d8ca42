"""GPU edge-sample lists at their edges: tables whose edges all count as
silhouettes (no second face), so that the list of outer rays fills and is traced
many times in a run, and thinned ones, whose short lists are traced in parts;
sample counts that do not divide a run; vertex arrays with 4- and 8-byte
alignment.  Decisions and weights against the oracle, with the tolerance of the
parity test."""
import numpy as np
import pytest
import torch

from tests import parity_util as PU
from tests.test_gpu_shadow_grad import ETA, _parity_case, weight_tol

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("keep,M,offset", [(1, 1, 0), (1, 32, 1), (1, 7, 1), (40, 32, 0), (0, 5, 0)])
def test_lists_match_oracle(cuda_lib, orc, keep, M, offset):
    """keep: every keep-th edge loses its second face (0: none)."""
    mcdi, tau = cuda_lib, 0.7
    sc, pipe, rows, prm = _parity_case(mcdi, orc, tau)
    W, H = sc.width, sc.height
    edges = orc.edge_table(sc.tris).copy()
    if keep:
        edges[::keep, 3] = -1
    et = mcdi.EdgeTable.allocate(len(sc.tris), "cuda")
    et.records[:len(edges)].copy_(torch.from_numpy(edges.astype(np.int32)))
    et.count.fill_(len(edges))
    V = pipe.verts.shape[0]
    verts = torch.empty(3 * V + 4, device="cuda")[offset:offset + 3 * V].view(V, 3).copy_(pipe.verts)
    rng = np.random.default_rng(17)
    gcd, gcs = (rng.normal(size=(H * W, 3)).astype(np.float32) for _ in range(2))
    pad = lambda a: torch.from_numpy(np.concatenate([a, np.zeros((len(a), 1), np.float32)], 1)).cuda().reshape(
        1, H, W, 4)
    g = torch.zeros(V, 3, device="cuda")
    w = torch.full((H * W, M), float("nan"), device="cuda")
    mcdi.shadow_edge_grad(pipe.bvh, verts, et, pipe.probe, pipe.gb, pipe.cams, prm, M, pad(gcd), pad(gcs), g, w,
                          eta=ETA)
    torch.cuda.synchronize()
    pix = np.arange(W * H)
    cam = np.tile(sc.cams[0, :3].astype(np.float64), (len(pix), 1))
    ctr = np.stack([pix, np.zeros_like(pix)], 1).astype(np.uint32)
    _, rec = orc.shadow_edge_grad(sc.verts, sc.tris, edges, sc.env, rows, cam, ctr, gcd, gcs, n_samples=M,
                                  seed=sc.seed, stream=2, tau=tau, ray_eps=1e-4, eta=ETA)
    w_orc, margin, w_gpu = rec[..., 0], rec[..., 1], w.cpu().numpy()
    safe = margin >= PU.MARGIN
    assert np.array_equal((w_gpu != 0)[safe], (w_orc != 0)[safe])
    c = safe & (w_orc != 0)
    assert c.sum() > 0
    floor = 1e-3 * np.abs(w_orc[w_orc != 0]).mean()
    err = np.abs(w_gpu - w_orc) / np.maximum(np.abs(w_orc), floor)
    assert np.all(err[safe] <= weight_tol(margin[safe])), err[safe].max()
    # every sample's weight reached its edge's two ends, and nothing else: sums of w n_out ((1 - s) + s)
    assert np.isfinite(g.cpu().numpy()).all()
    touched = np.unique(edges[rec[..., 2].astype(np.int64)[(w_gpu != 0)]][:, :2])
    rest = np.ones(V, bool)
    rest[touched] = False
    assert np.all(g.cpu().numpy()[rest] == 0) and np.any(g.cpu().numpy()[touched] != 0)
