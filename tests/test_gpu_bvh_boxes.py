"""The boxes of the two-child nodes at the edges of the runs of leaves that a CTA
completes by itself: every box is exactly the union of its subtree's leaf boxes,
for meshes around a multiple of a run and of 32 leaves, for equal centroids (ties
by position) and for a chain-like tree, after a build and after a refit."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _mesh(n, kind, seed):
    rng = np.random.default_rng(seed)
    if kind == "soup":
        c = rng.uniform(-1, 1, (n, 3))
    elif kind == "equal":
        c = np.zeros((n, 3))
    else:  # chain: halving distances along one axis
        c = np.zeros((n, 3))
        c[:, 0] = 2.0 ** -(np.arange(n) % 40) + 1e-9 * np.arange(n)
    v = c[:, None, :] + rng.normal(0, 0.05, (n, 3, 3))
    if kind != "soup":
        v -= (v.mean(1) - c)[:, None, :]
    return v.reshape(-1, 3).astype(np.float32), np.arange(3 * n, dtype=np.int32).reshape(n, 3)


def _check(bvh, verts, tris, n):
    raw = bvh.nodes.cpu().numpy()[:64 * (n - 1)].reshape(n - 1, 64)
    f, d = raw.view(np.float32).reshape(n - 1, 16), raw.view(np.int32).reshape(n - 1, 16)[:, 12:]
    lo = np.stack([f[:, [0, 2, 8]], f[:, [4, 6, 10]]], 1)  # node, child, axis
    hi = np.stack([f[:, [1, 3, 9]], f[:, [5, 7, 11]]], 1)
    order = bvh.tri_records.cpu().numpy()[:48 * n].reshape(n, 48).view(np.int32).reshape(n, 12)[:, 3]
    assert np.array_equal(np.sort(order), np.arange(n))
    t = verts[tris[order]]
    llo, lhi = np.full((n, 3), np.nan, np.float32), np.full((n, 3), np.nan, np.float32)
    for h in range(2):  # leaf children: the triangle, a few ulps wider
        leaf = d[:, h] < 0
        p = ~d[leaf, h]
        llo[p], lhi[p] = lo[leaf, h], hi[leaf, h]
    assert not np.isnan(llo).any()
    assert np.all(llo <= t.min(1)) and np.all(lhi >= t.max(1))
    slack = 1e-6 * np.maximum(np.abs(t.min(1)), np.abs(t.max(1))) + 2e-30
    assert np.all(t.min(1) - llo <= slack) and np.all(lhi - t.max(1) <= slack)
    first, last = d[:, 2], d[:, 3]
    for h in range(2):  # inner children: the union of their leaves, to the bit
        inner = np.nonzero(d[:, h] >= 0)[0]
        c = d[inner, h]
        e_lo = np.stack([llo[first[k]:last[k] + 1].min(0) for k in c]) if len(c) else np.zeros((0, 3))
        e_hi = np.stack([lhi[first[k]:last[k] + 1].max(0) for k in c]) if len(c) else np.zeros((0, 3))
        assert np.array_equal(lo[inner, h], e_lo) and np.array_equal(hi[inner, h], e_hi)


@pytest.mark.parametrize("kind", ["soup", "equal", "chain"])
@pytest.mark.parametrize("n", [2, 31, 33, 255, 257, 511, 512, 513, 1025, 5000])
def test_boxes_are_unions(cuda_lib, n, kind):
    mcdi = cuda_lib
    verts, tris = _mesh(n, kind, n)
    t = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    bvh = mcdi.Bvh.allocate(n)
    bvh.scratch.fill_(0xFF)
    bvh.build(t(verts), t(tris))
    torch.cuda.synchronize()
    _check(bvh, verts, tris, n)
    moved = (verts + 0.3 * np.sin(5 * verts[:, [1, 2, 0]])).astype(np.float32)
    bvh.refit(t(moved), t(tris))
    torch.cuda.synchronize()
    _check(bvh, moved, tris, n)
