"""The spatial-index search against the scan of every candidate (itself held to
the oracle in test_gpu_knn.py): neighbour rows and distances are bit-exact,
whatever the distribution, so the comparison needs no tolerance."""
import numpy as np
import pytest
import torch

from paper_2007_08501_gb300 import ops

pytestmark = pytest.mark.gpu


def _T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _cloud(rng, n, D, kind):
    if kind == "sphere":
        v = rng.normal(size=(n, D))
        return v / np.maximum(np.linalg.norm(v, axis=1, keepdims=True), 1e-9) + 0.3
    if kind == "lattice":       # equal distances everywhere: ranked by row
        return rng.integers(0, 9, size=(n, D)).astype(np.float64)
    if kind == "one_point":     # every candidate at the same place
        return np.full((n, D), 0.25)
    v = rng.normal(size=(n, D)) * 1e-3
    v[: max(1, n // 50)] *= 1e6   # "clustered": nearly all points in one grid cell
    return v


def _packed(rng, lens, D, kind, gap):
    # `gap` unused rows before every cloud
    first, at = [], 0
    for n in lens:
        at += gap
        first.append(at)
        at += n
    x = rng.normal(size=(at + gap, D))
    for f, n in zip(first, lens):
        x[f:f + n] = _cloud(rng, n, D, kind)
    return _T(x.astype(np.float32)), _T(np.asarray(first, np.int64)), _T(np.asarray(lens, np.int64))


def _both(a, b, K):
    D, out = a[0].shape[1], []
    big = ops.alloc_knn_workspace(len(a[1]), "cuda", a[0].shape[0], b[0].shape[0], D, K)
    small = ops.alloc_knn_workspace(len(a[1]))
    assert big.numel() > small.numel(), "the sizes do not take the index"
    for ws in (big, small):
        idx = torch.full((a[0].shape[0], K), -7, dtype=torch.int64, device="cuda")
        d = torch.full((a[0].shape[0], K), -7.0, device="cuda")
        ops.knn_points(*a, *b, K, idx, d, ws)
        out.append((idx, d))
    torch.cuda.synchronize()
    return out


@pytest.mark.parametrize("kind,gap", [("sphere", 0), ("lattice", 0), ("one_point", 0), ("clustered", 5)])
@pytest.mark.parametrize("D,K", [(1, 1), (2, 3), (3, 1), (3, 8), (3, 20), (4, 2), (4, 32)])
@pytest.mark.parametrize("few", [False, True])   # few queries: one per warp; else one per lane
def test_index_equals_scan(kind, gap, D, K, few):
    rng = np.random.default_rng(D * 100 + K)
    # leaf, node and grid-tile edges: 31, 32, 33, 1023, 1025 candidates; empty clouds; fewer candidates than K
    n2 = [90_001, 0, 31, 33, 1025, 1, 70_000, 32, 1023]
    n1 = [20_000, 50, 100, 129, 0, 127, 30_001, 33, 64]
    if few:
        n1 = [9_000, 3, 1, 0, 5, 7, 9_501, 2, 33]
        n2 = [200_001] + n2[1:]
    a, b = _packed(rng, n1, D, kind, gap), _packed(rng, n2, D, kind, gap)
    (i0, d0), (i1, d1) = _both(a, b, K)
    assert torch.equal(i0, i1)
    assert torch.equal(d0.view(torch.int32), d1.view(torch.int32))


@pytest.mark.parametrize("D", [2, 3])
def test_chamfer_with_the_index_equals_the_scan(D):
    rng = np.random.default_rng(D)
    a = _packed(rng, [700, 0, 1000, 9], D, "sphere", 3)
    b = _packed(rng, [900_000, 40, 800_000, 0], D, "sphere", 0)
    P, Q, N = a[0].shape[0], b[0].shape[0], 4
    res = []
    for ws in (ops.alloc_knn_workspace(N, "cuda", P, Q, D), ops.alloc_knn_workspace(N)):
        o = [torch.full((P,), -7, dtype=torch.int64, device="cuda"), torch.full((P,), -7.0, device="cuda"),
             torch.full((Q,), -7, dtype=torch.int64, device="cuda"), torch.full((Q,), -7.0, device="cuda"),
             torch.empty(N, device="cuda"), torch.empty(1, device="cuda")]
        ops.chamfer_fwd(*a, *b, *o, ws)
        res.append(o)
    torch.cuda.synchronize()
    assert all(torch.equal(x, y) for x, y in zip(*res))
