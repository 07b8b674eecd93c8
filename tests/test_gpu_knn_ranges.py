"""Clouds whose ranges are not ascending and disjoint -- one candidate cloud
shared by several query clouds, clouds in another order, empty clouds that start
anywhere -- get the scan's answer at sizes the spatial index serves too.  Rows
and distances are bit-exact."""
import numpy as np
import pytest
import torch

from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops

pytestmark = pytest.mark.gpu


def _T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _ranges(kind):
    """(first1, len1, first2, len2), rows of either array."""
    P1, P2 = 70_000, 90_000
    if kind == "shared":                    # three query clouds, one candidate cloud
        return [0, 30_000, 50_000], [30_000, 20_000, 20_000], [0, 0, 0], [P2] * 3, P1, P2
    if kind == "overlapping":
        return [0, 30_000, 50_000], [30_000, 20_000, 20_000], [0, 20_000, 10_001], [50_000, 60_000, 79_999], P1, P2
    if kind == "reversed":
        return [40_000, 33, 0], [30_000, 39_967, 33], [60_001, 31, 0], [29_999, 59_970, 31], P1, P2
    if kind == "queries_reversed":
        return [40_000, 0], [30_000, 40_000], [0, 45_000], [45_000, 45_000], P1, P2
    # an empty cloud in the middle that starts at 0
    return [0, 0, 30_000], [30_000, 0, 40_000], [0, 0, 50_000], [50_000, 0, 40_000], P1, P2


KINDS = ["shared", "overlapping", "reversed", "queries_reversed", "empty_anywhere"]


@pytest.mark.parametrize("kind", KINDS)
@pytest.mark.parametrize("D,K", [(3, 1), (2, 3), (3, 8), (4, 20)])
def test_ranges_in_any_order_equal_the_scan(kind, D, K):
    f1, l1, f2, l2, P1, P2 = _ranges(kind)
    rng = np.random.default_rng(K)
    p1, p2 = _T(rng.normal(size=(P1, D)).astype(np.float32)), _T(rng.normal(size=(P2, D)).astype(np.float32))
    F1, L1, F2, L2 = (_T(np.asarray(v, np.int64)) for v in (f1, l1, f2, l2))
    small = ops.alloc_knn_workspace(len(f1))
    big = ops.alloc_knn_workspace(len(f1), "cuda", P1, P2, D, K)
    assert big.numel() > small.numel(), "the sizes do not take the index"
    idx, d = torch.empty((P1, K), dtype=torch.int64, device="cuda"), torch.empty((P1, K), device="cuda")
    ops.knn_points(p1, F1, L1, p2, F2, L2, K, idx, d, small)
    got_d, got_i = ag.knn_points(p1, F1, L1, p2, F2, L2, K)
    assert torch.equal(got_i, idx) and torch.equal(got_d.view(torch.int32), d.view(torch.int32))
    # and the clouds laid out one after the other, which the index answers
    a = torch.cat([p1[f:f + n] for f, n in zip(f1, l1)])
    b = torch.cat([p2[f:f + n] for f, n in zip(f2, l2)])
    A, B = (_T(np.concatenate([[0], np.cumsum(v)[:-1]]).astype(np.int64)) for v in (l1, l2))
    want_d, want_i = ag.knn_points(a, A, L1, b, B, L2, K)
    for i, (f, n) in enumerate(zip(f1, l1)):
        at = int(A[i])
        assert torch.equal(got_i[f:f + n], want_i[at:at + n] - int(B[i]) + f2[i])
        assert torch.equal(got_d[f:f + n], want_d[at:at + n])


@pytest.mark.parametrize("kind", ["reversed", "queries_reversed", "empty_anywhere"])
def test_chamfer_ranges_in_any_order_equal_the_scan(kind):
    f1, l1, f2, l2, P1, P2 = _ranges(kind)
    rng = np.random.default_rng(5)
    p, q = _T(rng.normal(size=(P1, 3)).astype(np.float32)), _T(rng.normal(size=(P2, 3)).astype(np.float32))
    r = [_T(np.asarray(v, np.int64)) for v in (f1, l1, f2, l2)]
    N, res = len(f1), []
    for ws in (ops.alloc_knn_workspace(N, "cuda", P1, P2, 3), ops.alloc_knn_workspace(N)):
        o = [torch.full((P1,), -7, dtype=torch.int64, device="cuda"), torch.full((P1,), -7.0, device="cuda"),
             torch.full((P2,), -7, dtype=torch.int64, device="cuda"), torch.full((P2,), -7.0, device="cuda"),
             torch.empty(N, device="cuda"), torch.empty(1, device="cuda")]
        ops.chamfer_fwd(p, r[0], r[1], q, r[2], r[3], *o, ws)
        res.append((ws.numel(), o))
    assert res[0][0] > res[1][0], "the sizes do not take the index"
    assert all(torch.equal(x, y) for x, y in zip(res[0][1], res[1][1]))
