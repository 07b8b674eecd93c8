"""Both searches of the spatial index and the scan, at every list length: the
neighbours and distances of a call with room for the index against the scan's,
bit for bit; the benchmark batches through the public calls against the oracle
(bounds as in test_gpu_knn.py)."""
import numpy as np
import pytest
import torch

from _gpu import grad_close
from oracle import knn as ok
from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops, workloads

pytestmark = pytest.mark.gpu


def _T(a):
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _packed(rng, lens, D):
    lens = np.asarray(lens, np.int64)
    first = np.concatenate([[0], np.cumsum(lens)[:-1]]).astype(np.int64)
    x = rng.normal(size=(int(lens.sum()), D))
    x[first[lens > 0]] *= 1e3   # one far point in every cloud
    return _T(x.astype(np.float32)), _T(first), _T(lens)


# ragged last warps and leaves, clouds smaller than K, empty clouds on either side
LANES = ([120_001, 0, 33, 90_000, 5, 31], [12_001, 700, 31, 12_500, 0, 3])
WARPS = ([901, 0, 33, 640, 5, 31], [60_001, 700, 31, 42_500, 0, 3])


@pytest.mark.parametrize("D", [1, 2, 3, 4])
@pytest.mark.parametrize("K", [1, 2, 4, 8, 16, 32])
@pytest.mark.parametrize("form,lens", [(ops.KNN_INDEX_LANES, LANES), (ops.KNN_INDEX_WARPS, WARPS)])
def test_every_search_equals_the_scan(form, lens, D, K):
    rng = np.random.default_rng(D * 100 + K)
    (p1, f1, l1), (p2, f2, l2) = (_packed(rng, n, D) for n in lens)
    N, P1, P2 = len(lens[0]), p1.shape[0], p2.shape[0]
    if form == ops.KNN_INDEX_WARPS and K < 5:
        p1, f1, l1 = _packed(rng, [5_000, 0, 33, 4_500, 5, 31], D)
        p2, f2, l2 = _packed(rng, [160_001, 700, 31, 42_500, 0, 3], D)
        P1, P2 = p1.shape[0], p2.shape[0]
    assert ops.knn_search_form(N, P1, P2, D, K) == form
    res = []
    for ws in (ops.alloc_knn_workspace(N, "cuda", P1, P2, D, K), ops.alloc_knn_workspace(N)):
        idx = torch.full((P1, K), -7, dtype=torch.int64, device="cuda")
        d = torch.full((P1, K), -7.0, device="cuda")
        ops.knn_points(p1, f1, l1, p2, f2, l2, K, idx, d, ws)
        res.append((idx, d.view(torch.int32)))
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])


@pytest.mark.parametrize("kind", ["knn", "knn_het"])
def test_knn_benchmark_workloads_through_the_index(kind):
    w = workloads.knn_workload(kind)
    c = w.pairs
    P, Q = _T(c.p).requires_grad_(True), _T(c.q).requires_grad_(True)
    assert ops.knn_search_form(c.N, P.shape[0], Q.shape[0], 3, w.K) != ops.KNN_SCAN
    dists, idx = ag.knn_points(P, _T(c.first1), _T(c.len1), Q, _T(c.first2), _T(c.len2), w.K)
    gi, gd = idx.cpu().numpy(), dists.detach().cpu().numpy()
    rng = np.random.default_rng(3)
    rows = np.concatenate([f + rng.choice(n, size=min(16, n), replace=False) for f, n in zip(c.first1, c.len1)])
    ri, rd = ok.knn(c.p, c.first1, c.len1, c.q, c.first2, c.len2, w.K, rows=rows)
    np.testing.assert_array_equal(gi[rows], ri)
    np.testing.assert_array_equal(gd[rows].view(np.uint32), rd.view(np.uint32))
    g = _T(rng.normal(size=gd.shape).astype(np.float32))
    got = torch.autograd.grad(dists, (P, Q), g)
    want = torch.empty_like(P), torch.empty_like(Q)
    ops.knn_points_bwd(P.detach(), Q.detach(), idx, g, *want)
    # the same kernels both ways; the float atomics may add in another order
    for a, b in zip(got, want):
        assert torch.linalg.norm(a - b) <= 1e-6 * torch.linalg.norm(b)


def test_chamfer_benchmark_batch_through_the_index():
    w = workloads.knn_workload("chamfer")
    c = w.pairs
    P, Q = _T(c.p).requires_grad_(True), _T(c.q).requires_grad_(True)
    assert ops.knn_search_form(c.N, P.shape[0], Q.shape[0], 3, 1) != ops.KNN_SCAN
    loss, per = ag.chamfer_distance(P, _T(c.first1), _T(c.len1), Q, _T(c.first2), _T(c.len2))
    g_per = np.random.default_rng(w.grad_seed).normal(size=c.N)
    got = torch.autograd.grad((loss, per), (P, Q), (torch.ones((), device="cuda"), _T(g_per.astype(np.float32))))
    r_loss, r_per, ipq, iqp = ok.chamfer(c.p, c.first1, c.len1, c.q, c.first2, c.len2)
    assert np.all(np.abs(per.detach().cpu().numpy() - r_per) <= 1e-5 * np.abs(r_per))
    assert abs(float(loss) - r_loss) <= 1e-5 * abs(r_loss)
    ref = ok.chamfer_grad(c.p, c.first1, c.len1, c.q, c.first2, c.len2, ipq, iqp, g_per + 1.0 / c.N)
    for a, b in zip(got, ref):
        worst, glob = grad_close(a.cpu().numpy(), b)
        assert glob <= 1e-4 and worst <= 1, (worst, glob)
