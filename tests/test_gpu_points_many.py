"""Batches with enough points that staging and filling count a block's bins in
shared memory: blocks across several small clouds and an empty one, bins of
either size, bins that overflow.  Fragments are bit-exact against the plain
form; the packed image and gradients within 1e-6 and 1e-5 of the Fragment
calls' (as in test_gpu_points_packed.py)."""
import numpy as np
import pytest
import torch

from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops, workloads

pytestmark = pytest.mark.gpu

# the shared-memory counting starts at two blocks of 2,048 points per SM
COUNTS = [400_003, 300, 0, 700, 1, 2_047, 300_001, 513]


def _clouds(D):
    b = workloads.point_batch(np.asarray(COUNTS), 19, level=3, sigma=0.05, D=D)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    assert sum(COUNTS) >= 2 * 2048 * torch.cuda.get_device_properties(0).multi_processor_count
    return T(b.points), T(b.features), T(b.first_point), T(b.num_points), T(b.cams)


def _fragments(p, pts, first, num, cams):
    ws = ops.alloc_pts_workspace(p, pts.shape[0])
    out = ops.alloc_pts_fragments(p.N, p.image_size, p.points_per_pixel)
    ops.pts_rasterize_fwd(p, pts, first, num, cams, *out, ws)
    return out, ops.rast_query_status(ws), ws


@pytest.mark.parametrize("S,K,radius,bin_size", [(61, 3, 0.02, 8), (61, 20, 0.03, 16), (200, 10, 0.01, 8)])
def test_many_points_match_the_plain_form(S, K, radius, bin_size):
    pts, _, first, num, cams = _clouds(1)
    N, P = len(COUNTS), pts.shape[0]
    ref, _, _ = _fragments(ops.make_pts_params(N, S, K, radius, 0, 0, 0), pts, first, num, cams)
    got, status, _ = _fragments(ops.make_pts_params(N, S, K, radius, bin_size, P, 8 * P), pts, first, num, cams)
    assert status == 0
    for a, b in zip(got, ref):
        assert torch.equal(a, b)


@pytest.mark.parametrize("bin_size,D,mode", [(8, 3, ops.PTS_NORM), (16, 1, ops.PTS_ALPHA)])
def test_many_points_packed_match_the_fragment_path(bin_size, D, mode):
    pts, ft, first, num, cams = _clouds(D)
    N, P, S, K, radius = len(COUNTS), pts.shape[0], 61, 10, 0.02
    st = ag.PointSettings(S, K, radius, bin_size=bin_size, max_points_per_bin=P, max_bin_entries=8 * P, mode=mode)
    g = torch.randn((N, S, S, D), device="cuda", generator=torch.Generator("cuda").manual_seed(D))
    p = st.params(N)
    (idx, _, dists), status, ws = _fragments(p, pts, first, num, cams)
    assert status == 0
    ref = torch.empty((N, S, S, D), device="cuda")
    ops.pts_composite_fwd(p, mode, idx, dists, ft, ref)
    gd, wf, wp = torch.empty_like(dists), torch.empty_like(ft), torch.empty_like(pts)
    ops.pts_composite_bwd(p, mode, idx, dists, ft, g, gd, wf)
    ops.pts_rasterize_bwd(p, pts, first, num, cams, idx, None, gd, wp, ws)
    img = ag.render_points(pts.requires_grad_(True), ft.requires_grad_(True), first, num, cams, st)
    gp, gf = torch.autograd.grad(img, (pts, ft), g)
    assert (img - ref).abs().max() <= 1e-6
    for got, want in ((gp, wp), (gf, wf)):
        assert want.abs().max() > 0
        assert (got - want).norm() <= 1e-5 * want.norm()


@pytest.mark.parametrize("bin_size", [8, 16])
def test_overflowing_bins_keep_valid_points(bin_size):
    pts, _, first, num, cams = _clouds(1)
    N, S, K = len(COUNTS), 61, 10
    for cap, entries in ((100, 0), (pts.shape[0], 50_000)):
        (idx, _, _), status, ws = _fragments(ops.make_pts_params(N, S, K, 0.02, bin_size, cap, entries), pts, first,
                                             num, cams)
        assert status & ops.ST_BIN_OVERFLOW
        for n in range(N):
            i = idx[n][idx[n] >= 0]
            lo = int(first[n])
            assert bool(((i >= lo) & (i < lo + COUNTS[n])).all())
    assert int((idx >= 0).sum()) > 0
