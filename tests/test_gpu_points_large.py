"""Splats of 16 pixels and more, whose gradients a warp sums before it sends them,
against the Fragment entry points (bounds as in test_gpu_points_packed.py)."""
import numpy as np
import pytest
import torch

from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts,S,K,radius,D,mode,bin_size", [
    ([70, 0, 3], 64, 1, 0.5, 1, ops.PTS_ALPHA, 8), ([400, 90], 70, 10, 0.6, 3, ops.PTS_NORM, 16),
    ([500], 45, 50, 0.8, 1, ops.PTS_ALPHA, 16), ([300, 10], 100, 17, 0.4, 2, ops.PTS_ALPHA, 16),
    ([250], 65, 64, 1.5, 4, ops.PTS_NORM, 8), ([5], 130, 8, 0.3, 6, ops.PTS_ALPHA, 16),
    ([150, 150], 47, 9, 0.7, 8, ops.PTS_NORM, 8)])
def test_large_splats_match_fragment_path(counts, S, K, radius, D, mode, bin_size):
    assert 0.5 * radius * S >= 16
    b = workloads.point_batch(np.asarray(counts), 78, level=3, sigma=0.05, D=D)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    pts, ft, first, num, cams = T(b.points), T(b.features), T(b.first_point), T(b.num_points), T(b.cams)
    N, P = len(counts), pts.shape[0]
    st = ag.PointSettings(S, K, radius, bin_size=bin_size, max_points_per_bin=max(counts), mode=mode)
    g = torch.randn((N, S, S, D), device="cuda", generator=torch.Generator("cuda").manual_seed(K))
    p = st.params(N)
    ws = ops.alloc_pts_workspace(p, P)
    idx, zbuf, dists = ops.alloc_pts_fragments(N, S, K)
    ops.pts_rasterize_fwd(p, pts, first, num, cams, idx, zbuf, dists, ws)
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
