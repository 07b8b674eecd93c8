"""render_points on packed slots against the Fragment entry points (themselves
held to the oracle): the image is the same arithmetic, the gradients differ by
the order of their sums and the rounding of the projected point (1e-5 of their
norm; images 1e-6)."""
import numpy as np
import pytest
import torch

from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops, workloads

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("counts,S,K,radius,D,mode,bin_size", [
    ([700, 0, 33], 33, 1, 0.05, 1, ops.PTS_ALPHA, 8), ([4000, 900], 64, 10, 0.03, 3, ops.PTS_NORM, 16),
    ([5000], 40, 50, 0.04, 1, ops.PTS_ALPHA, 8), ([3000, 10], 50, 17, 0.3, 2, ops.PTS_ALPHA, 16),
    ([2500], 36, 64, 0.06, 4, ops.PTS_NORM, 8), ([2500], 36, 8, 0.06, 6, ops.PTS_ALPHA, 16),
    ([1500, 1500], 36, 9, 0.06, 8, ops.PTS_NORM, 8), ([1500], 36, 5, 0.06, 7, ops.PTS_ALPHA, 8)])
def test_packed_points_match_fragment_path(counts, S, K, radius, D, mode, bin_size):
    b = workloads.point_batch(np.asarray(counts), 77, level=3, sigma=0.05, D=D)
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
