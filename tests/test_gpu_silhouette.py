"""render_meshes on packed silhouette slots against the Fragment entry points
(rast_blend_fwd and blend_rast_bwd, themselves held to the oracle): the image is
the same arithmetic (bit for bit where the product's order is too), the
gradients differ by the order of their sums only (1e-5, as in test_gpu_fused)."""
import numpy as np
import pytest
import torch

from paper_2007_08501_gb300 import autograd as ag
from paper_2007_08501_gb300 import ops, workloads

pytestmark = pytest.mark.gpu

BLUR = workloads.BLUR_SIGMA_1E4


@pytest.mark.parametrize("levels,S,K,bin_size,persp,blur", [
    ([2, 4, 3], 33, 1, 8, True, 0.0), ([4, 2], 70, 3, 16, False, BLUR), ([3, 3, 5], 64, 8, 16, True, BLUR),
    ([4], 48, 16, 8, True, 9 * BLUR), ([4, 3], 41, 20, 8, True, BLUR), ([5, 2], 64, 50, 16, True, 4 * BLUR),
    ([3], 40, 64, 16, False, 9 * BLUR)])
def test_packed_silhouette_matches_fragment_path(levels, S, K, bin_size, persp, blur):
    b = workloads.sphere_batch(levels, 0.05, seed_base=31)
    T = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    v, f, ff, nf, cams = T(b.verts), T(b.faces), T(b.first_face), T(b.num_faces), T(b.cams)
    rs = ag.RasterSettings(S, K, float(np.float32(blur)), bin_size, 8192, 0, persp, blur > 0)
    bs = ag.BlendSettings(rgb=False)
    N = len(levels)
    g = torch.randn((N, S, S, 4), device="cuda", generator=torch.Generator("cuda").manual_seed(K))
    p, bp = rs.params(N), bs.params()
    ws = ops.alloc_workspace(p, b.V, b.F)
    fr = ops.alloc_fragments(N, S, K)
    ref = torch.empty((N, S, S, 4), device="cuda")
    ops.rast_blend_fwd(p, bp, v, f, ff, nf, cams, None, *fr, ref, ws)
    want = torch.empty_like(v)
    ops.blend_rast_bwd(p, bp, v, f, ff, nf, cams, fr[0], None, None, fr[3], None, g, want, None, ws)
    assert ops.sil_packed(p, b.V, b.F)
    v.requires_grad_(True)
    img = ag.render_meshes(v, f, ff, nf, cams, rs, bs)
    got, = torch.autograd.grad(img, v, g)
    assert torch.equal(img, ref)
    assert (got - want).norm() <= 1e-5 * want.norm()
    assert want.abs().max() > 0


def test_faces_without_pixels_and_empty_batches():
    rs, bs = ag.RasterSettings(16, 4, BLUR, 8, clip_barycentric_coords=True), ag.BlendSettings(rgb=False)
    I = lambda *x: torch.tensor(x, dtype=torch.int64, device="cuda")
    for N, F in ((1, 0), (0, 0), (2, 0)):
        v = torch.zeros((3, 3), device="cuda", requires_grad=True)
        f = torch.zeros((F, 3), dtype=torch.int64, device="cuda")
        img = ag.render_meshes(v, f, I(*[0] * N), I(*[0] * N), torch.zeros((N, 16), device="cuda"), rs, bs)
        assert img.shape == (N, 16, 16, 4) and not img.any()
        g, = torch.autograd.grad(img.sum(), v)
        assert not g.any()
