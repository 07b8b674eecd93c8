"""The binned fine passes' front-to-back windows against the plain form, which
meets the faces in packed order and evaluates each with the same arithmetic:
every Fragment value is bit-exact, so the comparison needs no tolerance.  Depth
distributions that leave the common path: everything at one depth, outliers
that squeeze the rest into one bucket, both at once."""
import numpy as np
import pytest
import torch

import _gpu as G
import _scenes as SC
from paper_2007_08501_gb300 import ops

pytestmark = pytest.mark.gpu


def _depths(kind, n, rng):
    if kind == "ramp":
        return np.linspace(3.0, 1.0, n)
    z = 2.0 + (1e-4 * rng.random(n) if kind == "near_far" else np.zeros(n))
    if kind in ("near_far", "flat_outliers"):
        z[n // 2], z[n // 3] = 0.2, 60.0
    return z


@pytest.mark.parametrize("kind", ["ramp", "flat", "near_far", "flat_outliers"])
@pytest.mark.parametrize("n,K,blur,clip", [
    (64, 1, 0.0, False), (65, 8, 1e-3, True), (1025, 5, 1e-3, True), (3000, 8, 1e-3, True), (3000, 3, 0.0, False),
    (3000, 16, 1e-3, False), (1500, 24, 1e-3, False), (9000, 20, 1e-3, True)])
def test_windows_match_the_plain_form(kind, n, K, blur, clip):
    rng = np.random.default_rng(7 * n + K)
    tris = []
    for z in _depths(kind, n, rng):
        c = rng.uniform(-0.4, 0.4, 2)
        p = c + rng.uniform(-0.12, 0.12, (3, 2))
        tris.append(SC.ndc_triangle(*p, z + rng.uniform(0.0, 0.02, 3) * (kind == "ramp")))
    d = G.to_dev(SC.scene(tris, cams=np.stack([SC.identity_cam()])))
    S = 36
    ref, _, _, _ = G.gpu_fwd(d, S, K, blur, bin_size=0, clip=clip)
    for bin_size in (8, 16):
        out, status, _, _ = G.gpu_fwd(d, S, K, blur, bin_size=bin_size, clip=clip, max_faces_per_bin=n)
        assert status == 0
        for a, b in zip(out, ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("kind", ["ramp", "flat", "near_far", "flat_outliers"])
@pytest.mark.parametrize("n,K,radius", [
    (32, 1, 0.05), (33, 10, 0.05), (600, 3, 0.9), (1025, 50, 0.02), (5000, 50, 0.05), (5000, 64, 0.3), (9000, 8, 0.1)])
def test_point_windows_match_the_plain_form(kind, n, K, radius):
    rng = np.random.default_rng(11 * n + K)
    z = rng.permutation(_depths(kind, n, rng))
    xy = rng.uniform(-0.5, 0.5, (n, 2))
    pts = torch.from_numpy(np.concatenate([xy * z[:, None], z[:, None]], 1).astype(np.float32)).cuda()
    cams = torch.from_numpy(SC.identity_cam()[None].astype(np.float32)).cuda()
    first, num = torch.zeros(1, dtype=torch.int64).cuda(), torch.tensor([n]).cuda()
    S = 36

    def run(bin_size):
        p = ops.make_pts_params(1, S, K, radius, bin_size, n, 0)
        ws = torch.empty(ops.pts_workspace_bytes(p, n), dtype=torch.uint8, device="cuda")
        out = ops.alloc_pts_fragments(1, S, K, "cuda")
        ops.pts_rasterize_fwd(p, pts, first, num, cams, *out, ws)
        assert ops.rast_query_status(ws) == 0
        return out

    ref = run(0)
    for bin_size in (8, 16):
        for a, b in zip(run(bin_size), ref):
            assert torch.equal(a, b)
