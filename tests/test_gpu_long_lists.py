"""Bins of so many entries that the fine pass leaves them to a second round on
sorted lists, beside bins that it finishes.  Every Fragment value is bit-exact
against the plain form, which meets faces and points in packed order."""
import numpy as np
import pytest
import torch

import _gpu as G
import _scenes as SC
from paper_2007_08501_gb300 import ops

pytestmark = pytest.mark.gpu


def _depths(kind, n, rng):
    z = {"mixed": lambda: rng.uniform(1.0, 3.0, n), "flat": lambda: np.full(n, 2.0),
         "levels": lambda: 1.0 + rng.integers(0, 5, n) / 4.0}[kind]()
    z[n // 2], z[n // 3] = 0.2, 60.0
    return z


@pytest.mark.parametrize("kind,n,K,blur,clip", [
    ("mixed", 32_768, 1, 0.0, False), ("mixed", 32_769, 8, 1e-3, True), ("levels", 40_961, 5, 1e-3, True),
    ("flat", 50_000, 3, 0.0, False), ("mixed", 70_001, 8, 1e-3, True), ("mixed", 33_000, 24, 1e-3, True),
    ("levels", 40_000, 50, 0.0, False), ("mixed", 40_000, 24, 1e-3, False), ("mixed", 40_000, 16, 1e-3, False), ("mixed", 17_000, 4, 1e-3, True)])
def test_long_face_lists_match_the_plain_form(kind, n, K, blur, clip):
    rng = np.random.default_rng(n + K)
    z = _depths(kind, n, rng)[:, None] * np.ones(3)
    p = rng.uniform(-0.3, 0.3, (n, 1, 2)) + rng.uniform(-0.05, 0.05, (n, 3, 2))
    verts = np.concatenate([p * z[..., None], z[..., None]], -1).reshape(-1, 3)
    d = G.to_dev(dict(verts=verts, faces=np.arange(3 * n, dtype=np.int64).reshape(-1, 3),
                      first_face=np.array([0], np.int64), num_faces=np.array([n], np.int64),
                      cams=SC.identity_cam()[None]))
    S = 20
    ref, _, _, _ = G.gpu_fwd(d, S, K, blur, bin_size=0, clip=clip)
    for bin_size in (8, 16):
        out, status, _, _ = G.gpu_fwd(d, S, K, blur, bin_size=bin_size, clip=clip, max_faces_per_bin=n)
        assert status == 0
        for a, b in zip(out, ref):
            assert torch.equal(a, b)


@pytest.mark.parametrize("kind,n,K,radius", [
    ("mixed", 32_768, 4, 0.05), ("mixed", 32_769, 10, 0.02), ("levels", 40_961, 50, 0.1), ("flat", 50_000, 3, 0.9),
    ("mixed", 70_001, 50, 0.03), ("levels", 300_000, 1, 0.02), ("mixed", 131_073, 64, 0.02)])
def test_long_point_lists_match_the_plain_form(kind, n, K, radius):
    rng = np.random.default_rng(3 * n + K)
    z = _depths(kind, n, rng)
    xy = rng.uniform(-0.3, 0.3, (n, 2))
    pts = torch.from_numpy(np.concatenate([xy * z[:, None], z[:, None]], 1).astype(np.float32)).cuda()
    cams = torch.from_numpy(SC.identity_cam()[None].astype(np.float32)).cuda()
    first, num = torch.zeros(1, dtype=torch.int64).cuda(), torch.tensor([n]).cuda()
    S = 20

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
