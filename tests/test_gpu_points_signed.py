"""Points on both sides of the camera plane (znear below 0 culls neither): the
binned form ranks negative depths in front of positive ones as the plain form
does, bit for bit."""
import numpy as np
import pytest
import torch

import _scenes as SC
from paper_2007_08501_gb300 import ops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sides", ["behind", "both"])
@pytest.mark.parametrize("n,K,radius", [(20, 4, 0.3), (600, 3, 0.9), (1025, 50, 0.02), (5000, 16, 0.3)])
def test_depths_of_either_sign_match_the_plain_form(sides, n, K, radius):
    rng = np.random.default_rng(n + K)
    z = rng.uniform(0.5, 3.0, n) * (-1.0 if sides == "behind" else rng.choice([-1.0, 1.0], n))
    xy = rng.uniform(-0.5, 0.5, (n, 2))
    pts = torch.from_numpy(np.concatenate([xy * z[:, None], z[:, None]], 1).astype(np.float32)).cuda()
    cam = SC.identity_cam()
    cam[13] = -10.0
    cams = torch.from_numpy(cam[None].astype(np.float32)).cuda()
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
    assert int((ref[0] >= 0).sum()) > n // 4
    for bin_size in (8, 16):
        for a, b in zip(run(bin_size), ref):
            assert torch.equal(a, b)
