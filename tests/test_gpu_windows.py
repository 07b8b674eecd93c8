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
