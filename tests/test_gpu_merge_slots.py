"""The merge's split of a head's slots over warps: slot counts on both sides of every line between 1, 2, 4 and 8 warps per head and
of the 32 slots that a warp takes at once, numbers of heads that do not fill a CTA, slots not in use whose rows hold NaN."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workloads
from test_gpu_parity import iq, torch  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d", (128, 256))
@pytest.mark.parametrize("S", (1, 8, 9, 16, 17, 32, 33, 64, 65, 256, 257))
def test_slots_per_warp(iq, torch, S, d):  # noqa: F811
    B, H_q, H_kv = 3, 5, 1
    g = np.random.default_rng(100 * S + d)
    pa = g.standard_normal((B, H_q, S, d)).astype(np.float32)
    pm = np.stack([g.standard_normal((B, H_q, S)) * 3, g.uniform(0.5, 40, (B, H_q, S))], -1).astype(np.float32)
    pg = g.integers(0, 10000, (B, H_q, S)).astype(np.int32)
    unused = g.random((B, H_q, S)) < 0.4
    unused[0, 0] = True                      # a head without a slot in use
    unused[1, 1] = False
    unused[2, 2, :] = True
    unused[2, 2, S - 1] = False              # one with the last only
    pm[unused] = (-np.inf, 0)
    pg[unused] = -1
    quats = workloads.quaternion_pairs(g, H_kv, d)
    ref = oracle.combine_splits(quats, np.where(unused[..., None], 0, pa).astype(np.float32), pm, pg, H_kv)
    pa[unused] = np.nan                      # rows of slots that are not in use are not written
    shape = iq.Shape(B, H_q, H_kv, d, 128)
    rot = torch.empty(iq.iq_rotation_floats(d, H_kv), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H_kv, 0, np.ascontiguousarray(quats), rot)
    out = torch.empty((B, H_q, d), dtype=torch.float32, device="cuda")
    lse = torch.empty((B, H_q), dtype=torch.float32, device="cuda")
    am = torch.empty((B, H_q), dtype=torch.int32, device="cuda")
    tt = lambda a: torch.from_numpy(a).cuda()  # noqa: E731
    iq.iq_combine_splits(shape, rot, S, tt(pa), tt(pm), tt(pg), out, lse, am)
    # S + 64 roundings of 2^-24 (sums, weights, rotation) of rows below 5 per coordinate; an orthogonal map spreads the error over d
    tol = np.sqrt(d) * (S + 64) * 2.0 ** -24 * 5
    assert np.max(np.abs(out.cpu().numpy() - ref["out"])) <= tol
    assert np.allclose(lse.cpu().numpy(), ref["lse"], atol=1e-4)
    assert np.array_equal(am.cpu().numpy(), ref["argmax"]) and am[0, 0].item() == -1
