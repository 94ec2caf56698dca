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


def _merge(iq, torch, g, B, H_q, S1, d, shards=1):  # noqa: F811
    """Random partials of `shards` x S1 slots with equal maxima in the first and the last slot in use of every head (the lower row in
    the last) and NaN rows in the others, merged by the library and by the oracle over the slots side by side."""
    S = S1 * shards
    pa = g.standard_normal((B, H_q, S, d)).astype(np.float32)
    pm = np.stack([g.standard_normal((B, H_q, S)) * 3, g.uniform(0.5, 40, (B, H_q, S))], -1).astype(np.float32)
    row = g.integers(5000, 10000, (B, H_q, S)).astype(np.int32)      # rows of the whole sequence
    pm[..., 0, 0] = pm[..., S - 1, 0] = 20.0
    row[..., S - 1] = g.integers(4000, 5000, (B, H_q))
    unused = g.random((B, H_q, S)) < 0.4
    unused[..., 0] = unused[..., S - 1] = False
    pm[unused] = (-np.inf, 0)
    row[unused] = -1
    quats = workloads.quaternion_pairs(g, 1, d)
    ref = oracle.combine_splits(quats, np.where(unused[..., None], 0, pa).astype(np.float32), pm, row, 1)
    assert np.array_equal(ref["argmax"], row[..., S - 1])
    pa[unused] = np.nan
    shape = iq.Shape(B, H_q, 1, d, 128)
    rot = torch.empty(iq.iq_rotation_floats(d, 1), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, 1, 0, np.ascontiguousarray(quats), rot)
    out = torch.empty((B, H_q, d), dtype=torch.float32, device="cuda")
    lse = torch.empty((B, H_q), dtype=torch.float32, device="cuda")
    am = torch.empty((B, H_q), dtype=torch.int32, device="cuda")
    tt = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()  # noqa: E731
    if shards == 1:
        iq.iq_combine_splits(shape, rot, S, tt(pa), tt(pm), tt(row), out, lse, am)
    else:  # shard after shard, rows counted from the shard's first one of the sequence
        offs = g.integers(1, 4000, (shards, B)).astype(np.int32)
        rank = lambda a: np.moveaxis(a.reshape((B, H_q, shards, S1) + a.shape[3:]), 2, 0)  # noqa: E731
        local = rank(row) - np.where(rank(unused), 0, offs[:, :, None, None]).astype(np.int32)
        iq.iq_combine_splits_sharded(shape, rot, S1, shards, tt(rank(pa)), tt(rank(pm)), tt(local), tt(offs), out, lse, am)
    # S + 64 roundings of 2^-24 (sums, weights, rotation) of rows below 5 per coordinate; an orthogonal map spreads the error over d
    tol = np.sqrt(d) * (S + 64) * 2.0 ** -24 * 5
    assert np.max(np.abs(out.cpu().numpy() - ref["out"])) <= tol
    assert np.allclose(lse.cpu().numpy(), ref["lse"], atol=1e-4)
    assert np.array_equal(am.cpu().numpy(), ref["argmax"])


@pytest.mark.parametrize("d", (128, 256))
@pytest.mark.parametrize("B,H_q,S", [(3, 5, 9), (3, 5, 17), (3, 5, 33), (3, 5, 257), (16, 8, 17), (43, 3, 17), (43, 3, 32), (43, 3, 33),
                                     (64, 8, 9), (64, 8, 16), (27, 19, 9), (27, 19, 16)])
def test_equal_maxima_and_heads_on_both_sides_of_each_line(iq, torch, B, H_q, S, d):  # noqa: F811
    """The lowest row wins a tie between slots of different warps; 128 and 129 heads at 17 - 33 slots, 512 and 513 at 9 - 16."""
    _merge(iq, torch, np.random.default_rng(1000 * S + B), B, H_q, S, d)


@pytest.mark.parametrize("d", (128, 256))
@pytest.mark.parametrize("shards,S1", [(3, 3), (3, 5), (3, 7), (3, 13), (5, 13), (3, 86)])
@pytest.mark.parametrize("B,H_q", [(3, 5), (43, 3)])
def test_shards_whose_slots_straddle_warps(iq, torch, B, H_q, shards, S1, d):  # noqa: F811
    """9 - 258 slots of three and five shards: runs of a warp that begin and end inside a shard, rows counted from the shard's first."""
    _merge(iq, torch, np.random.default_rng(100 * S1 + B), B, H_q, S1, d, shards)
