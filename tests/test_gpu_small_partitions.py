"""The decode kernel's two ways to cut a launch into ranges: launches with little work give every item its own pieces of
whole CTAs, larger ones share the blocks out whatever item they belong to. Ragged batches on both sides of the line and
at its edges (one block, one block more than a piece, items with fewer pieces than others, empty sequences between them,
as many items as CTAs and one more), with and without the append in the launch, against the oracle."""
from __future__ import annotations

import numpy as np
import pytest

import workloads
from helpers import cache_to_numpy, check_decode, codebook_for, gpu_decode, gpu_quantize
from test_gpu_parity import iq, torch  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu

CASES = [  # (lens, query heads, KV heads, head_dim, splits)
    ([1], 4, 1, 128, 8), ([128], 4, 1, 128, 8), ([129], 4, 1, 128, 8), ([1024], 4, 1, 128, 8), ([1153], 8, 2, 128, 64),
    ([0, 700, 0, 0, 3, 129, 513], 8, 2, 128, 12), ([2048, 100, 1, 1025], 2, 1, 256, 32), ([600, 0, 1800], 20, 2, 128, 20),
    ([130] * 147, 1, 1, 128, 8), ([130] * 148, 1, 1, 128, 8), ([130] * 149, 1, 1, 128, 8), ([257] * 74, 2, 2, 256, 4),
    ([5] * 700 + [0] * 5 + [400], 1, 1, 128, 16), ([4096, 4000, 3000], 16, 2, 128, 40),
]


@pytest.mark.parametrize("i", range(len(CASES)))
def test_partitions_of_small_launches(iq, torch, codebooks, i):  # noqa: F811
    lens, H_q, H_kv, d, splits = CASES[i]
    lens = np.asarray(lens, np.int32)
    B = len(lens)
    w = workloads.tiny(700 + i, B, H_q, H_kv, d, max(1, int(lens.max())), lens=lens)
    lv, th = codebooks[d]
    cb = codebook_for(iq, codebooks, d)
    shape, rot, cache, _ = gpu_quantize(iq, torch, w, cb, n_new=lens)
    g = cache_to_numpy(cache)
    res = gpu_decode(iq, torch, shape, rot, cb, w.q, cache, lens, splits)
    check_decode(w, lv, w.q, res, g, lens)
