"""Reconstruction on the tensor cores (levels that are binary16 values times one factor per side) and by the general kernel
(any other levels) against the oracle's dense R^T: block edges, every bit width, a K and a V codebook of different forms,
an output shorter than the longest sequence."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workloads
from helpers import cache_to_numpy
from test_gpu_bits import iq, torch, two_codebooks  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("form", ["8-bit grid", "binary16 keys, 8-bit grid values", "other levels"])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("d", [128, 256])
def test_reconstructed_rows_at_block_edges(iq, torch, d, bits, form):  # noqa: F811
    lens, T_out, H = np.array([1, 127, 0, 128, 129, 300], np.int32), 290, 3
    w = workloads.tiny(860 + bits, len(lens), H, H, d, 300, lens=lens)
    lv, th, lvv, thv = two_codebooks(d, bits, "int8")
    if form.startswith("binary16"):
        lv, th = two_codebooks(d, bits, "fp16", False)[:2]
    if form.startswith("other"):
        lvv = (lvv.astype(np.float64) * 1.0001 + 1e-3).astype(np.float32)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)), tuple(map(float, lvv)), tuple(map(float, thv)))
    shape = iq.Shape(len(lens), H, H, d, w.t_cap, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 0, np.ascontiguousarray(w.quats), rot)
    cache = iq.new_cache(shape)
    lens_dev = torch.from_numpy(lens).cuda()
    iq.iq_quantize_append(shape, rot, cb, torch.from_numpy(w.k).cuda(), torch.from_numpy(w.v).cuda(),
                          torch.zeros(len(lens), dtype=torch.int32, device="cuda"), lens_dev, 300, cache)
    kv = torch.full((len(lens), T_out, H, 2 * d), 7.0, dtype=torch.float16, device="cuda")
    iq.iq_reconstruct_rows(shape, rot, cb, cache, lens_dev, kv[..., :d], kv[..., d:])
    torch.cuda.synchronize()
    K, V = oracle.reconstruct_rows(w.quats, lv, cache_to_numpy(cache), lens, H, levels_v=lvv, d=d)
    for got, ref in ((kv[..., :d].cpu().numpy().astype(np.float64), K), (kv[..., d:].cpu().numpy().astype(np.float64), V)):
        for b in range(len(lens)):
            n = min(int(lens[b]), T_out)
            assert np.all(got[b, n:] == 7.0)
            if n:
                r = ref[b, :n]   # one rounding to binary16 and fp32 sums: the bound of the parity test of the general kernel
                assert np.all(np.abs(got[b, :n] - r) <= 2.0 ** -11 * 1.001 * np.abs(r) + 1e-5 * np.abs(r).max(axis=-1, keepdims=True) + 2.0 ** -25)


@pytest.mark.parametrize("d", [128, 256])
def test_a_wait_that_gives_up_leaves_no_ordinary_rows(iq, torch, d):  # noqa: F811
    """A limit of 0 polls: every group gives up on its first tile and owes the rest of its share. The rows are NaN and not
    the numbers of an unfinished product, rows past the lengths stay, the next call is an ordinary one."""
    lens, H = [3000, 0, 129, 1500], 4
    B, T = len(lens), max(lens)
    shape = iq.Shape(B, H, H, d, 3072)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 5, None, rot)
    cb, cache = iq.iq_lloyd_max_codebook(d, 3, "int8"), iq.new_cache(shape)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d)
    k, v = (torch.randn((B, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    lens_dev = torch.tensor(lens, dtype=torch.int32, device="cuda")
    iq.iq_quantize_append(shape, rot, cb, k, v, torch.zeros_like(lens_dev), lens_dev, T, cache)
    outs = {}
    for polls in (65536, 0, None):
        ko, vo = (torch.full((B, T, H, d), 7.0, dtype=torch.float16, device="cuda") for _ in range(2))
        if polls is None:
            iq.iq_reconstruct_rows(shape, rot, cb, cache, lens_dev, ko, vo)
        else:
            iq.iq_selftest_reconstruct_wait(shape, rot, cb, cache, lens_dev, ko, vo, polls)
        outs[polls] = (ko, vo)
    torch.cuda.synchronize()
    for side in range(2):
        for b, n in enumerate(lens):
            assert torch.isnan(outs[0][side][b, :n]).all() and (outs[0][side][b, n:] == 7.0).all()
        assert torch.equal(outs[65536][side], outs[None][side]) and not torch.isnan(outs[None][side]).any()


@pytest.mark.parametrize("form", ["int8", "fp16"])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("d", [128, 256])
def test_error_before_the_rounding_is_that_of_fp32(iq, torch, d, bits, form):  # noqa: F811
    """Rows with outlier channels: beyond the rounding to binary16 an element is off by the fp32 operations on it (the cuts of
    the sum as it grows, the factors: 2^-22 of it) and by the lower term of W, rounded at 2^-23: sigma 2^-23 / sqrt(3) of the
    row's rms, 6e-7 is more than eight sigma."""
    B, H, T = 1, 2, 1024
    shape = iq.Shape(B, H, H, d, T, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 3, None, rot)
    cb, cache = iq.iq_lloyd_max_codebook(d, bits, form), iq.new_cache(shape)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + bits)
    k, v = (torch.randn((B, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    k[..., :4] *= 20
    v[..., 7:11] *= 20
    lens = torch.full((B,), T, dtype=torch.int32, device="cuda")
    iq.iq_quantize_append(shape, rot, cb, k, v, torch.zeros_like(lens), None, T, cache)
    ko, vo = torch.empty_like(k), torch.empty_like(v)
    iq.iq_reconstruct_rows(shape, rot, cb, cache, lens, ko, vo)
    torch.cuda.synchronize()
    refs = oracle.reconstruct_rows(rot.cpu().numpy().reshape(H, d // 4, 8), np.array(cb.levels, np.float32), cache_to_numpy(cache),
                                   np.array([T], np.int32), H, d=d)
    for got, ref in zip((ko, vo), refs):
        r = np.asarray(ref)[:, :T]
        err = np.abs(got.cpu().numpy().astype(np.float64) - r)
        rms = np.sqrt((r ** 2).mean(axis=-1, keepdims=True))
        beyond = err - 0.5 * np.spacing(np.abs(r).astype(np.float16)).astype(np.float64)
        assert np.all(beyond <= 2.0 ** -22 * np.abs(r) + 6e-7 * rms), float((beyond / (2.0 ** -22 * np.abs(r) + 6e-7 * rms)).max())


@pytest.mark.parametrize("d", [128, 256])
def test_levels_off_the_grid_by_an_fp32_place_are_used_as_they_are(iq, torch, d):  # noqa: F811
    """Identity blocks and a row of equal codes: its first element is scale * level. The level 1 + 2^-11 + 2^-23 is one place
    above a multiple of the grid and rounds to 1 + 2^-10 in binary16, the multiple (a tie) to 1."""
    f = np.float32(2049 / 2 ** 17)
    level = np.float32(1 + 2.0 ** -11 + 2.0 ** -23)
    lv = (-127 * float(f), 3 * float(f), float(level), 127 * float(f))
    cb = iq.Codebook(lv, (-1.0, 0.5, 1.5))
    shape = iq.Shape(1, 1, 1, d, 128, bits=2)
    rot = torch.empty(iq.iq_rotation_floats(d, 1), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, 1, 0, np.tile(np.array([1, 0, 0, 0, 1, 0, 0, 0], np.float32), (1, d // 4, 1)), rot)
    cache = iq.new_cache(shape)
    for codes, scales in ((cache.k_codes, cache.k_scales), (cache.v_codes, cache.v_scales)):
        codes.fill_(0xAA)   # code 2 everywhere
        scales.fill_(1.0)
    ko, vo = (torch.zeros((1, 128, 1, d), dtype=torch.float16, device="cuda") for _ in range(2))
    iq.iq_reconstruct_rows(shape, rot, cb, cache, torch.tensor([128], dtype=torch.int32, device="cuda"), ko, vo)
    torch.cuda.synchronize()
    for o in (ko, vo):
        assert (o[..., 0] == 1 + 2.0 ** -10).all() and (o[..., 1:] == 0).all()


def _against_the_oracle(iq, torch, d, bits, form, H, T, table_of, lens):  # noqa: F811
    """Five sequences of T rows in a scattered pool of 128-row pages; sequence b of the call reads the pages of sequence
    table_of[b], lens[b] rows."""
    t_cap = (T + 127) // 128 * 128
    pages = np.random.default_rng(d + bits).permutation(5 * (t_cap // 128)).astype(np.int32).reshape(5, -1)
    part, shape = (iq.Shape(n, H, H, d, t_cap, bits=bits) for n in (5, len(lens)))
    cb = iq.iq_lloyd_max_codebook(d, bits, form)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 8, None, rot)
    pool, whole = iq.new_paged_cache(part, pages.size, 128, torch.from_numpy(pages).cuda()), iq.new_cache(part)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + bits)
    k, v = (torch.randn((5, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    for c in (pool, whole):   # (contiguous for the oracle)
        iq.iq_quantize_append(part, rot, cb, k, v, torch.zeros(5, dtype=torch.int32, device="cuda"), None, T, c)
    cache = iq.Cache(pool.k_codes, pool.k_scales, pool.v_codes, pool.v_scales, torch.from_numpy(pages[table_of]).cuda(), 128)
    ko, vo = (torch.full((len(lens), T, H, d), 7.0, dtype=torch.float16, device="cuda") for _ in range(2))
    iq.iq_reconstruct_rows(shape, rot, cb, cache, torch.tensor(lens, dtype=torch.int32, device="cuda"), ko, vo)
    torch.cuda.synchronize()
    refs = oracle.reconstruct_rows(rot.cpu().numpy().reshape(H, d // 4, 8), np.array(cb.levels, np.float32), cache_to_numpy(whole),
                                   np.full(5, T, np.int32), H, d=d)
    for out, ref in zip((ko, vo), refs):
        want = torch.from_numpy(np.ascontiguousarray(np.asarray(ref)[:, :T])).cuda()
        bound = 2.0 ** -11 * 1.001 * want.abs() + 1e-5 * want.abs().amax(dim=-1, keepdim=True) + 2.0 ** -25
        for b, n in enumerate(lens):
            assert (out[b, n:] == 7.0).all()
            assert ((out[b, :n].double() - want[table_of[b], :n]).abs() <= bound[table_of[b], :n]).all(), b


@pytest.mark.parametrize("form", ["int8", "fp16"])
@pytest.mark.parametrize("d,bits", [(128, 2), (128, 3), (128, 4), (256, 2), (256, 3), (256, 4)])
def test_many_tiles_per_group(iq, torch, d, bits, form):  # noqa: F811
    """Enough 128-row tiles that every group of every CTA takes at least four, one after the other, K and then V, and goes on
    to another head: buffers, accumulators and barrier phases are used again."""
    groups = (4 if d == 128 else 2) * torch.cuda.get_device_properties(0).multi_processor_count
    H = 3
    T = 128 * -(-4 * groups // (2 * H * 4))
    _against_the_oracle(iq, torch, d, bits, form, H, T, [3, 0, 4, 1, 2], [T, T - 1, T - 127, T - 300, T])


@pytest.mark.parametrize("d,bits", [(128, 3), (256, 4)])
def test_more_sequences_than_threads_of_a_cta(iq, torch, d, bits):  # noqa: F811
    lens = [(b * 37) % 300 * (b % 3 != 1) for b in range(1100)]
    _against_the_oracle(iq, torch, d, bits, "int8", 1, 300, [b % 5 for b in range(1100)], lens)
