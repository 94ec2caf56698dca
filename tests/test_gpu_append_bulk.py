"""The bulk append kernel (Algorithm 1 on the tensor cores) against the warp-per-row kernel that calls of a few rows
take, byte for byte, and against the oracle: tile edges (first and last rows inside 128-row blocks), every bit width, both
forms of the decision (thresholds symmetric about zero or not), two codebooks, strided inputs, paged caches, binary16
scales, rows whose coordinates all sit on a threshold, zero rows, rows that end a sequence outside the cache."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import workloads
from helpers import cache_to_numpy
from test_gpu_bits import compare_codes, iq, torch, two_codebooks  # noqa: F401 (fixtures)

pytestmark = pytest.mark.gpu


def _append(iq, torch, shape, rot, cb, k, v, first, lens, rows, page_rows, scales):
    """The rows of k, v appended `rows` at a time into a cache whose bytes are not zero to begin with."""
    B, T = k.shape[:2]
    if page_rows:
        n = B * (shape.t_cap // page_rows)
        table = torch.arange(n - 1, -1, -1, dtype=torch.int32, device="cuda").reshape(B, -1).contiguous()
        cache = iq.new_paged_cache(shape, n, page_rows, table, scales_dtype=scales)
    else:
        cache = iq.new_cache(shape, scales_dtype=scales)
    for a in (cache.k_codes, cache.v_codes):
        a.fill_(0x5A)
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    for i in range(0, T, rows):
        n = [int(min(max(x - i, 0), rows)) for x in lens]
        iq.iq_quantize_append(shape, rot, cb, k[:, i:i + rows], v[:, i:i + rows], torch.tensor([f + i for f in first], dtype=torch.int32, device="cuda"),
                              torch.tensor(n, dtype=torch.int32, device="cuda"), min(rows, T - i), cache, status)
    torch.cuda.synchronize()
    return cache, status.cpu().numpy()


@pytest.mark.parametrize("d", [128, 256])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("variant", ["symmetric", "shifted", "two codebooks, paged, binary16 scales"])
def test_bulk_append_equals_the_row_kernel(iq, torch, bits, d, variant):  # noqa: F811
    B, H, T, t_cap = 5, 3, 300, 512
    first, lens = [0, 3, 127, 128, 400], [300, 125, 129, 5, 200]   # sequence 4 runs past t_cap
    lv, th, lvv, thv = two_codebooks(d, bits, "int8", variant.startswith("two"))
    if variant == "shifted":
        th = (th.astype(np.float64) + 0.01 * ((np.arange(len(th)) * 7) % 5 - 2)).astype(np.float32)
        thv = th
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)), tuple(map(float, lvv)), tuple(map(float, thv)))
    shape = iq.Shape(B, H, H, d, t_cap, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 11 + bits, None, rot)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + bits)
    kv = torch.randn((B, T, H, 2 * d), generator=gen, device="cuda").half()
    kv[..., ::37] *= 20
    kv[:, 2::11] = 0                    # zero rows
    kv[:, 5::13] = 1                    # all but four coordinates exactly on a threshold at zero: more than a warp's list takes
    kv[:, 7::17, :, 1:] = 0             # one element
    kv[:, 9::19] *= 1e-4                # subnormal elements
    k, v = kv[..., :d], kv[..., d:]     # strided
    page_rows, scales = (128, torch.float16) if variant.startswith("two") else (0, torch.float32)
    bulk, st = _append(iq, torch, shape, rot, cb, k, v, first, lens, T, page_rows, scales)
    rows, st_rows = _append(iq, torch, shape, rot, cb, k, v, first, lens, 4, page_rows, scales)
    for name in ("k_codes", "v_codes", "k_scales", "v_scales"):
        a, b = getattr(bulk, name), getattr(rows, name)
        assert torch.equal(a, b), f"{name}: {int((a != b).sum())} of {a.numel()} differ"
    assert st[0] == st_rows[0] == 1 and st[2] == st_rows[2] == 88 * H * 2


@pytest.mark.parametrize("n", [5, 64, 127, 128, 129, 257])
@pytest.mark.parametrize("d,bits", [(128, 3), (256, 4)])
def test_bulk_append_codes_match_the_oracle(iq, torch, d, bits, n):  # noqa: F811
    w = workloads.tiny(840 + n, 1, 2, 2, d, n, lens=[n])
    lv, th, _, _ = two_codebooks(d, bits, "int8", False)
    shape = iq.Shape(1, 2, 2, d, w.t_cap, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, 2), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, 2, 0, np.ascontiguousarray(w.quats), rot)
    cache, status = iq.new_cache(shape), torch.zeros(4, dtype=torch.int32, device="cuda")
    iq.iq_quantize_append(shape, rot, iq.Codebook(tuple(map(float, lv)), tuple(map(float, th))), torch.from_numpy(w.k).cuda(),
                          torch.from_numpy(w.v).cuda(), torch.zeros(1, dtype=torch.int32, device="cuda"), None, n, cache, status)
    torch.cuda.synchronize()
    ref = oracle.new_cache(1, 2, d, w.t_cap, bits)
    oracle.quantize_append(w.quats, th, w.k, w.v, np.zeros(1, np.int32), np.array([n], np.int32), ref, thresholds_v=th)
    assert status[0] == 0 and status[2] == 0
    compare_codes(w, bits, th, th, cache_to_numpy(cache), ref, [n])


def test_codebook_with_close_thresholds_keeps_its_path(iq, torch):  # noqa: F811
    """Thresholds 1e-5 apart cannot be told apart by the bulk kernel's saturating sums: such a call is decided in another way
    and gives what calls of four rows give."""
    d, T = 128, 200
    lv, th, _, _ = two_codebooks(d, 3, "int8", False)
    th = th.copy()
    th[4] = th[3] + np.float32(1e-5)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)))
    shape = iq.Shape(1, 1, 1, d, 256)
    rot = torch.empty(iq.iq_rotation_floats(d, 1), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, 1, 1, None, rot)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(1)
    k, v = (torch.randn((1, T, 1, d), generator=gen, device="cuda").half() for _ in range(2))
    a, _ = _append(iq, torch, shape, rot, cb, k, v, [0], [T], T, 0, torch.float32)
    b, _ = _append(iq, torch, shape, rot, cb, k, v, [0], [T], 4, 0, torch.float32)
    assert torch.equal(a.k_codes, b.k_codes) and torch.equal(a.v_codes, b.v_codes)


@pytest.mark.parametrize("d", [128, 256])
def test_a_wait_that_gives_up_is_reported(iq, torch, d):  # noqa: F811
    """A limit of 0 polls for the tensor-core results: the flag is set, the call returns within the limit of the other waits,
    rows that it was not to append stay, and the next call over the same rows is an ordinary one."""
    B, H, T = 3, 2, 700
    shape = iq.Shape(B, H, H, d, 1024)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 5, None, rot)
    cb = iq.iq_lloyd_max_codebook(d, 3, "int8")
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d)
    k, v = (torch.randn((B, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    caches = [iq.new_cache(shape) for _ in range(2)]
    for c in caches:
        c.k_codes.fill_(0x5A)
        c.k_scales.fill_(3.0)
    pos = torch.tensor([0, 100, 250], dtype=torch.int32, device="cuda")
    status = torch.zeros(4, dtype=torch.int32, device="cuda")
    iq.iq_selftest_append_wait(shape, rot, cb, k, v, pos, None, T, caches[0], status, 0)
    torch.cuda.synchronize()
    assert int(status[0]) == 2
    for b, p in enumerate(pos.tolist()):
        for a in (caches[0].k_codes, caches[0].k_scales):
            outside = torch.cat([a[b, :, :p], a[b, :, p + T:]], dim=1)
            assert (outside == (0x5A if a is caches[0].k_codes else 3.0)).all()
    status.zero_()
    for c in caches:
        iq.iq_quantize_append(shape, rot, cb, k, v, pos, None, T, c, status)
    torch.cuda.synchronize()
    assert int(status[0]) == 0
    assert torch.equal(caches[0].k_codes, caches[1].k_codes) and torch.equal(caches[0].k_scales, caches[1].k_scales)
    for b, p in enumerate(pos.tolist()):   # whole new blocks of V
        lo, hi = (p + 127) // 128, (p + T) // 128
        va, vb = (c.v_codes.reshape(B, H, 8, -1)[b, :, lo:hi] for c in caches)
        assert torch.equal(va, vb)


@pytest.mark.parametrize("d", [128, 256])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("grid", ["symmetric", "shifted"])
def test_rows_that_are_not_finite(iq, torch, bits, d, grid):  # noqa: F811
    """Rows with an infinity or a NaN in a prompt: code 0 everywhere and a norm that is not finite, as in calls of up to four
    rows; the rows next to them in the same tile as if they were not there."""
    B, H, T = 1, 2, 260
    lv, th, _, _ = two_codebooks(d, bits, "int8", False)
    if grid == "shifted":
        th = (th.astype(np.float64) + 0.01 * ((np.arange(len(th)) * 7) % 5 - 2)).astype(np.float32)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)))
    shape = iq.Shape(B, H, H, d, 384, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 2, None, rot)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + bits)
    k, v = (torch.randn((B, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    bad = {0: float("inf"), 5: float("nan"), 64: float("-inf"), 127: float("nan"), 128: float("inf"), 259: float("-inf")}
    plain_k, plain_v = k.clone(), v.clone()
    for r, x in bad.items():
        for a in (k, v):
            a[:, r, :, r % d] = x
        if r == 64:
            k[:, r, :, 1] = float("inf")   # two infinities of opposite sign
    whole, _ = _append(iq, torch, shape, rot, cb, k, v, [0], [T], T, 0, torch.float32)
    rows, _ = _append(iq, torch, shape, rot, cb, k, v, [0], [T], 4, 0, torch.float32)
    plain, _ = _append(iq, torch, shape, rot, cb, plain_k, plain_v, [0], [T], T, 0, torch.float32)
    good = [r for r in range(T) if r not in bad]
    for h in range(H):
        for name in ("k_codes", "v_codes", "k_scales", "v_scales"):
            a, b, c = (cache_to_numpy(x)[name][0, h] for x in (whole, rows, plain))
            if name.endswith("scales"):
                assert np.array_equal(a.view(np.int32)[good], c.view(np.int32)[good]) and not np.isfinite(a[list(bad)]).any()
                assert np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.isinf(a), np.isinf(b))
                continue
            codes = [[oracle.unpack_row(d, x[r], bits) if name == "k_codes" else oracle.v_row_codes(d, x, r, bits) for r in range(T)] for x in (a, b, c)]
            codes = np.array(codes)
            assert np.array_equal(codes[0][good], codes[2][good]) and np.array_equal(codes[0], codes[1])
            assert (codes[0][list(bad)] == 0).all()


@pytest.mark.parametrize("d", [128, 256])
@pytest.mark.parametrize("bits", [2, 3, 4])
def test_each_row_that_is_decided_again_counts_once(iq, torch, bits, d):  # noqa: F811
    """status[1] of a prompt: the rows with a coordinate at a threshold (here: constant rows, 0 everywhere but in one block,
    and zero rows), one each per KV head and tensor, as calls of four rows count them. Other rows have no coordinate within
    2e-4 of a threshold, more than any band."""
    B, H, T = 2, 2, 700
    lv, th, _, _ = two_codebooks(d, bits, "int8", False)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)))
    shape = iq.Shape(B, H, H, d, 768, bits=bits)
    rng = np.random.default_rng(d + bits)
    q8 = rng.standard_normal((H, d // 4, 8)).astype(np.float32)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 0, q8, rot)
    W = [oracle.rotation_matrix(d, q) * np.sqrt(d) for q in q8]
    x = rng.standard_normal((2, B, T, H, d)).astype(np.float16)
    near = np.zeros((2, B, T, H), bool)
    for h in range(H):
        for _ in range(400):   # rows with a coordinate near a threshold are drawn again
            u = x[:, :, :, h].astype(np.float64) @ W[h].T / np.linalg.norm(x[:, :, :, h].astype(np.float64), axis=-1, keepdims=True)
            bad = np.zeros(u.shape[:-1], bool)
            for t in th:
                bad |= (np.abs(u - float(t)) < 2e-4).any(axis=-1)
            if not bad.any():
                break
            x[:, :, :, h][bad] = rng.standard_normal((int(bad.sum()), d)).astype(np.float16)
        assert not bad.any()
    x[:, :, 3::50] = 1
    x[:, :, 7::90] = 0
    near[:, :, 3::50] = near[:, :, 7::90] = True
    k, v = (torch.from_numpy(a).cuda() for a in x)
    _, whole = _append(iq, torch, shape, rot, cb, k, v, [0, 30], [T, T], T, 0, torch.float32)
    _, rows = _append(iq, torch, shape, rot, cb, k, v, [0, 30], [T, T], 4, 0, torch.float32)
    assert whole[0] == rows[0] == 0 and whole[1] == rows[1] == int(near.sum())


@pytest.mark.parametrize("d,bits", [(128, 2), (128, 3), (128, 4), (256, 2), (256, 3), (256, 4)])
def test_rows_built_against_the_band(iq, torch, d, bits):  # noqa: F811
    """Rows along a row of W up to some element and against it from there, so that the running sum is as large as it can be
    and comes back to a threshold: the nearest of 3000 variants on either side of it, and some a few 1e-6 to 1e-4 away. Every
    code of every row is that of an fp64 evaluation."""
    lv, th, _, _ = two_codebooks(d, bits, "int8", False)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)))
    rng = np.random.default_rng(d + bits)
    q8 = rng.standard_normal((1, d // 4, 8)).astype(np.float32)
    W = oracle.rotation_matrix(d, q8[0]) * np.sqrt(d)
    rows = []
    for case in range(80):
        w, t = W[rng.integers(d)], float(th[case % len(th)])
        m = int(d * rng.uniform(0.3, 0.95))
        A, Bq, Cq = m + m * m / (d - m), -2 * t * m / (d - m), t * t / (d - m) - 1   # |x| = 1, <w, x> = t
        a = (-Bq + np.sqrt(Bq * Bq - 4 * A * Cq)) / (2 * A)
        x = w * np.where(np.arange(d) < m, a, (t - a * m) / (d - m)) * rng.uniform(8, 64)
        x = (x * (1 + 0.003 * rng.standard_normal((3000, d)))).astype(np.float16)
        dist = x.astype(np.float64) @ w / np.linalg.norm(x.astype(np.float64), axis=1) - t
        for side in (1, -1):
            order = np.argsort(np.where(side * dist > 1e-9, np.abs(dist), np.inf))
            rows += [x[i] for i in order[:3]]
            for far in (3e-6, 1e-5, 3e-5, 1e-4):
                rows.append(x[np.argmin(np.abs(side * dist - far))])
    x = np.array(rows)
    T = len(x)
    shape = iq.Shape(1, 1, 1, d, (T + 127) // 128 * 128, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, 1), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, 1, 0, q8, rot)
    W = oracle.rotation_matrix(d, rot.cpu().numpy()) * np.sqrt(d)
    k = torch.from_numpy(x).cuda().reshape(1, T, 1, d)
    cache, _ = _append(iq, torch, shape, rot, cb, k, k, [0], [T], T, 0, torch.float32)
    x = x.astype(np.float64)
    u = x @ W.T / np.linalg.norm(x, axis=1, keepdims=True)
    gap = u[..., None] - th.astype(np.float64)
    want, tie = (gap > 0).sum(axis=-1), (np.abs(gap) < 1e-12).any(axis=-1)
    g = cache_to_numpy(cache)
    for got in ([oracle.unpack_row(d, g["k_codes"][0, 0, r], bits) for r in range(T)], [oracle.v_row_codes(d, g["v_codes"][0, 0], r, bits) for r in range(T)]):
        assert np.all((np.array(got) == want) | tie), int(((np.array(got) != want) & ~tie).sum())


@pytest.mark.parametrize("d", [128, 256])
@pytest.mark.parametrize("form", ["a pair", "seven in a band", "across two bands", "out of reach"])
def test_three_bit_codebooks_with_close_or_far_thresholds(iq, torch, d, form):  # noqa: F811
    """Thresholds within one another's bands (2e-6 to 1e-4 apart, some of them around 0, where constant rows tie) and
    thresholds that no coordinate reaches: the bytes of calls of four rows."""
    B, H, T = 3, 2, 900
    lv, th, _, _ = two_codebooks(d, 3, "int8", False)
    th = th.astype(np.float64)
    if form == "a pair":
        th[4] = th[3] + 1e-5
    elif form == "seven in a band":
        th = 0.4 + 2e-6 * np.arange(7)
    elif form == "across two bands":
        th = np.array([-1.0, -2e-5, -1e-5, 0.0, 4e-5, 8e-5, 0.7])
    else:
        th = np.array([-1e30, -100.0, -1.0, 0.0, 1.0, 1e5, 3e38])
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th.astype(np.float32))))
    shape = iq.Shape(B, H, H, d, 1024)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 1, None, rot)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d)
    k, v = (torch.randn((B, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    k[:, 3::17], v[:, 5::29] = 1, 1
    a, sa = _append(iq, torch, shape, rot, cb, k, v, [0, 60, 100], [T, T - 1, 300], T, 0, torch.float32)
    b, sb = _append(iq, torch, shape, rot, cb, k, v, [0, 60, 100], [T, T - 1, 300], 4, 0, torch.float32)
    assert torch.equal(a.k_codes, b.k_codes) and torch.equal(a.v_codes, b.v_codes) and sa[0] == sb[0] == 0


@pytest.mark.parametrize("d", [128, 256])
@pytest.mark.parametrize("bits", [2, 3, 4])
@pytest.mark.parametrize("B,H", [(3, 2), (30, 5), (130, 4)])
def test_calls_on_both_sides_of_the_line_between_the_kernels(iq, torch, bits, d, B, H):  # noqa: F811
    """2 to 44 rows per sequence (the line lies between 10 and 42, by batch and head size), starting and ending inside words,
    units and blocks of the V records: the bytes of calls of one row."""
    lv, th, lvv, thv = two_codebooks(d, bits, "int8", True)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)), tuple(map(float, lvv)), tuple(map(float, thv)))
    shape = iq.Shape(B, H, H, d, 256, bits=bits)
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 4, None, rot)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + bits + B)
    T = 44
    k, v = (torch.randn((B, T, H, d), generator=gen, device="cuda").half() for _ in range(2))
    first = [(37 * b) % 190 for b in range(B)]
    lens = [T - (b % 5 == 3) * 7 for b in range(B)]
    ref, _ = _append(iq, torch, shape, rot, cb, k, v, first, lens, 1, 0, torch.float32)
    for rows in (2, 7, 10, 11, 20, 24, 25, 28, 29, 42, 43, 44):
        got, status = _append(iq, torch, shape, rot, cb, k, v, first, lens, rows, 0, torch.float32)
        for name in ("k_codes", "v_codes", "k_scales", "v_scales"):
            assert torch.equal(getattr(got, name), getattr(ref, name)), (rows, name)
        assert status[0] == 0 and status[2] == 0


@pytest.mark.parametrize("d,bits,variant", [(128, 2, "paged"), (128, 3, "shifted"), (128, 3, "binary16 scales"), (128, 4, "paged"), (128, 4, "shifted"),
                                            (256, 2, "shifted"), (256, 3, "paged"), (256, 4, "binary16 scales"), (256, 4, "shifted")])
def test_many_tiles_per_group(iq, torch, bits, d, variant):  # noqa: F811
    """Enough 128-row tiles that every group of every CTA takes several of a head one after the other and goes on to another
    head: buffers, accumulators and barrier phases are used again, lists and marks carry over tiles. Rows that tie throughout,
    rows with one element, zero rows; sequences that start and end inside blocks. Bytes of calls of four rows (the row kernel)."""
    sm = torch.cuda.get_device_properties(0).multi_processor_count
    B, H = 6, 7
    groups = 4 if d == 128 else 2
    T = 128 * -(-(4 * groups * sm) // (2 * B * H)) + 77     # at least four tiles per group
    shape = iq.Shape(B, H, H, d, (T + 300 + 127) // 128 * 128, bits=bits)
    lv, th, lvv, thv = two_codebooks(d, bits, "int8", True)
    if variant == "shifted":
        th = (th.astype(np.float64) + 0.01 * ((np.arange(len(th)) * 7) % 5 - 2)).astype(np.float32)
    cb = iq.Codebook(tuple(map(float, lv)), tuple(map(float, th)), tuple(map(float, lvv)), tuple(map(float, thv)))
    rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, 21, None, rot)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(d + bits)
    kv = torch.randn((B, T, H, 2 * d), generator=gen, device="cuda").half()
    kv[..., ::37] *= 20
    kv[:, 5::43] = 1
    kv[:, 400:437] = 1                    # a run that fills units and crosses blocks
    kv[:, 7::91, :, 1:] = 0
    kv[:, 2::111] = 0
    k, v = kv[..., :d], kv[..., d:]
    first, lens = [0, 3, 127, 128, 200, 291], [T, T - 1, T - 100, T, T - 64, T]
    page_rows, scales = (128 if variant == "paged" else 0), (torch.float16 if variant == "binary16 scales" else torch.float32)
    bulk, st = _append(iq, torch, shape, rot, cb, k, v, first, lens, T, page_rows, scales)
    rows, st_rows = _append(iq, torch, shape, rot, cb, k, v, first, lens, 4, page_rows, scales)
    for name in ("k_codes", "v_codes", "k_scales", "v_scales"):
        a, b = getattr(bulk, name), getattr(rows, name)
        assert torch.equal(a, b), f"{name}: {int((a != b).sum())} of {a.numel()} differ"
    assert st[0] == st_rows[0] == 0 and st[2] == st_rows[2] == 0
