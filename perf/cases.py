"""The work that a program using this library has it do, as cases that can be timed and compared.

Five kinds of call, through the Python binding:

  step      one decode step of a batch: the step's new K and V rows are appended, the queries attend to the packed cache,
            the partials are merged (``call``: "fused" = iq_decode_step_fused, "separate" = iq_quantize_append + decode_step)
  layers    the same step for a stack of layers with a cache each, captured once in a CUDA graph and replayed: what a
            token costs a single-sequence server
  host      the step from and to pinned host buffers (HostStepper), the call blocks until the output has arrived
  prefill   a prompt (or a chunk of one) quantised and appended in one call
  readback  the packed cache reconstructed as binary16 K and V rows

Shapes are those of this repository's configurations (query heads / KV heads 4/1, 32/4, 16/8, 32/8, 64/8; head_dim 128 and
256; contexts up to 32 K rows, batches up to 32) and odd sizes between them. Rows are Gaussian with four channels scaled by
20 for K and for V, as in the batched serving configuration.
"""
import math

import torch

import paper_2608_08081_b200 as iq

HEADS = ((4, 1), (32, 4), (16, 8), (32, 8), (64, 8))
MAX_CACHE_ROWS = 32 * 32768 * 8   # rows x KV heads of the largest cache a step reads
MAX_NEW_ROWS = 4 * 32768 * 8      # rows x KV heads of the largest prompt


def _case(kind, **kw):
    case = dict(kind=kind, batch=1, heads=32, kv_heads=8, head_dim=128, ctx=4096, bits=3, grid="int8", scales="fp32", page_rows=0,
                ragged=True, argmax=False, call="fused", layers=1)
    case.update(kw)
    return case


def listed():
    def c(name, kind, **kw):
        return dict(_case(kind, **kw), name=name)

    return [
        # the smallest step: one short sequence with one KV head (a small model, or one shard of a larger one); latency
        c("step_tiny", "step", heads=4, kv_heads=1, ctx=1024, ragged=False),
        # a token of a single-sequence server at long context: 16 layers in one graph
        c("layers_one_seq_32k", "layers", layers=16, ctx=32768, ragged=False),
        # interactive serving: eight ragged sequences of a few thousand rows, the three calls of the README
        c("step_batch8_4k", "step", batch=8, heads=64, ctx=4096, call="separate"),
        # the headline workload: 32 long ragged sequences
        c("step_batch32_32k", "step", batch=32, heads=64, ctx=32768),
        # a step whose inputs and outputs live on the host
        c("host_batch16_6k", "host", batch=16, heads=64, ctx=6144),
        # the library's default codebook (exact binary16 levels), with the retrieval argmax
        c("step_fp16_levels_argmax", "step", batch=8, heads=32, kv_heads=4, ctx=32768, grid="fp16", argmax=True),
        # wide heads
        c("step_d256_16k", "step", batch=4, heads=16, kv_heads=8, head_dim=256, ctx=16384),
        # 4-bit codes in a pool of pages with binary16 scales
        c("step_4bit_paged", "step", batch=16, heads=32, ctx=12288, bits=4, scales="fp16", page_rows=256),
        # chunked prefill: a few hundred new rows per sequence, starting and ending inside 128-row blocks
        c("prefill_chunk_500", "prefill", batch=8, ctx=500),
        # long prompts
        c("prefill_batch4_32k", "prefill", batch=4, ctx=32768),
        # a long prompt at another width and head size
        c("prefill_4bit_d256", "prefill", heads=16, kv_heads=8, head_dim=256, ctx=16384, bits=4, ragged=False),
        # the cache read back as fp16 rows (hand-over to a standard attention kernel, migration)
        c("readback_batch4_8k", "readback", batch=4, ctx=8192),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choices(("step", "layers", "host", "prefill", "readback"), (6, 1, 1, 4, 1))[0]
    heads, kv_heads = rng.choice(HEADS)
    head_dim = rng.choice((128, 128, 256))
    bits = rng.choices((3, 2, 4), (3, 1, 1))[0]
    grid = rng.choice(("int8", "int8", "fp16"))
    scales = rng.choice(("fp32", "fp32", "fp16"))
    page_rows = rng.choice((0, 0, 128, 512))
    cap = (MAX_NEW_ROWS if kind in ("prefill", "readback") else MAX_CACHE_ROWS) * 128 // head_dim
    if kind == "layers":  # a stack of single-sequence caches with the layers in place of the batch
        layers = rng.choice((4, 8, 16))
        ctx = _log_int(rng, 512, min(32768, cap // (kv_heads * layers)))
        return _case(kind, heads=heads, kv_heads=kv_heads, head_dim=head_dim, ctx=ctx, bits=bits, grid=grid, scales=scales,
                     ragged=False, layers=layers)
    batch = _log_int(rng, 1, 32)
    ctx = _log_int(rng, 64 if kind == "prefill" else 256, max(256, min(32768, cap // (kv_heads * batch))))
    return _case(kind, batch=batch, heads=heads, kv_heads=kv_heads, head_dim=head_dim, ctx=ctx, bits=bits, grid=grid, scales=scales,
                 page_rows=page_rows, ragged=rng.random() < 0.7, argmax=kind == "step" and rng.random() < 0.25,
                 call=rng.choice(("fused", "fused", "separate")))


def _lengths(case):
    """Rows per sequence (of the prompt, or in the cache before the step): the sizes are the case's, not the seed's."""
    ctx, B = case["ctx"], case["batch"]
    if not case["ragged"]:
        return [ctx - 1 if case["kind"] in ("step", "layers", "host") else ctx] * B
    return [min(ctx - 1, max(1, int(ctx * (0.5 + 0.5 * ((0.6180339887 * (b + 1)) % 1.0))))) for b in range(B)]


def _capacity(rows):
    return (rows + 127) // 128 * 128


def _rows(gen, n, T, H, d, channels):
    x = torch.randn((n, T, H, d), generator=gen, device="cuda", dtype=torch.float16)
    x[..., channels] *= 20.0
    return x


class _State:
    pass


def _new_cache(case, shape, gen):
    scales = torch.float16 if case["scales"] == "fp16" else torch.float32
    pr = case["page_rows"]
    if not pr:
        return shape, iq.new_cache(shape, scales_dtype=scales)
    t_cap = (shape.t_cap + pr - 1) // pr * pr
    shape = iq.Shape(shape.batch, shape.n_q_heads, shape.n_kv_heads, shape.head_dim, t_cap, shape.bits)
    n = shape.batch * (t_cap // pr)
    table = torch.randperm(n, generator=gen, device="cuda").to(torch.int32).reshape(shape.batch, t_cap // pr)  # a pool in use is scattered
    return shape, iq.new_paged_cache(shape, n, pr, table, scales_dtype=scales)


def _fill(st, gen, case, cache, lens, channels):
    """Prompts of the given lengths into an empty cache, a few sequences at a time."""
    shape, H, d = st.shape, case["kv_heads"], case["head_dim"]
    B, T = case["batch"], max(lens)
    at_once = max(1, min(B, (1 << 28) // (T * H * d)))
    for b0 in range(0, B, at_once):
        nb = min(at_once, B - b0)
        k, v = _rows(gen, nb, T, H, d, channels[0]), _rows(gen, nb, T, H, d, channels[1])
        part = iq.Shape(nb, shape.n_q_heads, H, d, shape.t_cap, shape.bits)
        n_new = torch.tensor(lens[b0:b0 + nb], dtype=torch.int32, device="cuda")
        pos = torch.zeros(nb, dtype=torch.int32, device="cuda")
        if cache.block_table is None:
            sub = iq.Cache(cache.k_codes[b0:b0 + nb], cache.k_scales[b0:b0 + nb], cache.v_codes[b0:b0 + nb], cache.v_scales[b0:b0 + nb])
        else:
            sub = iq.Cache(cache.k_codes, cache.k_scales, cache.v_codes, cache.v_scales, cache.block_table[b0:b0 + nb], cache.page_rows)
        iq.iq_quantize_append(part, st.rot, st.cb, k, v, pos, n_new, T, sub, st.status)


def prepare(case, seed):
    kind, B, Hq, H, d = case["kind"], case["batch"], case["heads"], case["kv_heads"], case["head_dim"]
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed)
    st = _State()
    st.kind, st.call = kind, case["call"]
    lens = _lengths(case)
    st.cb = iq.iq_lloyd_max_codebook(d, case["bits"], case["grid"])
    st.rot = torch.empty(iq.iq_rotation_floats(d, H), dtype=torch.float32, device="cuda")
    iq.iq_make_rotation(d, H, seed + 1, None, st.rot)
    st.status = torch.zeros(4, dtype=torch.int32, device="cuda")
    channels = [torch.randperm(d, generator=gen, device="cuda")[:4] for _ in range(2)]

    if kind == "prefill":
        first = [0 if case["ctx"] > 2048 else (37 * (b + 1)) % 200 for b in range(B)]  # a chunk continues a sequence that is there
        st.shape = iq.Shape(B, Hq, H, d, _capacity(max(f + n for f, n in zip(first, lens))), case["bits"])
        st.shape, st.cache = _new_cache(case, st.shape, gen)
        st.n_max = max(lens)
        st.k, st.v = _rows(gen, B, st.n_max, H, d, channels[0]), _rows(gen, B, st.n_max, H, d, channels[1])
        st.pos = torch.tensor(first, dtype=torch.int32, device="cuda")
        st.n_new = torch.tensor(lens, dtype=torch.int32, device="cuda") if case["ragged"] else None
        return st

    # a graph of layers keeps one cache per layer, the others one cache
    st.shape = iq.Shape(B, Hq, H, d, _capacity(case["ctx"]), case["bits"])
    shape, st.caches = st.shape, []
    for _ in range(case["layers"]):
        st.shape, cache = _new_cache(case, shape, gen)
        _fill(st, gen, case, cache, lens, channels)
        st.caches.append(cache)
    st.cache = st.caches[0]
    st.lens = torch.tensor(lens, dtype=torch.int32, device="cuda")

    if kind == "readback":
        st.k_out = torch.zeros((B, max(lens), H, d), dtype=torch.float16, device="cuda")
        st.v_out = torch.zeros_like(st.k_out)
        return st

    L = case["layers"]
    st.q = torch.randn((L, B, Hq, d), generator=gen, device="cuda", dtype=torch.float16)
    st.k_new = torch.stack([_rows(gen, B, 1, H, d, channels[0]) for _ in range(L)])
    st.v_new = torch.stack([_rows(gen, B, 1, H, d, channels[1]) for _ in range(L)])
    st.after = st.lens + 1
    st.splits = iq.iq_suggest_splits(st.shape, max(lens) + 1)
    if kind == "host":
        one = torch.cat([st.q[0].reshape(-1), st.k_new[0].reshape(-1), st.v_new[0].reshape(-1)])
        st.inputs_host = torch.empty((1, one.numel()), dtype=torch.float16, pin_memory=True)
        st.inputs_host[0].copy_(one)
        st.ws = iq.DecodeWorkspace(st.shape, st.splits)
        st.out_dev = torch.empty((B, Hq, d), dtype=torch.float16, device="cuda")
        st.out_host = torch.empty((B, Hq, d), dtype=torch.float16, pin_memory=True)
        st.stepper = iq.HostStepper(st.shape, st.rot, st.cb, st.inputs_host, torch.empty_like(one), torch.stack([st.lens, st.after]),
                                    st.cache, st.ws, st.out_dev, st.out_host)
        return st
    if kind == "step" and st.call == "separate":
        st.ws = iq.DecodeWorkspace(st.shape, st.splits, want_argmax=case["argmax"])
        return st
    st.work = torch.empty(iq.iq_decode_step_workspace_bytes(st.shape, st.splits), dtype=torch.uint8, device="cuda")
    st.out = torch.empty((L, B, Hq, d), dtype=torch.float32, device="cuda")
    st.lse = torch.empty((L, B, Hq), dtype=torch.float32, device="cuda")
    st.argmax = torch.empty((L, B, Hq), dtype=torch.int32, device="cuda") if case["argmax"] else None
    st.steps = [dict(q=st.q[i], k=st.k_new[i], v=st.v_new[i], cache=st.caches[i], out=st.out[i], lse=st.lse[i],
                     argmax=None if st.argmax is None else st.argmax[i]) for i in range(L)]
    if kind == "layers":
        torch.cuda.synchronize()
        st.graph = torch.cuda.CUDAGraph()
        _fused(st)  # the kernels are loaded before the capture begins
        torch.cuda.synchronize()
        with torch.cuda.graph(st.graph):
            _fused(st)
    return st


def _fused(st):
    for s in st.steps:
        iq.iq_decode_step_fused(st.shape, st.rot, st.cb, s["q"], s["k"], s["v"], s["cache"], st.lens, st.splits, st.work, s["out"],
                                s["lse"], s["argmax"], st.status)


def _cache_arrays(cache):
    return {"k_codes": cache.k_codes, "k_scales": cache.k_scales, "v_codes": cache.v_codes, "v_scales": cache.v_scales}


def run(st):
    if st.kind == "prefill":
        iq.iq_quantize_append(st.shape, st.rot, st.cb, st.k, st.v, st.pos, st.n_new, st.n_max, st.cache, st.status)
        return _cache_arrays(st.cache)
    if st.kind == "readback":
        iq.iq_reconstruct_rows(st.shape, st.rot, st.cb, st.cache, st.lens, st.k_out, st.v_out)
        return st.k_out, st.v_out
    if st.kind == "host":
        st.stepper.step(0)
        return st.out_host, _cache_arrays(st.cache)
    if st.kind == "layers":
        st.graph.replay()
        return st.out, st.lse, [_cache_arrays(c) for c in st.caches[:2]] + [_cache_arrays(st.caches[-1])]
    if st.call == "separate":
        iq.iq_quantize_append(st.shape, st.rot, st.cb, st.k_new[0], st.v_new[0], st.lens, None, 1, st.cache, st.status)
        iq.decode_step(st.shape, st.rot, st.cb, st.q[0], st.cache, st.after, st.ws)
        return st.ws.out, st.ws.lse, st.ws.argmax, _cache_arrays(st.cache)
    _fused(st)
    return st.out, st.lse, st.argmax, _cache_arrays(st.cache)


def work(case):
    d, H, Hq = case["head_dim"], case["kv_heads"], case["heads"]
    rows = sum(_lengths(case))
    packed = 2 * (case["bits"] * d // 8 + (2 if case["scales"] == "fp16" else 4))  # a K and a V row of one KV head
    rotate = d * math.log2(d) + 7 * d                                              # butterfly and 4x4 blocks of one row
    if case["kind"] in ("prefill", "readback"):
        return {"bytes": rows * H * (packed + 4 * d), "flops": rows * H * 2 * (rotate + 3 * d)}
    L, B = case["layers"], case["batch"]
    out = 2 if case["kind"] == "host" else 4
    per_layer = (rows + B) * H * packed + B * (Hq * d * (2 + out) + 2 * H * d * 2 + Hq * 4)
    return {"bytes": L * per_layer, "flops": L * (4.0 * (rows + B) * Hq * d + B * (2 * Hq + 2 * H) * rotate)}


def tolerance(case):
    if case["kind"] == "prefill":
        return {"rel": 1e-7}      # codes are those of an fp64 evaluation, scales fp32 roundings of an fp64 sum
    if case["kind"] == "readback":
        return {"rel": 1e-4, "max": 2e-3}   # one rounding to binary16 of an fp32 evaluation: an ulp here and there
    if case["kind"] == "host":
        return {"rel": 1e-4, "max": 4e-3}   # the output is binary16 (an ulp here and there: measured 2.5e-5, 1e-3)
    return {"rel": 2e-5, "max": 6e-4}       # fp32 scores of a 21- or 22-bit query, fp32 sums in any order: 4e-6 and 1.6e-4 between
                                            # two split counts, 3e-6 to 1.4e-5 of a head against an fp64 evaluation
