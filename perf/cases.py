"""The work that users of libkvb have it do, as cases that can be timed and compared.

A case is a dict of plain values.  `call` says which entry points a pass goes through:

  path        kvb_assemble_select, then kvb_selective_attn: a request (or a batch) whose prompt is stitched
              from cached chunks, with the rows to recompute chosen and attended -- the serving path
  two_call    kvb_assemble, kvb_deviation_topk, kvb_patch: the same decisions for an engine that keeps the
              stitched buffer between the steps and splices the fresh rows in (Algorithms 1 and 2)
  attention   kvb_selective_attn alone, on a stitched buffer and a selection that are already there
  quantize    kvb_quantize_chunks: the chunks of a prefilled prompt enter the cache
  importance  kvb_chunk_importance: the eviction scores of prompts that are held as stitched buffers

Prompts are multiples of the 128-token chunk (the library takes no others).  Values follow the recipe of
paper_2608_21362_b200/synth.py; chunk order, positions and modes are drawn from the seed.
"""
import math
import random

import torch

from paper_2608_21362_b200 import binding as B
from paper_2608_21362_b200 import synth

CHUNK = 128
SEAM_NOISE_TOKENS = 16  # the recipe's strongly deviating tokens at the start of every cached chunk
BASE = {"layers": 36, "q_heads": 16, "kv_heads": 2, "dtype": "bf16", "hit": 0.75, "mode": "int8", "ratio": 0.15, "k": -1,
        "seam": 16, "sinks": 0, "which": 3, "compact": False, "importance": False}


def _case(name, call, prompts, **more):
    c = {"name": name, "call": call, "prompts": prompts}
    if call == "quantize":
        keep = ("layers", "kv_heads", "dtype", "compact")
        c.update({k: BASE[k] for k in keep}, bits=8, unrotate=False)
    elif call == "importance":
        c.update({k: BASE[k] for k in ("layers", "kv_heads", "dtype")})
    else:
        c.update(BASE)
    c.update(more)
    return c


def listed():
    return [
        # one layer of a short prompt, any original positions: a pass is launches and latency
        _case("short_one_layer", "path", "512", layers=1, dtype="fp16"),
        # an ordinary chat or code prompt, three quarters of it cached
        _case("prompt_2k_int8", "path", "2048"),
        # a long document at the smallest cache footprint, top-k only, no seam windows
        _case("prompt_8k_int4", "path", "8192", mode="int4", hit=0.875, seam=0),
        # a serving batch of very different prompts, chunks in every cache format
        _case("batch_ragged", "path", "512,1152,2304,3712,5632,8576,11776,16384", mode="mixed"),
        # many short prompts in one step, compact metadata, attention sinks, eviction scores on the way
        _case("batch_short", "path", ",".join(str(CHUNK * (4 + (5 * i) % 11)) for i in range(24)), hit=0.9, sinks=4, compact=True, importance=True),
        # four query heads for each of four KV heads, in fp16: another head geometry, an odd number of chunks
        _case("prompt_3k_gqa4_fp16", "path", "3200", kv_heads=4, dtype="fp16", hit=0.8),
        # the engine that goes step by step: stitch, select by the keys alone, splice
        _case("steps_4k_patch", "two_call", "4224", mode="mixed", which=1),
        # the repair pass's attention alone: 1229 rows over 8192 keys
        _case("attention_8k", "attention", "8192", mode="int4", hit=0.875, k=1229, seam=0),
        # a 2K prompt's chunks go into the cache as int8
        _case("quantize_2k_int8", "quantize", "2048"),
        # a 16K prompt's chunks go in as int4, position-free and with compact metadata
        _case("quantize_16k_int4", "quantize", "16384", bits=4, unrotate=True, compact=True),
        # the cache manager scores the chunks of the prompts it holds
        _case("importance_batch", "importance", "1024,2176,4096,8192,12288"),
    ]


def _prompts(case):
    return [int(t) for t in str(case["prompts"]).split(",")]


def draw(rng):
    """One more case of the same ranges: every call, prompts of 512 to 16384 tokens, batches, the head
    geometries, data types and options above."""
    call = rng.choice(["path"] * 5 + ["two_call"] * 2 + ["attention"] + ["quantize"] * 2 + ["importance"])
    q_heads, kv_heads = rng.choice([(16, 2), (16, 2), (16, 2), (16, 4), (8, 1), (8, 8), (16, 16)])
    layers = rng.choice([1, 3, 12, 28, 36, 36])
    # totals stay below the ragged batch's (50,048 tokens of 36 layers and 2 KV heads; its attention)
    room = 50048 * 72 // (layers * kv_heads)
    total = int(math.exp(rng.uniform(math.log(512), math.log(min(room, 50048)))))
    n = rng.choice([1, 1, 1, 2, 5, 12])
    prompts, left = [], total
    for i in range(n):
        t = left if i == n - 1 else int(left * rng.uniform(0.3, 1.5) / (n - i))
        t = max(4, min(128, t // CHUNK)) * CHUNK
        prompts.append(t)
        left = max(512, left - t)
    while sum(prompts) * layers * kv_heads > 50048 * 72 or sum(t * t for t in prompts) * layers * q_heads > 5.3e8 * 36 * 16:
        prompts = [max(4, t // CHUNK // 2) * CHUNK for t in prompts]
    text = ",".join(str(t) for t in prompts)
    dtype = rng.choice(["bf16", "bf16", "fp16"])
    if call == "quantize":
        return _drawn(call, text, layers=layers, kv_heads=kv_heads, dtype=dtype, bits=rng.choice([4, 8]),
                      unrotate=rng.random() < 0.5, compact=rng.random() < 0.5)
    if call == "importance":
        return _drawn(call, text, layers=layers, kv_heads=kv_heads, dtype=dtype)
    return _drawn(call, text, layers=layers, q_heads=q_heads, kv_heads=kv_heads, dtype=dtype,
                  hit=round(rng.uniform(0.5, 0.95), 3), mode=rng.choice(["int8", "int4", "mixed", "mixed"]),
                  ratio=round(rng.uniform(0.05, 0.3), 3), seam=rng.choice([0, 16, 16]), sinks=rng.choice([0, 0, 4]),
                  which=rng.choice([1, 3, 3]), compact=rng.random() < 0.3, importance=rng.random() < 0.2)


def _drawn(call, prompts, **more):
    c = _case("", call, prompts, **more)
    del c["name"]
    return c


# ------------------------------------------------------------------ what a program has in hand
def _shape(case):
    return synth.Shape(L=case["layers"], Hq=case.get("q_heads", case["kv_heads"]), Hkv=case["kv_heads"], kv_dtype=case["dtype"])


def _mode_counts(case, n):
    """(fresh, fp16, int8, int4) chunks of a prompt of n chunks: fixed by the case, their places are not."""
    cached = max(1, min(n - 1, round(case["hit"] * n)))
    if case["mode"] == "mixed":
        fp16, int8 = round(0.4 * cached), round(0.4 * cached)
        return n - cached, fp16, int8, cached - fp16 - int8
    return n - cached, 0, cached if case["mode"] == "int8" else 0, cached if case["mode"] == "int4" else 0


def _workload(case, seed):
    rng, sh, plans = random.Random(seed), _shape(case), []
    for t in _prompts(case):
        n = t // CHUNK
        modes = [m for m, k in zip((synth.MODE_FRESH, synth.MODE_FP16, synth.MODE_INT8, synth.MODE_INT4), _mode_counts(case, n)) for _ in range(k)]
        rng.shuffle(modes)
        chunks = []
        for i, m in enumerate(modes):
            orig = i * CHUNK if m == synth.MODE_FRESH else rng.randrange(0, 32768 - CHUNK + 1)
            match = synth.MATCH_MISS if m == synth.MODE_FRESH else synth.MATCH_EXACT if orig == i * CHUNK else synth.MATCH_APPROX
            chunks.append(synth.ChunkPlan(i * CHUNK, orig, m, match))
        plans.append(synth.RequestPlan(t, chunks))
    sel = synth.SelectPlan(ratio=case["ratio"], k_override=case["k"], seam_before=case["seam"], seam_after=0, which=case["which"])
    return synth.Workload("case", seed, sh, plans, sel)


class _State:
    """A context and the tables and tensors of one batch; the context goes with it."""

    def __init__(self, ctx):
        self.ctx = ctx

    def __del__(self):
        if B is not None:  # None while the interpreter ends
            B.kvb_destroy(self.ctx)


def _flat(tensors_shapes, dtype, device):
    """One allocation for a batch's buffers of a kind, as a serving engine's pool holds them, and its views
    (every view starts on a 256-byte boundary: all sizes here are multiples of it)."""
    sizes = [math.prod(s) for s in tensors_shapes]
    pool = torch.zeros(sum(sizes), dtype=dtype, device=device)
    views, at = [], 0
    for size, shape in zip(sizes, tensors_shapes):
        views.append(pool[at : at + size].view(shape))
        at += size
    return pool, views


def prepare(case, seed):
    dev, sh = torch.device("cuda", 0), _shape(case)
    prompts = _prompts(case)
    s = _State(B.create_for_shape(sh, 0))
    s.case = case
    if case["call"] == "quantize":
        _prepare_quantize(s, case, seed, sh, dev)
        return s
    if case["call"] == "importance":
        g = torch.Generator(device=dev).manual_seed(seed)
        s.requests = []
        for t in prompts:
            kv = torch.randn((sh.L, 2, t, sh.Hkv, sh.d), generator=g, device=dev)
            kv[:, 0] *= torch.exp(torch.rand((sh.L, 1, sh.Hkv, sh.d), generator=g, device=dev) * 4.6 - 2.3)
            kv = kv.to(sh.torch_dtype)
            chunks = [synth.Chunk(synth.ChunkPlan(i * CHUNK, i * CHUNK, synth.MODE_FRESH, synth.MATCH_MISS)) for i in range(t // CHUNK)]
            s.requests.append(synth.Request(synth.RequestPlan(t, [c.plan for c in chunks]), chunks, kv, kv, None, 0))
        s.table = B.RequestTable(s.requests)
        s.scores = [torch.zeros(t // CHUNK, dtype=torch.float32, device=dev) for t in prompts]
        return s
    wl = _workload(case, seed)
    bq = B.BatchedQuantizer(s.ctx, sh, meta_fp16=case["compact"])

    def stitch(shape, plan, chunks, fresh):
        for c in chunks:  # the table has to say which metadata a chunk carries
            c.meta_fp16 = int(case["compact"] and c.k_meta is not None)
        return bq.assemble(shape, plan, chunks, fresh)

    s.requests = synth.materialize(wl, dev, bq.quantize_k, bq.quantize_v, stitch)
    caps = [min(r.plan.T, r.sel_capacity + case["sinks"]) for r in s.requests]
    s.kv_pool, kv = _flat([r.fresh.shape for r in s.requests], sh.torch_dtype, dev)
    s.importance = None
    if case["importance"]:
        s.importance, imp = _flat([(max(64, t // CHUNK),) for t in prompts], torch.float32, dev)
    for i, r in enumerate(s.requests):
        if case["call"] == "attention":
            kv[i].copy_(r.kv_buf)
        r.kv_buf = kv[i]
        if s.importance is not None:
            r.importance = imp[i]
    s.table = B.RequestTable(s.requests)
    ks = [case["k"] if case["k"] >= 0 else B.kvb_select_count(t, case["ratio"]) for t in prompts]
    s.sel = B.SelectionTable(prompts, ks, caps, dev)
    if case["call"] != "two_call":
        g = torch.Generator(device=dev).manual_seed(seed + 7)
        s.q = [(torch.randn((sh.L, cap, sh.Hq, sh.d), generator=g, device=dev) / math.sqrt(sh.d)).to(sh.torch_dtype) for cap in caps]
        s.out_pool, s.out = _flat([q.shape for q in s.q], sh.torch_dtype, dev)
    if case["call"] == "attention":
        _select(s, B.kvb_deviation_topk)
        torch.cuda.synchronize()
    for r in s.requests:
        r.q = None
    return s


def _prepare_quantize(s, case, seed, sh, dev):
    g = torch.Generator(device=dev).manual_seed(seed)
    n, H, mt = sum(_prompts(case)) // CHUNK, sh.Hkv, torch.float16 if case["compact"] else torch.float32
    byte, groups = case["bits"] / 8, 1 if case["bits"] == 8 else CHUNK // sh.int4_group
    scale = torch.exp(torch.rand((sh.L, 1, H, sh.d), generator=g, device=dev) * 4.6 - 2.3)
    s.k = torch.empty((n, sh.L, CHUNK, H, sh.d), dtype=sh.torch_dtype, device=dev)
    s.v = torch.empty_like(s.k)
    for i in range(n):
        s.k[i] = torch.randn((sh.L, CHUNK, H, sh.d), generator=g, device=dev) * scale
        s.v[i] = torch.randn((sh.L, CHUNK, H, sh.d), generator=g, device=dev)
    codes = (n, sh.L, CHUNK, H, int(sh.d * byte))
    s.k_codes, s.v_codes = (torch.zeros(codes, dtype=torch.uint8, device=dev) for _ in range(2))
    s.k_meta = torch.zeros((n, sh.L, groups, H, sh.d, 2), dtype=mt, device=dev)
    s.v_meta = torch.zeros((n, sh.L, CHUNK, H, groups, 2), dtype=mt, device=dev)
    s.jobs = B.QuantizeTable([dict(k=s.k[i], v=s.v[i], k_codes=s.k_codes[i], v_codes=s.v_codes[i], k_meta=s.k_meta[i], v_meta=s.v_meta[i],
                                   bits=case["bits"], meta_fp16=case["compact"], unrotate_from=i * CHUNK if case["unrotate"] else -1)
                              for i in range(n)])


def _select(s, call):
    c = s.case
    call(s.ctx, s.table, c["ratio"], c["k"], c["seam"], 0, c["which"], s.sel, sink_tokens=c["sinks"])


def run(s):
    call = s.case["call"]
    if call == "quantize":
        B.kvb_quantize_chunks(s.ctx, s.jobs)
        return {"k_codes": s.k_codes, "v_codes": s.v_codes, "k_meta": s.k_meta, "v_meta": s.v_meta}
    if call == "importance":
        B.kvb_chunk_importance(s.ctx, s.table, s.scores)
        return s.scores
    if call == "two_call":
        B.kvb_assemble(s.ctx, s.table)
        _select(s, B.kvb_deviation_topk)
        B.kvb_patch(s.ctx, s.table, s.sel)
        return {"kv": s.kv_pool, "importance": s.importance, **_selection(s)}
    if call == "path":
        _select(s, B.kvb_assemble_select)
    B.kvb_selective_attn(s.ctx, s.table, s.sel, s.q, s.out, 1.0 / math.sqrt(128))
    if call == "path":
        return {"kv": s.kv_pool, "out": s.out_pool, "importance": s.importance, **_selection(s)}
    return s.out_pool


def _selection(s):
    sel, several = s.sel, len(s.requests) <= 12
    whole = {"n_sel": sel.n_sel, "sel": sel.sel}
    return {**whole, "delta": sel.delta, "rank": sel.rank} if several else {**whole, "delta": sel.delta}


# ------------------------------------------------------------------ what a pass cannot do without
def _selected_rows(case, t):
    """Rows that the selection holds: the top k, and the part of the seam windows that is not among them
    (k takes the strongly deviating tokens first, then cached tokens anywhere)."""
    k = case["k"] if case["k"] >= 0 else math.floor(case["ratio"] * t)
    n = t // CHUNK
    cached = n - _mode_counts(case, n)[0]
    spare = max(0, k - SEAM_NOISE_TOKENS * cached)
    hit_again = min(1.0, spare / max(1, (CHUNK - SEAM_NOISE_TOKENS) * cached)) * cached / n
    return min(t, k + (n - 1) * case["seam"] * (1.0 - hit_again) + case["sinks"])


def work(case):
    sh = _shape(case)
    L, H, d, pair = sh.L, sh.Hkv, sh.d, 4 if case.get("compact") else 8
    row = H * d * 2  # bytes of one token's 16-bit keys (or values) of one layer
    n_bytes = flops = 0.0
    for t in _prompts(case):
        if case["call"] == "quantize":
            codes = t * row * case["bits"] / 16
            groups = (t // CHUNK if case["bits"] == 8 else t // sh.int4_group) * H * d, t * H * (1 if case["bits"] == 8 else d // sh.int4_group)
            n_bytes += L * (2 * t * row + 2 * codes + sum(groups) * pair)
        elif case["call"] == "importance":
            n_bytes += L * t * row + 4 * t // CHUNK
        else:
            n = t // CHUNK
            fresh, fp16, int8, int4 = _mode_counts(case, n)
            rows = _selected_rows(case, t)
            if case["call"] != "attention":
                codes = 2 * CHUNK * row * (fresh + fp16 + int8 / 2 + int4 / 4)
                meta = pair * CHUNK * H * (int8 * (1 + d // CHUNK) + int4 * (d // 32 + 4))
                sides = (case["which"] & 1) + (case["which"] >> 1)
                n_bytes += L * (codes + meta + 2 * t * row + sides * CHUNK * (n - fresh) * row)
                if case["call"] == "two_call":
                    n_bytes += L * 2 * rows * row * (1 if sides == 1 else 0)  # the spliced values' fresh rows; keys were read
            if case["call"] != "two_call":
                n_bytes += L * (2 * rows * sh.Hq * d * 2 + (2 * t * row if case["call"] == "attention" else 0))
                flops += L * sh.Hq * 4.0 * d * rows * (t + 1) / 2
    return {"bytes": n_bytes, "flops": flops}


def tolerance(case):
    if case["call"] == "quantize":
        return "exact"  # the codes and their metadata are fixed bit for bit
    if case["call"] == "importance":
        return {"rel": 5e-7, "max": 2e-6}  # 3.2e-8 against float64
    bf16 = case["dtype"] == "bf16"
    # whole values: the ranks of positions whose deviations agree to a float32 rounding (0.2 % to 0.9 % of
    # them change places between the one-pass and the two-call sums)
    if case["call"] == "two_call":  # a stitched value may round to the other 16-bit neighbour (under 0.1 % / 0.5 % do)
        return {"rel": 4e-4 if bf16 else 1e-4, "max": 8e-3 if bf16 else 2e-3, "differ": 0.01}
    # attention outputs against float64: rel 2.4e-3, max 0.045 (bf16); 2.9e-4, 2.3e-3 (fp16, 3200 keys)
    return {"rel": 1e-2 if bf16 else 1.2e-3, "max": 0.18 if bf16 else 0.03, "differ": 0.01}
