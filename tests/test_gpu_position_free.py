"""Position-free cache population (kvb_quantize_keys_at): keys rotated back by their original position
before Eq. 6, so that a cached chunk is listed with orig_pos = 0 and re-used with one rotation."""
import numpy as np
import pytest
import torch

import oracle
from paper_2608_21362_b200 import binding as B
from paper_2608_21362_b200 import synth
from paper_2608_21362_b200.build import build_library

import oracle_glue as helpers

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    build_library()


def _keys(sh, seed):
    g = torch.Generator().manual_seed(seed)
    x = torch.randn((sh.L, sh.C, sh.Hkv, sh.d), generator=g) * torch.exp(torch.rand((sh.L, 1, sh.Hkv, sh.d), generator=g) * 3.0 - 1.5)
    return x.to(sh.torch_dtype)


def _quantize_at(ctx, sh, x_dev, pos, bits):
    L, Cn, H, d = x_dev.shape
    codes = torch.empty((L, Cn, H, d * bits // 8), dtype=torch.uint8, device=DEV)
    meta = torch.empty((L, 1 if bits == 8 else Cn // sh.int4_group, H, d, 2), dtype=torch.float32, device=DEV)
    B.kvb_quantize_keys_at(ctx, x_dev, pos, bits, codes, meta)
    B.kvb_last_status(ctx)
    return codes, meta


@pytest.mark.parametrize("kv_dtype", ["bf16", "fp16"])
def test_codes_and_metadata_bit_exact(kv_dtype):
    sh = synth.Shape(L=2, kv_dtype=kv_dtype)
    dtc = helpers.dt_code(sh)
    ctx = B.create_for_shape(sh, 0)
    try:
        x = _keys(sh, 5)
        xb = helpers.bits_of(x)
        for pos in (0, 128, 4096 * 3 + 128, (1 << 24) - 128):
            for bits, group in ((8, sh.C), (4, sh.int4_group)):
                codes, meta = _quantize_at(ctx, sh, x.to(DEV), pos, bits)
                for l in range(sh.L):
                    u = oracle.unrotate_keys(xb[l], dtc, sh.theta, pos)
                    oc, om = oracle.quantize_k(u, bits, group)
                    assert np.array_equal(codes[l].cpu().numpy(), oc), "codes, pos %d bits %d" % (pos, bits)
                    assert np.array_equal(meta[l].cpu().numpy(), om), "metadata, pos %d bits %d" % (pos, bits)
        # position 0 is the plain quantiser
        qk, _ = B.quantize_fns(ctx, sh)
        c0, m0 = _quantize_at(ctx, sh, x.to(DEV), 0, 8)
        c1, m1 = qk(x.to(DEV), 8, sh.C)
        assert torch.equal(c0, c1) and torch.equal(m0, m1)
        assert B.kvb_quantize_keys_at(ctx, x.to(DEV), -1, 8, c0, m0, check=False) == B.KVB_ERR_INVALID_ARG
        assert B.kvb_quantize_keys_at(ctx, x.to(DEV), 0, 5, c0, m0, check=False) == B.KVB_ERR_INVALID_ARG
    finally:
        B.kvb_destroy(ctx)


def test_reuse_at_another_position_is_one_rotation():
    """Keys encoded at position 896, stored position-free, re-used at position 256: the stitched rows are
    the original keys rotated by 256 - 896, up to the quantisation step (Eq. 6: half a step per channel,
    a rotation mixes two channels)."""
    sh = synth.Shape(L=2)
    dtc = helpers.dt_code(sh)
    orig, new, T = 896, 256, 512
    ctx = B.create_for_shape(sh, 0)
    try:
        x = _keys(sh, 9)
        vals = _keys(sh, 10)
        codes, meta = _quantize_at(ctx, sh, x.to(DEV), orig, 8)
        qk, qv = B.quantize_fns(ctx, sh)
        vcodes, vmeta = qv(vals.to(DEV), 8, sh.d)
        plan = synth._request(T, sh.C, [synth.MODE_FRESH, synth.MODE_FRESH, synth.MODE_INT8, synth.MODE_FRESH], [0, 0, 0, 0])
        assert plan.chunks[2].new_pos == new and plan.chunks[2].orig_pos == 0

        class R:
            pass

        r = R()
        r.plan = plan
        r.chunks = [synth.Chunk(c) for c in plan.chunks]
        r.chunks[2] = synth.Chunk(plan.chunks[2], codes, vcodes, meta, vmeta)
        r.fresh = torch.zeros((sh.L, 2, T, sh.Hkv, sh.d), dtype=sh.torch_dtype, device=DEV)
        r.kv_buf = torch.zeros_like(r.fresh)
        B.kvb_assemble(ctx, B.RequestTable([r]))
        B.kvb_last_status(ctx)
        got = oracle.bits_to_f64(helpers.bits_of(r.kv_buf[:, 0, new : new + sh.C]), dtc)  # [L,C,H,d]
        x64 = oracle.bits_to_f64(helpers.bits_of(x), dtc)
        half = sh.d // 2
        for l in range(sh.L):
            want = oracle.rope_rotate(x64[l], sh.theta, float(new - orig))
            scale = meta[l, 0].cpu().numpy()[..., 0].astype(np.float64)  # [H,d] step of each stored channel
            step_pair = np.sqrt(scale[:, :half] ** 2 + scale[:, half:] ** 2)
            bound = 0.5 * np.concatenate([step_pair, step_pair], -1)[None] * 1.01 + 2.0**-8 * np.abs(want) + 1e-6
            assert np.all(np.abs(got[l] - want) <= bound)
    finally:
        B.kvb_destroy(ctx)


@pytest.mark.parametrize("kv_dtype,Hkv", [("bf16", 2), ("fp16", 1), ("bf16", 4), ("fp16", 8)])
def test_batched_quantiser_codes_bit_exact(kv_dtype, Hkv):
    """kvb_quantize_chunks: one launch for a batch of chunks with mixed widths, keys only / values only
    / both, keys rotated back or not, compact or float32 metadata.  Codes and metadata equal the
    oracle's bit for bit (Eq. 6 forward: float32 subtract, divide, round-half-even on both sides),
    including groups with tiny and with zero range, where the fast reciprocal must not decide."""
    sh = synth.Shape(L=3, Hq=8, Hkv=Hkv, kv_dtype=kv_dtype)
    dtc = helpers.dt_code(sh)
    ctx = B.create_for_shape(sh, 0, max_chunks_total=16)
    try:
        specs = [  # (bits, keys?, values?, unrotate_from, meta_fp16)
            (8, True, True, -1, False), (4, True, True, -1, False), (8, True, False, 4096 + 128, False), (4, True, True, 77, False),
            (8, False, True, -1, False), (4, True, True, -1, True), (8, True, True, (1 << 24) - 128, True), (8, True, True, -1, False),
            (8, True, True, -1, False), (4, True, True, -1, True),  # 8, 9: every other quotient an exact tie (below)
        ]
        jobs, xs = [], []
        for i, (bits, has_k, has_v, pos, m16) in enumerate(specs):
            k = _keys(sh, 100 + i)
            v = _keys(sh, 200 + i)
            if i == 7:  # degenerate groups: a constant channel, a constant row, a range of a few float32 ulps, a huge range
                k[:, :, :, 3] = 1.25
                v[:, 5] = -0.5
                k[:, :, :, 9] = 1.0
                k[:, 64:, :, 9] = 1.0 + 2.0 ** -7
                v[:, 7, :, ::2] = 3.0e4 if kv_dtype == "fp16" else 1.0e30
            if i >= 8:  # integers in [0, 2 * levels] with both ends in every group: scale 2, the odd ones tie, and the
                # quotient without a division has to round them as the division would
                top = 2 * ((1 << bits) - 1)
                g = torch.Generator().manual_seed(300 + i)
                k = torch.randint(0, top // 2 + 1, (sh.L, sh.C, Hkv, sh.d), generator=g).float()
                v = torch.randint(0, top // 2 + 1, (sh.L, sh.C, Hkv, sh.d), generator=g).float()
                k[:, 0::32], k[:, 1::32] = 0.0, float(top)              # keys: groups run over tokens
                v[:, :, :, 0::32], v[:, :, :, 1::32] = 0.0, float(top)  # values: over channels
                k, v = k.to(sh.torch_dtype), v.to(sh.torch_dtype)
            mt = torch.float16 if m16 else torch.float32
            j = dict(bits=bits, unrotate_from=pos, meta_fp16=m16)
            if has_k:
                j.update(k=k.to(DEV), k_codes=torch.zeros((sh.L, sh.C, Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV),
                         k_meta=torch.zeros((sh.L, 1 if bits == 8 else sh.C // sh.int4_group, Hkv, sh.d, 2), dtype=mt, device=DEV))
            if has_v:
                j.update(v=v.to(DEV), v_codes=torch.zeros((sh.L, sh.C, Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV),
                         v_meta=torch.zeros((sh.L, sh.C, Hkv, 1 if bits == 8 else sh.d // sh.int4_group, 2), dtype=mt, device=DEV))
            jobs.append(j)
            xs.append((k, v))
        B.kvb_quantize_chunks(ctx, jobs)
        B.kvb_last_status(ctx)
        for (bits, has_k, has_v, pos, m16), j, (k, v) in zip(specs, jobs, xs):
            gk, gv = (sh.C, sh.d) if bits == 8 else (sh.int4_group, sh.int4_group)
            for l in range(sh.L):
                if has_k:
                    u = oracle.unrotate_keys(helpers.bits_of(k)[l], dtc, sh.theta, pos) if pos >= 0 else helpers.f64_of(k)[l]
                    oc, om = oracle.quantize_k(u, bits, gk, meta16=m16)
                    assert np.array_equal(j["k_codes"][l].cpu().numpy(), oc), ("key codes", bits, pos, m16)
                    assert np.array_equal(j["k_meta"][l].float().cpu().numpy(), om.astype(np.float32)), ("key metadata", bits, pos, m16)
                if has_v:
                    oc, om = oracle.quantize_v(helpers.f64_of(v)[l], bits, gv, meta16=m16)
                    assert np.array_equal(j["v_codes"][l].cpu().numpy(), oc), ("value codes", bits, m16)
                    assert np.array_equal(j["v_meta"][l].float().cpu().numpy(), om.astype(np.float32)), ("value metadata", bits, m16)
        # the one-chunk entry points are the same kernel with one job
        c1 = torch.zeros_like(jobs[0]["k_codes"])
        m1 = torch.zeros_like(jobs[0]["k_meta"])
        B.kvb_quantize_chunk(ctx, jobs[0]["k"], False, 8, c1, m1)
        B.kvb_last_status(ctx)
        assert torch.equal(c1, jobs[0]["k_codes"]) and torch.equal(m1, jobs[0]["k_meta"])
        # rejected: no side wanted, a missing output, too many jobs for the context
        assert B.kvb_quantize_chunks(ctx, [dict(bits=8)], check=False) == B.KVB_ERR_INVALID_ARG
        assert B.kvb_quantize_chunks(ctx, [dict(bits=8, k=jobs[0]["k"], k_codes=c1)], check=False) == B.KVB_ERR_INVALID_ARG
        assert B.kvb_quantize_chunks(ctx, [jobs[0]] * 4096, check=False) == B.KVB_ERR_WORKSPACE
        assert B.kvb_quantize_chunks(ctx, []) == B.KVB_OK
    finally:
        B.kvb_destroy(ctx)


def _eq6(x, bits):
    """Eq. 6 on [..., group] rows in float32, as the library states it: (codes, scale, min)."""
    x = x.float()
    mn, mx = x.amin(-1, keepdim=True), x.amax(-1, keepdim=True)
    s = torch.where(mx > mn, (mx - mn) / float(2**bits - 1), torch.ones_like(mn))
    return torch.clamp(torch.round((x - mn) / s), 0, 2**bits - 1), s, mn


@pytest.mark.parametrize("n_jobs,L,Hkv,bits", [(1, 1, 1, 8), (60, 1, 2, 4), (61, 1, 2, 8), (256, 1, 1, 4), (257, 1, 2, 8), (3, 5, 4, 4)])
def test_job_counts_and_extreme_ranges(n_jobs, L, Hkv, bits):
    """Both argument sizes and the table beyond them, fewer tiles than SMs and ranges that do not divide, and channels
    whose range is zero, tiny (below the reciprocal's range), huge or ordinary: codes and metadata bit for bit."""
    sh = synth.Shape(L=L, Hq=Hkv, Hkv=Hkv)
    ctx = B.create_for_shape(sh, 0, max_chunks_total=512)
    try:
        g = torch.Generator().manual_seed(n_jobs)
        k = torch.randn((n_jobs, L, sh.C, Hkv, sh.d), generator=g)
        v = torch.randn((n_jobs, L, sh.C, Hkv, sh.d), generator=g)
        k[..., 5] = 1.5                    # no range
        k[..., 6] *= 1e-30                 # scale below 1e-20
        k[..., 70] *= 1e30                 # scale above 1e20
        k[..., 71] = torch.round(k[..., 71] * 4)  # a coarse lattice: ties
        v[:, :, 3] *= 1e-30
        v[:, :, 4] *= 1e30
        v[:, :, 5] = -2.0
        k, v = k.to(sh.torch_dtype), v.to(sh.torch_dtype)
        G = 1 if bits == 8 else 4
        kc = torch.zeros((n_jobs, L, sh.C, Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV)
        vc = torch.zeros_like(kc)
        km = torch.zeros((n_jobs, L, G, Hkv, sh.d, 2), dtype=torch.float32, device=DEV)
        vm = torch.zeros((n_jobs, L, sh.C, Hkv, G, 2), dtype=torch.float32, device=DEV)
        kd, vd = k.to(DEV), v.to(DEV)
        skip_v = n_jobs // 2  # one job without values
        B.kvb_quantize_chunks(ctx, [dict(k=kd[i], k_codes=kc[i], k_meta=km[i], bits=bits, **({} if i == skip_v and n_jobs > 1 else
                                    dict(v=vd[i], v_codes=vc[i], v_meta=vm[i]))) for i in range(n_jobs)])
        B.kvb_last_status(ctx)
        kg = k.view(n_jobs, L, G, sh.C // G, Hkv, sh.d).permute(0, 1, 2, 4, 5, 3)  # tokens of a group last
        codes, s, mn = _eq6(kg, bits)
        codes = codes.permute(0, 1, 2, 5, 3, 4).reshape(n_jobs, L, sh.C, Hkv, sh.d).to(torch.uint8)
        vcodes, vs, vmn = _eq6(v.view(n_jobs, L, sh.C, Hkv, G, sh.d // G), bits)
        vcodes = vcodes.reshape(n_jobs, L, sh.C, Hkv, sh.d).to(torch.uint8)
        if bits == 4:
            codes, vcodes = codes[..., 0::2] | (codes[..., 1::2] << 4), vcodes[..., 0::2] | (vcodes[..., 1::2] << 4)
        if n_jobs > 1:
            vcodes[skip_v], vs[skip_v], vmn[skip_v] = 0, 0, 0
        assert torch.equal(kc.cpu(), codes)
        assert torch.equal(km.cpu(), torch.stack([s[..., 0], mn[..., 0]], -1))
        assert torch.equal(vc.cpu(), vcodes)
        assert torch.equal(vm.cpu(), torch.stack([vs[..., 0], vmn[..., 0]], -1))
    finally:
        B.kvb_destroy(ctx)


@pytest.mark.parametrize("Hkv,bits,compact", [(1, 8, False), (2, 8, True), (2, 4, False), (4, 4, True)])
def test_quantiser_whose_loads_stop_reports_it_and_writes_nothing_else(Hkv, bits, compact):
    """The fetching warps stop a different number of tiles into every CTA (none in some), as if the loads never landed:
    every wait gives up, the status says so, a tile is written as a whole or not at all, and the context stays usable."""
    sh = synth.Shape(L=36, Hq=Hkv, Hkv=Hkv)
    n, G, pad = 8 // Hkv, 1 if bits == 8 else 4, 4096
    mt = torch.float16 if compact else torch.float32
    ctx = B.create_for_shape(sh, 0)
    try:
        g = torch.Generator(device=DEV).manual_seed(3)
        k, v = (torch.randn((n, sh.L, sh.C, Hkv, sh.d), generator=g, device=DEV).to(sh.torch_dtype) for _ in range(2))
        shapes = {"k_codes": (n, sh.L, sh.C, Hkv, sh.d * bits // 8), "v_codes": (n, sh.L, sh.C, Hkv, sh.d * bits // 8),
                  "k_meta": (n, sh.L, G, Hkv, sh.d, 2 * mt.itemsize), "v_meta": (n, sh.L, sh.C, Hkv, G, 2 * mt.itemsize)}
        size = {a: int(np.prod(s)) for a, s in shapes.items()}
        pool = torch.empty(sum(size.values()) + pad * (len(size) + 1), dtype=torch.uint8, device=DEV)
        guard = torch.ones(pool.numel(), dtype=torch.bool, device=DEV)
        out, at = {}, pad
        for a, s in shapes.items():
            out[a] = pool[at : at + size[a]].view(s)
            guard[at : at + size[a]] = False
            at += size[a] + pad
        jobs = [dict(bits=bits, unrotate_from=i - 1, meta_fp16=compact, k=k[i], v=v[i], k_codes=out["k_codes"][i], v_codes=out["v_codes"][i],
                     k_meta=out["k_meta"][i].view(mt), v_meta=out["v_meta"][i].view(mt)) for i in range(n)]

        def run(stalled):
            pool.fill_(0xA5)
            B.kvb_set_debug_option(ctx, "quantize_stalled_fetch", stalled)
            B.kvb_quantize_chunks(ctx, jobs)
            assert B.kvb_last_status(ctx, check=False) == (B.KVB_ERR_DEVICE_STATUS if stalled else B.KVB_OK)
            assert B.kvb_last_status(ctx, check=False) == B.KVB_OK
            assert bool((pool[guard] == 0xA5).all())
            # a row per tile: the tokens of one head's keys, or 128 (token, head) rows of values
            tiles = lambda a: (out[a].transpose(2, 3) if a[0] == "k" else out[a]).reshape(n * sh.L * Hkv, -1).clone()
            return torch.cat([tiles("k_codes"), tiles("k_meta")], 1), torch.cat([tiles("v_codes"), tiles("v_meta")], 1)

        want = run(0)
        for got, whole in zip(run(1), want):
            written = (got == whole).all(1)
            untouched = (got == 0xA5).all(1)
            assert bool((written | untouched).all()) and bool(written.any()) and bool(untouched.any())
        for got, whole in zip(run(0), want):
            assert torch.equal(got, whole)
    finally:
        B.kvb_destroy(ctx)


@pytest.mark.parametrize("Hkv", [1, 2])
@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("pos", [-1, 4096 + 128])
@pytest.mark.parametrize("lattice", [False, True])
def test_scales_of_every_magnitude(Hkv, bits, pos, lattice):
    """Channels and rows whose scales spread over all that bfloat16 holds, on both sides of the range in which the
    reciprocal decides, alone among ordinary ones and all over; a lattice whose every other quotient is a tie.  Codes and
    metadata equal the oracle's bit for bit, rotated keys too (a channel's partner has another magnitude)."""
    sh = synth.Shape(L=2, Hq=Hkv, Hkv=Hkv)
    top = 2 * ((1 << bits) - 1)
    g = torch.Generator().manual_seed(bits + 100 * Hkv)
    ctx = B.create_for_shape(sh, 0)
    try:
        if lattice:
            k, v = (torch.randint(0, top // 2 + 1, (sh.L, sh.C, Hkv, sh.d), generator=g).float() for _ in range(2))
            k[:, 0::32], k[:, 1::32] = 0.0, float(top)
            v[..., 0::32], v[..., 1::32] = 0.0, float(top)
        else:
            k, v = (torch.randn((sh.L, sh.C, Hkv, sh.d), generator=g) for _ in range(2))
        e = torch.linspace(-120, 116, 128).round()
        edges = torch.tensor([-106, -105, -104, -103, -102, -101, -100, -99, -98, 90, 91, 92, 93, 94, 95, 96, 97, 98, 99, 100])
        e[10 : 10 + len(edges)] = edges.float()  # scales about 1e-30 and 1e30 for ranges of 16 and 256 steps
        e = e[torch.randperm(128, generator=g)]
        k[0] *= torch.exp2(e)             # layer 0: every channel and every row another magnitude
        v[0] *= torch.exp2(e).view(-1, 1, 1)
        k[1, ..., 70] *= 2.0**-110        # layer 1: one of either among ordinary ones
        v[1, 70] *= 2.0**110
        k, v = k.to(sh.torch_dtype), v.to(sh.torch_dtype)
        G = 1 if bits == 8 else 4
        out = dict(k_codes=torch.zeros((sh.L, sh.C, Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV), k_meta=torch.zeros((sh.L, G, Hkv, sh.d, 2), device=DEV),
                   v_codes=torch.zeros((sh.L, sh.C, Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV), v_meta=torch.zeros((sh.L, sh.C, Hkv, G, 2), device=DEV))
        B.kvb_quantize_chunks(ctx, [dict(bits=bits, k=k.to(DEV), v=v.to(DEV), unrotate_from=pos, **out)])
        B.kvb_last_status(ctx)
        gk, gv = (sh.C, sh.d) if bits == 8 else (sh.int4_group, sh.int4_group)
        for l in range(sh.L):
            u = oracle.unrotate_keys(helpers.bits_of(k)[l], helpers.dt_code(sh), sh.theta, pos) if pos >= 0 else helpers.f64_of(k)[l]
            for side, (codes, meta) in (("k", oracle.quantize_k(u, bits, gk)), ("v", oracle.quantize_v(helpers.f64_of(v)[l], bits, gv))):
                assert np.array_equal(out[side + "_codes"][l].cpu().numpy(), codes), (side, l)
                assert np.array_equal(out[side + "_meta"][l].cpu().numpy(), meta), (side, l)
    finally:
        B.kvb_destroy(ctx)


def _eq6_of_numbers(x, bits):
    """Eq. 6 on [..., group] rows with the NaNs left out of the extremes; a quotient that is no number gives code 0."""
    x = x.float()
    nan = torch.isnan(x)
    mn = torch.where(nan, float("inf"), x).amin(-1, keepdim=True)
    mx = torch.where(nan, -float("inf"), x).amax(-1, keepdim=True)
    s = torch.where(mx > mn, (mx - mn) / float(2**bits - 1), torch.ones_like(mn))
    codes = torch.round((x - mn) / s)
    return torch.where(torch.isnan(codes), 0.0, torch.clamp(codes, 0, 2**bits - 1)), s, mn


@pytest.mark.parametrize("kv_dtype", ["bf16", "fp16"])
@pytest.mark.parametrize("bits", [8, 4])
@pytest.mark.parametrize("rotated", [False, True])
def test_values_that_are_no_numbers_stay_in_their_place(kv_dtype, bits, rotated):
    """NaN and infinity in even and odd channels, alone and all over a group, keys and values: codes and metadata equal
    Eq. 6 bit for bit, those of the groups beside it among them, and a NaN has code 0."""
    sh = synth.Shape(L=1, Hq=2, Hkv=2, kv_dtype=kv_dtype)
    nan, inf = float("nan"), float("inf")
    ctx = B.create_for_shape(sh, 0)
    try:
        g = torch.Generator().manual_seed(17)
        k, v = (torch.randn((sh.L, sh.C, sh.Hkv, sh.d), generator=g) for _ in range(2))
        for i, c in enumerate((4, 9, 14, 19)):  # every parity and place of a thread's four channels
            k[:, 5 + 31 * i, :, c] = nan
            v[:, 3 + i, :, c + 32 * (i & 1)] = nan
        k[:, 70, :, 24], k[:, 71, :, 27], k[:, 72, :, 33], k[:, 73, :, 33] = inf, -inf, inf, -inf
        k[..., 40], k[..., 41], k[..., 50] = inf, -inf, nan
        v[:, 10, :, 10], v[:, 11, :, 11], v[:, 12, :, 64], v[:, 12, :, 67] = inf, -inf, inf, -inf
        v[:, 13], v[:, 14], v[:, 15] = inf, -inf, nan
        k, v = k.to(sh.torch_dtype), v.to(sh.torch_dtype)
        G = 1 if bits == 8 else 4
        out = dict(k_codes=torch.zeros((sh.L, sh.C, sh.Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV), k_meta=torch.zeros((sh.L, G, sh.Hkv, sh.d, 2), device=DEV),
                   v_codes=torch.zeros((sh.L, sh.C, sh.Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV), v_meta=torch.zeros((sh.L, sh.C, sh.Hkv, G, 2), device=DEV))
        B.kvb_quantize_chunks(ctx, [dict(bits=bits, k=k.to(DEV), v=v.to(DEV), unrotate_from=0 if rotated else -1, **out)])
        B.kvb_last_status(ctx)
        u = k.float()
        if rotated:  # by the angle 0: cos 1, sin 0 (0 times infinity is no number)
            lo, hi = u[..., :64], u[..., 64:]
            u = torch.cat([lo + hi * 0.0, hi + lo * -0.0], -1)
        x = {"k": u.view(sh.L, G, sh.C // G, sh.Hkv, sh.d).permute(0, 1, 3, 4, 2), "v": v.float().view(sh.L, sh.C, sh.Hkv, G, sh.d // G)}
        back = {"k": lambda t: t.permute(0, 1, 4, 2, 3).reshape(k.shape), "v": lambda t: t.reshape(v.shape)}
        for side in ("k", "v"):
            codes, s, mn = _eq6_of_numbers(x[side], bits)
            none = torch.isnan(x[side]).all(-1, keepdim=True)  # a group without a number
            if side == "v" or not rotated:
                mn = torch.where(none, nan, mn)
            else:
                assert torch.equal(mn[none], torch.full_like(mn[none], inf))
            got = out[side + "_codes"].cpu()
            if bits == 4:
                got = torch.stack([got & 15, got >> 4], -1).flatten(-2)
            assert bool((torch.isnan(x[side]) & ~none).any()) and torch.equal(got, back[side](codes).to(torch.uint8))
            np.testing.assert_array_equal(out[side + "_meta"].cpu().numpy(), torch.stack([s[..., 0], mn[..., 0]], -1).numpy())
    finally:
        B.kvb_destroy(ctx)


@pytest.mark.parametrize("side", ["k", "v"])
@pytest.mark.parametrize("Hkv", [1, 16])
def test_long_runs_of_one_side(side, Hkv):
    """Sixteen chunks of 36 layers, one side only, again and again: tens of tiles for every CTA, all of a kind, as fast as
    they come, so that loads land out of order and the warps of a group drift apart.  Codes and metadata of every call equal
    Eq. 6 bit for bit."""
    sh = synth.Shape(L=36, Hq=16, Hkv=Hkv)
    n = 256 // Hkv
    ctx = B.create_for_shape(sh, 0)
    try:
        g = torch.Generator(device=DEV).manual_seed(5)
        x = torch.empty((n, sh.L, sh.C, Hkv, sh.d), dtype=sh.torch_dtype, device=DEV)
        want_codes = torch.empty(x.shape, dtype=torch.uint8, device=DEV)
        meta_shape = (n, sh.L, 1, Hkv, sh.d, 2) if side == "k" else (n, sh.L, sh.C, Hkv, 1, 2)
        want_meta = torch.empty(meta_shape, device=DEV)
        for i in range(n):
            x[i] = torch.randn(x.shape[1:], generator=g, device=DEV)
            rows = x[i].permute(0, 2, 3, 1) if side == "k" else x[i]  # tokens, or channels, last
            mn, mx = rows.float().amin(-1, keepdim=True), rows.float().amax(-1, keepdim=True)
            s = (mx - mn) / torch.full_like(mn, 255.0)  # (a division by a number would be a multiplication by its reciprocal)
            codes = torch.round((rows.float() - mn) / s)
            want_codes[i] = codes.permute(0, 3, 1, 2) if side == "k" else codes
            want_meta[i] = torch.cat([s, mn], -1).view(meta_shape[1:])
        codes, meta = torch.empty_like(want_codes), torch.empty_like(want_meta)
        jobs = B.QuantizeTable([{"bits": 8, side: x[i], side + "_codes": codes[i], side + "_meta": meta[i]} for i in range(n)])
        for _ in range(20):
            codes.zero_(), meta.zero_()
            for _ in range(5):
                B.kvb_quantize_chunks(ctx, jobs)
            B.kvb_last_status(ctx)
            assert torch.equal(codes, want_codes) and torch.equal(meta, want_meta)
    finally:
        B.kvb_destroy(ctx)


@pytest.mark.parametrize("n_jobs,L,Hkv,kv_dtype", [(1000, 1, 1, "bf16"), (250, 3, 2, "fp16"), (40, 12, 4, "fp16"), (3, 36, 16, "bf16")])
@pytest.mark.parametrize("sides", [("kv", "k", "v", "v", "kv"), ("k",), ("v", "k")])
def test_jobs_of_every_kind_over_many_tiles(n_jobs, L, Hkv, kv_dtype, sides):
    """Keys only, values only and both, either code width, compact metadata or not, every job with a position of its own, in
    one call of many more tiles than a CTA has buffers (and of more rotations than it keeps).  Codes and metadata equal the
    oracle's bit for bit."""
    sh = synth.Shape(L=L, Hq=Hkv, Hkv=Hkv, kv_dtype=kv_dtype)
    dtc = helpers.dt_code(sh)
    ctx = B.create_for_shape(sh, 0)
    try:
        xs = [(_keys(sh, 400 + i), _keys(sh, 500 + i)) for i in range(3)]  # jobs share their inputs, not their outputs
        dev = [(k.to(DEV), v.to(DEV)) for k, v in xs]
        oracle_in = [(helpers.bits_of(k), helpers.f64_of(k), helpers.f64_of(v)) for k, v in xs]
        jobs, spec = [], []
        for i in range(n_jobs):
            side, bits, m16, pos = sides[i % len(sides)], 8 if i // 3 % 2 else 4, i % 4 == 1, -1 if i % 7 == 3 else 128 * i
            mt, G = torch.float16 if m16 else torch.float32, 1 if bits == 8 else 4
            j = dict(bits=bits, unrotate_from=pos, meta_fp16=m16)
            for s, x, meta in (("k", dev[i % 3][0], (L, G, Hkv, sh.d, 2)), ("v", dev[i % 3][1], (L, sh.C, Hkv, G, 2))):
                if s in side:
                    j.update({s: x, s + "_codes": torch.zeros((L, sh.C, Hkv, sh.d * bits // 8), dtype=torch.uint8, device=DEV), s + "_meta": torch.zeros(meta, dtype=mt, device=DEV)})
            jobs.append(j)
            spec.append((side, bits, m16, pos))
        B.kvb_quantize_chunks(ctx, jobs)
        B.kvb_last_status(ctx)
        values = {}  # (input, width, compact) -> the oracle's values
        for i, (j, (side, bits, m16, pos)) in enumerate(zip(jobs, spec)):
            kb, k64, v64 = oracle_in[i % 3]
            gk, gv = (sh.C, sh.d) if bits == 8 else (sh.int4_group, sh.int4_group)
            if "k" in side and (n_jobs < 100 or i % 9 < 3):
                got_c, got_m = j["k_codes"].cpu().numpy(), j["k_meta"].float().cpu().numpy()
                for l in range(L):
                    u = oracle.unrotate_keys(kb[l], dtc, sh.theta, pos) if pos >= 0 else k64[l]
                    c, m = oracle.quantize_k(u, bits, gk, meta16=m16)
                    assert np.array_equal(got_c[l], c) and np.array_equal(got_m[l], m.astype(np.float32)), ("keys", i, l)
            if "v" in side:
                key = (i % 3, bits, m16)
                if key not in values:
                    r = [oracle.quantize_v(v64[l], bits, gv, meta16=m16) for l in range(L)]
                    values[key] = np.stack([c for c, _ in r]), np.stack([m for _, m in r]).astype(np.float32)
                assert np.array_equal(j["v_codes"].cpu().numpy(), values[key][0]) and np.array_equal(j["v_meta"].float().cpu().numpy(), values[key][1]), ("values", i)
    finally:
        B.kvb_destroy(ctx)
