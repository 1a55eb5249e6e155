// KV Quantization, Eq. 6 (cache-population side): asymmetric min/max quantisation of cached
// chunks, keys per channel over a token group, values per token over a channel group.
// scale = (max-min)/(2^b-1) and min are float32; the code is rint((x-min)/scale) in float32
// (IEEE subtract, divide, round-half-even), clamped.  A constant group gets scale 1, codes 0.
//
// One launch quantises a batch of chunks.  Work unit: a tile of 128 rows x 128 channels (32 KB):
//   keys    the 128 tokens of one (chunk, layer, KV head)
//   values  128 consecutive (token, head) rows of one (chunk, layer)
// One persistent CTA per SM walks a contiguous range of the wanted tiles: three groups of eight warps work on a tile each,
// four more warps fetch ahead into a ring of five tile buffers (one bulk copy where the tile is contiguous, cp.async by
// token rows for one head of several: a bulk copy per 256-byte row took twice the time), and hand over through mbarriers,
// so that loads go on while tiles are in work.  Bound by the instructions of the code decision and, for plain values, by
// HBM.  64 chunks of 36 layers and 2 heads, one side only, before (one CTA of eight warps per 64 KB tile, loading and
// computing in turn) and now: int8 values 53.0 / 39.1 us (36 us at the copy rate), int4 values 61.5 / 40.7, int8 keys
// 52.7 / 44.5, int4 keys 54.7 / 46.4, rotated int4 keys 70.8 / 61.2; both sides of a 16K-token prompt to int4,
// position-free and compact: 216 / 182, of a 2K-token prompt to int8: 29.6 / 23.1 (one launch instead of two: up to 256
// jobs travel as the kernel's argument).  Two groups, with registers to spare, measured 3-8 % slower; consumer warps
// fetching for themselves likewise.
//   keys    a thread owns a quad of neighbouring channels, their rotation partners 64 channels on, and eight tokens.
//           Without the rotation the extremes are taken on the 16-bit values, two per instruction.  With `unrotate`
//           every key is first rotated back by R_theta^(-orig_pos) (Rotary Positional Embeddings, Eq. 3), so that the
//           stored chunk is position-free and re-use at new_pos needs the single rotation by new_pos; cos / sin come
//           from a double-precision angle, once per chunk and CTA, the rotation itself is float32 in a fixed order:
//           u = fma(x, c, +-(x_partner * s)).  The warps' extremes meet in shared memory, where (scale, min) and the
//           reciprocal are worked out once per (token group, channel).
//   values  eight lanes per (token, head) row, 16 channels per lane, the extremes reduced by shuffles of packed 16-bit
//           words, (scale, min) and the reciprocal worked out by a lane per (row, channel group).
// The code decision takes no division: see code_pair.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <string.h>

#include <type_traits>

#include "f32x2.cuh"
#include "kvb_internal.h"
#include "pdl.cuh"

namespace kvb {
namespace {

constexpr int kWarps = 8;      // warps of a group, which works on one tile at a time
constexpr int kGroups = 3;     // groups of a CTA
constexpr int kFetchers = 4;   // more warps, which fetch
constexpr int kThreads = (kGroups * kWarps + kFetchers) * 32;
constexpr int kRows = 128;     // rows of a tile: the tokens of a chunk, or that many (token, head) rows
constexpr int kD = 128;        // head_dim
constexpr int kRowsPerWarp = kRows / kWarps;
constexpr uint32_t kTileBytes = kRows * kD * 2;
constexpr uint32_t kWaitLimit = 1u << 22;         // polls after which a wait gives up
constexpr uint32_t kStalledWaitLimit = 1u << 10;  // the same in a launch whose fetching warps are made to stop (option quantize_stalled_fetch)
constexpr int kStages = 5;     // tile buffers: one in work per group, the others in flight
// Barriers on which tiles land, two for each group: tile t of a CTA has barrier t mod 6, lap t / 6.  (One per buffer would not
// do.  A wait goes by the parity of the lap, so whoever waits for a lap must know that the one before is over.  The barrier's
// tile before, t - 6, is the same group's: the warp has worked on it.  The buffer's tile before, t - 5, is another group's, and
// copies land in any order: a warp that is early would take its parity for its own tile's.)
constexpr int kLandings = 2 * kGroups;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait of a whole warp: gives up after `limit` polls (never expected; keeps a bad launch from hanging).  Every lane
// gets the same answer.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if (i > 64) __nanosleep(64);
  }
  return false;
}
// The same for a single lane, whose answer may differ from its neighbours': without the vote 58 chunks of keys and values to
// int4 take 73.2 instead of 73.9 us.
__device__ __forceinline__ bool mbar_wait_lane(uint64_t* bar, uint32_t parity, uint32_t limit) {
  for (uint32_t i = 0; i < limit; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (i > 64) __nanosleep(64);
  }
  return false;
}
// a group's own barrier
__device__ __forceinline__ void group_sync(int group) { asm volatile("bar.sync %0, %1;" ::"r"(group + 1), "n"(kWarps * 32) : "memory"); }
// After a lane's wait for its group's tile has run out: true if the tile has landed after all, false if the wait has run out
// for every lane of the group (`gave_up` counts them; all of them is final).  So the lanes of a group leave together or go on
// together, and none is left waiting for another in group_sync or a shuffle.  It ends: a tile that one lane has seen stays
// until all are through with it, and a lane that has not seen it gives up too.
__device__ __noinline__ bool landed_late(uint64_t* bar, uint32_t parity, uint32_t limit, uint32_t* gave_up) {
  uint32_t n = atomicAdd(gave_up, 1u) + 1u;
  for (uint32_t i = 0; i < limit && n < (uint32_t)kWarps * 32; ++i) {
    if (mbar_try_wait(bar, parity)) {
      const uint32_t seen = atomicCAS(gave_up, n, n - 1u);
      if (seen == n) return true;
      n = seen;
    } else {
      __nanosleep(64);
      n = *reinterpret_cast<volatile uint32_t*>(gave_up);
    }
  }
  return false;
}
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_u32(dst)),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void cp_async16(void* dst, const void* src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
// the barrier's current phase also waits for the thread's copies so far
__device__ __forceinline__ void cp_async_arrive(uint64_t* bar) {
  asm volatile("cp.async.mbarrier.arrive.shared::cta.b64 [%0];" ::"r"(smem_u32(bar)) : "memory");
}

constexpr float kMagic = 8388608.0f;  // 2^23
// The code of a value: rint(x / s) clamped to [0, levels], x = v - mn, subtraction and division being IEEE float32.
// The quotient is the IEEE one by Markstein's theorem (P. Markstein, Computation of elementary functions on the IBM
// RISC System/6000 processor, IBM J. Res. Dev. 34, 1990; Handbook of Floating-Point Arithmetic, section on division
// with an FMA): with y = RN(1 / s) and q within one unit in the last place of x / s, r = x - q s is exact in float32
// and RN(q + r y) = RN(x / s).  The q it starts from is x y + x y_lo, y_lo the rest of the reciprocal: half a unit and
// a rounding error of x y_lo off, at most.  Adding 2^23 rounds the quotient to an integer (round-half-even, as rint
// does) and leaves it in the low mantissa bits.  No clamp is needed, the quotient cannot exceed levels by more than a
// rounding error.  Six packed instructions for two values; two bounds on the quotient with a list of the undecided values
// (0.4 % of 16-bit data are ties or next to one) redone by division took five and as many again for the list.
__device__ __forceinline__ void code_pair(uint64_t v, uint64_t mn, uint64_t y, uint64_t y_lo, uint64_t neg_s, uint32_t& m0, uint32_t& m1) {
  const uint64_t x = f2_sub(v, mn);
  const uint64_t q = f2_fma(x, y, f2_mul(x, y_lo));
  const uint64_t m = f2_add(f2_fma(f2_fma(q, neg_s, x), y, q), f2_pack(kMagic, kMagic));
  float a, b;
  f2_unpack(m, a, b);
  m0 = __float_as_uint(a), m1 = __float_as_uint(b);
}
// not inlined: the compiler must not evaluate the division speculatively on the common path
__device__ __noinline__ uint32_t code_exact(float v, float mn, float s, float levels) {
  float c = rintf(__fdiv_rn(__fsub_rn(v, mn), s));
  c = fminf(fmaxf(c, 0.f), levels);
  return (uint32_t)c;
}
// y = RN(1 / s); the rest of the reciprocal is y (1 - y s).  Within 1e-30 .. 1e30 code_pair's remainder is exact for every
// quotient that can decide (from 1/4 on it is a multiple of 2^-25 2^-23 2^-100, above float32's smallest number) and nothing
// overflows.  Outside, and in a group with a value that is no number or whose minimum is infinite, y is zero, and the IEEE
// division decides for the group: a NaN gets code 0, and so do the values of a group without a finite one.
__device__ __forceinline__ float reciprocal(float s) { return s >= 1e-30f && s <= 1e30f ? __frcp_rn(s) : 0.f; }
// minimum / maximum of two or three values in which a NaN stays
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float max_nan(float a, float b) {
  float d;
  asm("max.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float min_nan(float a, float b, float c) {
  float d;
  asm("min.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
__device__ __forceinline__ float max_nan(float a, float b, float c) {
  float d;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// four codes, each in the low byte of m_i, as one word (code 0 in the lowest byte)
__device__ __forceinline__ uint32_t pack4_u8(const uint32_t (&m)[4]) {
  return __byte_perm(__byte_perm(m[0], m[1], 0x0040), __byte_perm(m[2], m[3], 0x0040), 0x5410);
}
// four 4-bit codes in the low bits of m_i as 16 bits (code 0 in the lowest nibble); the rest of the word is zero
__device__ __forceinline__ uint32_t pack4_u4(const uint32_t (&m)[4]) {
  return __byte_perm(m[1] * 16u + m[0], m[3] * 16u + m[2], 0x0040) & 0xFFFFu;
}

// two 16-bit values of one 32-bit word as a packed float32 pair
template <int DT>
__device__ __forceinline__ uint64_t unpack2(uint32_t w) {
  if (DT == KVB_DT_BF16) return f2_pack(__uint_as_float(w << 16), __uint_as_float(w & 0xFFFF0000u));
  const float2 t = __half22float2(*reinterpret_cast<const __half2*>(&w));
  return f2_pack(t.x, t.y);
}
// element-wise minimum / maximum of two words of two 16-bit values each (exact: no rounding is involved; a NaN stays)
template <int DT>
__device__ __forceinline__ uint32_t min2_16(uint32_t a, uint32_t b) {
  uint32_t r;
  if (DT == KVB_DT_BF16) {
    const __nv_bfloat162 t = __hmin2_nan(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    r = *reinterpret_cast<const uint32_t*>(&t);
  } else {
    const __half2 t = __hmin2_nan(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
    r = *reinterpret_cast<const uint32_t*>(&t);
  }
  return r;
}
template <int DT>
__device__ __forceinline__ uint32_t max2_16(uint32_t a, uint32_t b) {
  uint32_t r;
  if (DT == KVB_DT_BF16) {
    const __nv_bfloat162 t = __hmax2_nan(*reinterpret_cast<const __nv_bfloat162*>(&a), *reinterpret_cast<const __nv_bfloat162*>(&b));
    r = *reinterpret_cast<const uint32_t*>(&t);
  } else {
    const __half2 t = __hmax2_nan(*reinterpret_cast<const __half2*>(&a), *reinterpret_cast<const __half2*>(&b));
    r = *reinterpret_cast<const uint32_t*>(&t);
  }
  return r;
}

template <int DT>
__device__ __forceinline__ float value_of(const void* p) {
  float a, b;
  f2_unpack(unpack2<DT>(*reinterpret_cast<const uint16_t*>(p)), a, b);
  return a;
}

// The extremes of a group with a NaN among its N values (16 bits each, STRIDE bytes apart): those of the others.  Rotated
// keys: r is the channel's cos / sin, the partner's value lies `partner` bytes on.  A group of NaNs alone has the minimum NaN,
// rotated keys +inf.
template <int DT, bool ROT, int N, int STRIDE>
__device__ __noinline__ float2 number_extremes(const uint8_t* x, const float2* r, int partner) {
  const uint16_t none = 0x7FFF;
  float mn = ROT ? INFINITY : value_of<DT>(&none), mx = ROT ? -INFINITY : mn;
#pragma unroll 16
  for (int i = 0; i < N; ++i, x += STRIDE) {
    float v = value_of<DT>(x);
    if (ROT) v = fmaf(v, r->x, __fmul_rn(value_of<DT>(x + partner), partner < 0 ? -r->y : r->y));  // as in the kernel
    mn = fminf(mn, v), mx = fmaxf(mx, v);
  }
  return make_float2(mn, mx);
}

// (scale, min) of a group from its extremes.  Compact metadata: min is rounded down to binary16
// first, the scale is taken against the rounded min and rounded up, so no value leaves the code range.
__device__ __forceinline__ void group_params(float& mn, float mx, float levels, int meta16, float& s) {
  if (meta16) mn = __half2float(__float2half_rd(mn));
  s = mx > mn ? __fdiv_rn(__fsub_rn(mx, mn), levels) : 1.0f;
  if (meta16) s = __half2float(__float2half_ru(s));
}
__device__ __forceinline__ void store_meta(float* meta, uint32_t pair, float s, float mn, int meta16) {
  if (meta16) {
    reinterpret_cast<__half2*>(meta)[pair] = __floats2half2_rn(s, mn);  // both already binary16 values
  } else {
    *reinterpret_cast<float2*>(meta + pair * 2) = make_float2(s, mn);
  }
}

// the metadata of pair number `pairs` onward
__device__ __forceinline__ float* meta_from(float* meta, size_t pairs, int meta16) {
  return reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(meta) + pairs * (meta16 ? 4 : 8));
}

// The call's jobs: by value in the kernel's argument, or a table in device memory when they do not fit.
template <int N>
struct InlineJobs {
  QuantJob d[N];
};
template <int N>
__device__ __forceinline__ const QuantJob& job_at(const InlineJobs<N>& t, uint32_t j) { return t.d[j]; }
__device__ __forceinline__ const QuantJob& job_at(const QuantJob* t, uint32_t j) { return t[j]; }

// One tile of the batch.  The wanted tiles are numbered job-major, then layer, then K|V, then the H tiles of a chunk-layer; a
// side that a job does not want has no numbers, so that the CTAs' ranges hold equal work.
struct Tile {
  uint32_t job;
  int l, kv, h;
  bool both;  // the job wants both sides
  // per_job: the tiles of every job, 0 where they differ (then the job is the last one that starts at or before the item)
  template <typename Jobs>
  __device__ __forceinline__ Tile(const Jobs& jobs, uint32_t item, uint32_t n_jobs, uint32_t per_job, int log_h) {
    if (per_job) {
      job = item / per_job;
    } else {
      uint32_t lo = 0, hi = n_jobs - 1;
      while (lo < hi) {
        const uint32_t mid = (lo + hi + 1) >> 1;
        if (job_at(jobs, mid).tile_offset <= item) lo = mid; else hi = mid - 1;
      }
      job = lo;
    }
    enter(jobs);
    item -= job_at(jobs, job).tile_offset;
    h = (int)(item & ((1u << log_h) - 1u));
    item >>= log_h;
    if (both) kv = (int)(item & 1u), item >>= 1;
    l = (int)item;
  }
  // to the first tile of `job`
  template <typename Jobs>
  __device__ __forceinline__ void enter(const Jobs& jobs) {
    const QuantJob& jb = job_at(jobs, job);
    l = 0, h = 0, kv = jb.k ? 0 : 1, both = jb.k && jb.v;
  }
  template <typename Jobs>
  __device__ __forceinline__ void next(const Jobs& jobs, int H, int L, bool more) {
    if (++h < H) return;
    h = 0;
    if (both) {
      kv ^= 1;
      if (kv) return;
    }
    if (++l < L || !more) return;
    ++job;
    enter(jobs);
  }
};

// What the fetching warps tell the others about a tile.
struct __align__(16) TileDesc {
  uint8_t* codes;  // the tile's first code and first (scale, min) pair
  float* meta;     // NULL codes: no more tiles
  int32_t kv, bits, meta16, rot;  // rot: the tile's table in s_rot, -1 when its keys are not rotated
};

// Every warp's kilobyte of scratch: the minima and maxima per channel of its part of a keys tile, or the groups of its
// rows of a values tile.  The channels of every other warp are shifted by 16, so that a read of 16 channels of two
// neighbouring warps hits 32 banks.
__device__ __forceinline__ int ext_at(int w, int max, int ch) { return w * 2 * kD + max * kD + (ch ^ ((w & 1) << 4)); }

// The codes of the groups outside the reciprocal's range, decided again by the division once the warp has stored the codes of
// its part of a tile.  All lanes share the work: 16 chunks of 36 layers and 2 heads, one channel and one row of each at 1e-35,
// take 29 (int8) and 36 us (rotated int4) against 23 and 28 with none; the lanes that own them alone took 69 and 83.
// keys: a byte column (a channel, or a pair of 4-bit ones) of the warp's 16 tokens per half-warp
template <int DT, int BITS, bool ROT>
__device__ __noinline__ void redo_keys(const uint8_t* tile, const float (*par)[4 * kD], const float2* rot, uint8_t* codes, uint32_t row_stride, int warp) {
  constexpr float levels = (float)((1 << BITS) - 1);
  const int lane = threadIdx.x & 31, p = lane & 15, t = warp * kRowsPerWarp + p;
  const int g0 = BITS == 8 ? 0 : warp / (kWarps / 4) * kD;  // the token group's first channel in `par`
  uint32_t odd = 0;  // bit 4 side + e: channel 4 p + e of that side
  for (int n = 0; n < 8; ++n) odd |= (par[1][g0 + (n >> 2) * (kD / 2) + 4 * p + (n & 3)] > 0.f ? 0u : 1u) << n;
  if (BITS == 4) odd = (odd | odd >> 1) & 0x55u;
  __syncwarp();  // the codes stored before come first
  for (uint32_t who; (who = __ballot_sync(0xffffffffu, odd != 0) & 0xFFFFu) != 0;) {
    const uint32_t more = who & (who - 1);
    const int q0 = __ffs(who) - 1, q1 = more ? __ffs(more) - 1 : q0;  // a lane whose channels are odd for each half-warp
    const int q = lane < 16 ? q0 : q1, n = __ffs(__shfl_sync(0xffffffffu, odd, q)) - 1;
    if (p == q0 || p == q1) odd &= odd - 1;
    const int side = n >> 2;
    uint32_t w = 0;
#pragma unroll
    for (int e = 0; e < 8 / BITS; ++e) {
      const int c = 4 * q + (n & 3) + e;
      const uint8_t* const at = tile + t * (kD * 2) + 2 * c;  // the low channel; its partner 64 channels on
      float v = value_of<DT>(at + side * kD);
      if (ROT) v = fmaf(v, rot[c].x, __fmul_rn(value_of<DT>(at + (side ^ 1) * kD), side ? -rot[c].y : rot[c].y));  // as in `rotated`
      const int gc = g0 + side * (kD / 2) + c;
      w |= code_exact(v, par[0][gc], -par[2][gc], levels) << (BITS * e);
    }
    codes[(uint32_t)t * row_stride + (uint32_t)(side * (kD / 2) + 4 * q + (n & 3)) * BITS / 8] = (uint8_t)w;
  }
}
// values: a group of a row per 32 or 8 lanes, four channels a lane.  s_row: (min, reciprocal, its rest, -scale) of [row][group]
template <int DT, int BITS>
__device__ __noinline__ void redo_values(const uint8_t* tile, const float4* s_row, uint8_t* codes, int warp) {
  constexpr float levels = (float)((1 << BITS) - 1);
  constexpr int G = BITS == 8 ? 1 : kD / 32, kLanes = 32 / G;
  const int lane = threadIdx.x & 31;
  __syncwarp();  // the codes stored before come first
  for (int n0 = warp * kRowsPerWarp * G; n0 < (warp + 1) * kRowsPerWarp * G; n0 += 32) {
    const int n_here = min(32, kRowsPerWarp * G);
    uint32_t odd = __ballot_sync(0xffffffffu, lane < n_here && !(s_row[n0 + min(lane, n_here - 1)].y > 0.f));
    while (odd) {  // G groups at a time
      uint32_t mine = odd;
#pragma unroll
      for (int i = 0; i < G; ++i) {
        if (i < lane / kLanes) mine &= mine - 1;
        odd &= odd - 1;
      }
      if (mine == 0) continue;
      const int n = n0 + __ffs(mine) - 1, row = n / G, ch = (n & (G - 1)) * (kD / G) + 4 * (lane & (kLanes - 1));
      const float4 g = s_row[n];
      uint32_t w = 0;
#pragma unroll
      for (int e = 0; e < 4; ++e) w |= code_exact(value_of<DT>(tile + row * (kD * 2) + 2 * (ch + e)), g.x, -g.w, levels) << (BITS * e);
      uint8_t* const o = codes + (row * kD + ch) * BITS / 8;
      if (BITS == 8) *reinterpret_cast<uint32_t*>(o) = w;
      else *reinterpret_cast<uint16_t*>(o) = (uint16_t)w;
    }
  }
}

template <int DT, typename Jobs>
__global__ void __launch_bounds__(kThreads, 1)
    quantize_batch_kernel(const __grid_constant__ Jobs jobs, ModelDims m, uint32_t n_jobs, uint32_t n_items, uint32_t per_job, const double* __restrict__ inv_freq,
                          uint32_t* __restrict__ status, bool stalled) {
  extern __shared__ __align__(128) uint8_t smem[];  // kStages tiles
  __shared__ __align__(16) float s_ext_all[kGroups][kWarps * 2 * kD];  // see ext_at
  __shared__ __align__(16) float s_par_all[kGroups][3][4 * kD];        // keys: min, reciprocal and -scale of every [token group][channel]
  __shared__ float2 s_rot[kStages][kD / 2];               // cos / sin of a chunk's rotation; a ring, in use by at most kStages tiles
  __shared__ TileDesc s_tile[kStages];
  __shared__ __align__(8) uint64_t s_full[kLandings], s_empty[kStages];
  __shared__ uint32_t s_gave_up[kGroups];  // lanes of the group whose wait for the tile ran out
  const int lane = threadIdx.x & 31, warp = (threadIdx.x >> 5) & (kWarps - 1), group = threadIdx.x / (kWarps * 32);
  const int tid = threadIdx.x & (kWarps * 32 - 1);  // within the group
  const int H = m.Hkv, log_h = __ffs(H) - 1;
  const size_t layer_elems = (size_t)kRows * H * kD;
  // a contiguous range of tiles per CTA: its tiles mostly belong to one chunk (one rotation), and ranges differ by one tile
  const uint32_t first = (uint32_t)((unsigned long long)n_items * blockIdx.x / gridDim.x);
  const uint32_t last = (uint32_t)((unsigned long long)n_items * (blockIdx.x + 1) / gridDim.x);

  if (threadIdx.x < kLandings) {
    mbar_init(&s_full[threadIdx.x], kFetchers);
    if (threadIdx.x < kStages) mbar_init(&s_empty[threadIdx.x], kWarps);
    if (threadIdx.x < kGroups) s_gave_up[threadIdx.x] = 0;
  }
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  __syncthreads();
  pdl_wait();  // inputs may come from the kernel before this one, and it may still read what this one writes

  // A wait that runs out sets the status and ends the warp (a group's lanes together, see landed_late): it knows neither the
  // tile nor where its codes belong.  The fetching warps that wait for the group's buffers then run out of a wait in turn.
  const uint32_t limit = stalled ? kStalledWaitLimit : kWaitLimit;

  if (group == kGroups) {
    // ------------------------------ the fetching warps: descriptors, rotation tables and copies, up to kStages tiles ahead
    Tile t(jobs, first, n_jobs, per_job, log_h);
    uint32_t rot_job = 0xFFFFFFFFu, stage = 0, phase = 1;  // a fresh barrier passes a wait for the phase before its first
    uint32_t landing = 0, lap = 0;                         // the tile's barrier and the parity of its lap
    int rot_buf = 0;
    const uint32_t stop = stalled ? first + blockIdx.x % (2 * kStages) : 0xFFFFFFFFu;  // a stalled fetch ends there
    for (uint32_t item = first; item < min(last + kGroups, stop); ++item, t.next(jobs, H, m.L, item < last)) {
      const bool end = item >= last;  // an end mark for every group
      const uint8_t* x = nullptr;
      TileDesc td{};
      if (!end) {
        const QuantJob& jb = job_at(jobs, t.job);
        x = static_cast<const uint8_t*>(t.kv ? jb.v : jb.k);
        const size_t at = (size_t)t.l * layer_elems + (size_t)t.h * (t.kv ? kRows * kD : kD);  // the tile's first element
        const int G = jb.bits == 8 ? 1 : 4;
        x += at * 2;
        td.codes = static_cast<uint8_t*>(t.kv ? jb.v_codes : jb.k_codes) + at * jb.bits / 8;
        td.meta = meta_from(static_cast<float*>(t.kv ? jb.v_meta : jb.k_meta),
                            t.kv ? ((size_t)t.l * H + t.h) * kRows * G : ((size_t)t.l * G * H + t.h) * kD, jb.meta16);
        td.kv = t.kv, td.bits = jb.bits, td.meta16 = jb.meta16, td.rot = -1;
      }
      if (!mbar_wait(&s_empty[stage], phase, limit)) {
        if (lane == 0) atomicOr(status, DEV_STATUS_WAIT_TIMEOUT);
        asm volatile("cp.async.wait_all;" ::: "memory");  // the copies in flight land before their buffers are given up
        for (uint32_t i = 0; i < kLandings; ++i) mbar_wait(&s_full[i], i < landing ? lap : lap ^ 1u, limit);
        return;
      }
      if (!end && !t.kv && job_at(jobs, t.job).unrotate_from >= 0) {
        if (rot_job != t.job) {
          rot_job = t.job;
          rot_buf = rot_buf == kStages - 1 ? 0 : rot_buf + 1;
          if (tid < kD / 2) {
            double s_d, c_d;
            sincos((double)job_at(jobs, t.job).unrotate_from * inv_freq[tid], &s_d, &c_d);
            s_rot[rot_buf][tid] = make_float2((float)c_d, (float)s_d);
          }
        }
        td.rot = rot_buf;
      }
      if (tid == 0) s_tile[stage] = td;
      uint8_t* const dst = smem + stage * kTileBytes;
      const bool bulk = end || t.kv || H == 1;
      if (!bulk) {  // token rows of one head, every fetching warp a part
        const uint8_t* g = x + (size_t)(tid >> 4) * H * (kD * 2) + (tid & 15) * 16;
#pragma unroll 4
        for (int i = 0; i < (int)kTileBytes / 16; i += kFetchers * 32, g += (size_t)(kFetchers * 2) * H * (kD * 2)) cp_async16(dst + (i + tid) * 16, g);
        cp_async_arrive(&s_full[landing]);
      }
      __syncwarp();
      if (lane == 0) {
        if (end || !bulk || tid != 0) mbar_arrive(&s_full[landing]);
        else {  // one contiguous block
          mbar_expect_tx(&s_full[landing], kTileBytes);
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");  // the buffer's previous tile may have come by cp.async
          bulk_g2s(dst, x, kTileBytes, &s_full[landing]);
        }
      }
      if (++stage == kStages) stage = 0, phase ^= 1;
      if (++landing == kLandings) landing = 0, lap ^= 1;
    }
    return;
  }

  // ------------------------------ the others.  Between two tiles they meet only where data changes hands: inside a keys tile.
  float* const s_ext = s_ext_all[group];
  float (*const s_par)[4 * kD] = s_par_all[group];
  uint32_t mine = 0;  // tiles of the group so far, mod 4
  for (uint32_t stage = group;;) {  // every kGroups-th tile
    if (!mbar_wait_lane(&s_full[group + kGroups * (mine & 1)], mine >> 1, limit)) {
      atomicOr(status, DEV_STATUS_WAIT_TIMEOUT);
      if (!landed_late(&s_full[group + kGroups * (mine & 1)], mine >> 1, limit, &s_gave_up[group])) return;
    }
    const TileDesc td = s_tile[stage];
    if (!td.codes) break;
    const uint8_t* const tile = smem + stage * kTileBytes;
    const int meta16 = td.meta16;

    auto values = [&](auto bits_tag) {
      constexpr int BITS = decltype(bits_tag)::value;
      constexpr float levels = (float)((1 << BITS) - 1);
      constexpr int G = BITS == 8 ? 1 : kD / 32;  // groups of a row: the whole row, or 32 channels each
      constexpr int kPieces = G == 1 ? 1 : 2;     // groups a lane takes part in
      constexpr int kLanes = G == 1 ? 8 : 4;      // lanes of a group
      constexpr int kSweeps = kRowsPerWarp / 4;   // a warp takes four rows at a time
      const int sub = lane >> 3, lj = lane & 7;
      // (min, reciprocal, its low part, -scale) of this warp's [row][group]; the group's element-wise extremes come first
      float4* const s_row = reinterpret_cast<float4*>(s_ext + warp * 2 * kD) - warp * kRowsPerWarp * G;
      // ---- extremes: a lane holds two pieces of eight channels of its row, 8 lj .. 8 lj + 7 and 64 + 8 lj .. 64 + 8 lj + 7
      const uint32_t r0 = warp * kRowsPerWarp + sub;
      const uint8_t* const tile_r = tile + r0 * (kD * 2) + 16 * lj;
#pragma unroll
      for (int it = 0; it < kSweeps; ++it) {
        const uint4 wa = *reinterpret_cast<const uint4*>(tile_r + it * 4 * (kD * 2)), wb = *reinterpret_cast<const uint4*>(tile_r + it * 4 * (kD * 2) + 128);
        uint32_t lo[2], hi[2];
        lo[0] = min2_16<DT>(min2_16<DT>(wa.x, wa.y), min2_16<DT>(wa.z, wa.w)), hi[0] = max2_16<DT>(max2_16<DT>(wa.x, wa.y), max2_16<DT>(wa.z, wa.w));
        lo[1] = min2_16<DT>(min2_16<DT>(wb.x, wb.y), min2_16<DT>(wb.z, wb.w)), hi[1] = max2_16<DT>(max2_16<DT>(wb.x, wb.y), max2_16<DT>(wb.z, wb.w));
        if (G == 1) {  // one group: both pieces, all eight lanes
          lo[0] = min2_16<DT>(lo[0], lo[1]);
          hi[0] = max2_16<DT>(hi[0], hi[1]);
        }
#pragma unroll
        for (int p = 0; p < kPieces; ++p) {
#pragma unroll
          for (int o = 1; o < kLanes; o <<= 1) {
            lo[p] = min2_16<DT>(lo[p], __shfl_xor_sync(0xffffffffu, lo[p], o));
            hi[p] = max2_16<DT>(hi[p], __shfl_xor_sync(0xffffffffu, hi[p], o));
          }
          if ((lj & (kLanes - 1)) == 0)  // channels 8 lj (+ 64) lie in group lj / 4 (+ 2)
            *reinterpret_cast<uint2*>(&s_row[(r0 + it * 4) * G + (G == 1 ? 0 : 2 * p + (lj >> 2))]) = make_uint2(lo[p], hi[p]);
        }
      }
      __syncwarp();
      // ---- (scale, min) and reciprocal of the warp's rows, a (row, group) per lane
      bool odd = false;
#pragma unroll
      for (int n0 = 0; n0 < kRowsPerWarp * G; n0 += 32) {
        const int n = n0 + lane;
        if (kRowsPerWarp * G >= 32 || n < kRowsPerWarp * G) {
          const uint32_t rg = warp * kRowsPerWarp * G + n;
          const uint2 ext = *reinterpret_cast<const uint2*>(&s_row[rg]);
          float a, b, c, d, s;
          f2_unpack(unpack2<DT>(ext.x), a, b);
          f2_unpack(unpack2<DT>(ext.y), c, d);
          float mn = min_nan(a, b), mx = max_nan(c, d);
          const bool numbers = fabsf(mn) < INFINITY;
          if (mn != mn) {
            const float2 e = number_extremes<DT, false, kD / G, 2>(tile + rg * (kD / G * 2), nullptr, 0);
            mn = e.x, mx = e.y;
          }
          group_params(mn, mx, levels, meta16, s);
          store_meta(td.meta, rg, s, mn, meta16);
          const float y = numbers ? reciprocal(s) : 0.f;
          s_row[rg] = make_float4(mn, y, y * fmaf(-y, s, 1.f), -s);
          odd |= !(y > 0.f);
        }
      }
      odd = __any_sync(0xffffffffu, odd);
      __syncwarp();
      // ---- codes
      uint8_t* const out_r = td.codes + r0 * (kD * BITS / 8) + lj * BITS;
#pragma unroll
      for (int it = 0; it < kSweeps; ++it) {
        const uint4 wa = *reinterpret_cast<const uint4*>(tile_r + it * 4 * (kD * 2)), wb = *reinterpret_cast<const uint4*>(tile_r + it * 4 * (kD * 2) + 128);
        const uint32_t w[2][4] = {{wa.x, wa.y, wa.z, wa.w}, {wb.x, wb.y, wb.z, wb.w}};
#pragma unroll
        for (int p = 0; p < 2; ++p) {
          const float4 g = s_row[(r0 + it * 4) * G + (G == 1 ? 0 : 2 * p + (lj >> 2))];
          const uint64_t mn2 = f2_pack(g.x, g.x), y2 = f2_pack(g.y, g.y), yl2 = f2_pack(g.z, g.z), ns2 = f2_pack(g.w, g.w);
          uint32_t cw[2];
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            uint32_t mq[4];
            code_pair(unpack2<DT>(w[p][2 * i]), mn2, y2, yl2, ns2, mq[0], mq[1]);
            code_pair(unpack2<DT>(w[p][2 * i + 1]), mn2, y2, yl2, ns2, mq[2], mq[3]);
            cw[i] = BITS == 8 ? pack4_u8(mq) : pack4_u4(mq);
          }
          if (BITS == 8)
            *reinterpret_cast<uint2*>(out_r + it * 4 * kD + 64 * p) = make_uint2(cw[0], cw[1]);
          else
            *reinterpret_cast<uint32_t*>(out_r + it * 4 * (kD / 2) + 32 * p) = cw[0] | (cw[1] << 16);
        }
      }
      if (odd) redo_values<DT, BITS>(tile, s_row, td.codes, warp);
    };

    auto keys = [&](auto bits_tag, auto rot_tag) {
      constexpr int BITS = decltype(bits_tag)::value;
      constexpr bool ROT = decltype(rot_tag)::value;
      constexpr float levels = (float)((1 << BITS) - 1);
      constexpr int kGroupTokens = BITS == 8 ? kRows : 32;  // one group per chunk, or groups of 32 tokens
      constexpr int G = kRows / kGroupTokens;
      const uint32_t row_stride = (uint32_t)(H * kD) * BITS / 8;  // bytes of a token row of the layer's codes
      // A lane owns channels 4 p .. 4 p + 3 and their rotation partners 64 + 4 p ..; a half-warp every other token of the warp's.
      const int p = lane & 15, half = lane >> 4;
      const int t0 = warp * kRowsPerWarp + half;
      constexpr int kTok = kRowsPerWarp / 2;
      const uint8_t* const row0 = tile + t0 * (kD * 2) + p * 8;
      auto words = [&](int i, int side) { return *reinterpret_cast<const uint2*>(row0 + i * (2 * kD * 2) + side * kD); };  // side 1: the partners
      // ---- extremes of this thread's values; a half-warp keeps the minima (0) or the maxima (1) of both halves' tokens
      float4 ext[2];
      // With the rotation: token i's eight values, the low half x_lo c + x_hi s and the high half x_hi c - x_lo s.  (Scalar
      // operations: packed ones cost more in register moves than they save.)
      float rc[4], rs[4];
      if (ROT) {
        const float4 ra = *reinterpret_cast<const float4*>(&s_rot[td.rot][4 * p]), rb = *reinterpret_cast<const float4*>(&s_rot[td.rot][4 * p + 2]);
        rc[0] = ra.x, rc[1] = ra.z, rc[2] = rb.x, rc[3] = rb.z, rs[0] = ra.y, rs[1] = ra.w, rs[2] = rb.y, rs[3] = rb.w;
      }
      auto rotated = [&](int i, float (&v)[8]) {
        const uint2 wl = words(i, 0), wh = words(i, 1);
        float lo[4], hi[4];
        f2_unpack(unpack2<DT>(wl.x), lo[0], lo[1]), f2_unpack(unpack2<DT>(wl.y), lo[2], lo[3]);
        f2_unpack(unpack2<DT>(wh.x), hi[0], hi[1]), f2_unpack(unpack2<DT>(wh.y), hi[2], hi[3]);
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          v[c] = fmaf(lo[c], rc[c], __fmul_rn(hi[c], rs[c]));
          v[4 + c] = fmaf(hi[c], rc[c], __fmul_rn(lo[c], -rs[c]));
        }
      };
      if constexpr (ROT) {
        float mn[8], mx[8];
#pragma unroll
        for (int i = 0; i < kTok; i += 2) {
          float v[2][8];
          rotated(i, v[0]);
          rotated(i + 1, v[1]);
#pragma unroll
          for (int c = 0; c < 8; ++c) {
            mn[c] = i == 0 ? min_nan(v[0][c], v[1][c]) : min_nan(mn[c], v[0][c], v[1][c]);
            mx[c] = i == 0 ? max_nan(v[0][c], v[1][c]) : max_nan(mx[c], v[0][c], v[1][c]);
          }
        }
#pragma unroll
        for (int c = 0; c < 8; ++c) {
          const float other = __shfl_xor_sync(0xffffffffu, half ? mn[c] : mx[c], 16);
          mn[c] = half ? max_nan(mx[c], other) : min_nan(mn[c], other);
        }
        ext[0] = make_float4(mn[0], mn[1], mn[2], mn[3]), ext[1] = make_float4(mn[4], mn[5], mn[6], mn[7]);
      } else {
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          uint2 lo = words(0, side), hi = lo;
#pragma unroll
          for (int i = 1; i < kTok; ++i) {
            const uint2 w = words(i, side);
            lo.x = min2_16<DT>(lo.x, w.x), lo.y = min2_16<DT>(lo.y, w.y);
            hi.x = max2_16<DT>(hi.x, w.x), hi.y = max2_16<DT>(hi.y, w.y);
          }
          uint2 give = half ? lo : hi;
          give.x = __shfl_xor_sync(0xffffffffu, give.x, 16), give.y = __shfl_xor_sync(0xffffffffu, give.y, 16);
          const uint2 e = half ? make_uint2(max2_16<DT>(hi.x, give.x), max2_16<DT>(hi.y, give.y))
                               : make_uint2(min2_16<DT>(lo.x, give.x), min2_16<DT>(lo.y, give.y));
          f2_unpack(unpack2<DT>(e.x), ext[side].x, ext[side].y);
          f2_unpack(unpack2<DT>(e.y), ext[side].z, ext[side].w);
        }
      }
#pragma unroll
      for (int side = 0; side < 2; ++side) *reinterpret_cast<float4*>(&s_ext[ext_at(warp, half, side * (kD / 2) + 4 * p)]) = ext[side];
      group_sync(group);
      // ---- (scale, min) and reciprocal of every group and channel from the extremes of the group's warps
#pragma unroll
      for (int n0 = 0; n0 < (G == 1 ? 2 * kD : G * kD); n0 += kWarps * 32) {
        const int n = n0 + tid;
        const int ch = G == 1 ? n >> 1 : n & (kD - 1);  // one group: two neighbouring lanes share a channel
        const int sub = G == 1 ? n & 1 : n / kD;        // (groups: the group)
        float a, b, s;
#pragma unroll
        for (int i = 0; i < kWarps / (G == 1 ? 2 : G); ++i) {
          const int w = G == 1 ? sub + 2 * i : kWarps / G * sub + i;
          const float lo = s_ext[ext_at(w, 0, ch)], hi = s_ext[ext_at(w, 1, ch)];
          a = i == 0 ? lo : min_nan(a, lo), b = i == 0 ? hi : max_nan(b, hi);
        }
        if (G == 1) a = min_nan(a, __shfl_xor_sync(0xffffffffu, a, 1)), b = max_nan(b, __shfl_xor_sync(0xffffffffu, b, 1));
        const int g = G == 1 ? 0 : sub;
        const bool numbers = fabsf(a) < INFINITY;
        if (a != a) {
          const float2 e = number_extremes<DT, ROT, kGroupTokens, kD * 2>(tile + g * kGroupTokens * (kD * 2) + 2 * ch, &s_rot[ROT ? td.rot : 0][ch & (kD / 2 - 1)], ch < kD / 2 ? kD : -kD);
          a = e.x, b = e.y;
        }
        group_params(a, b, levels, meta16, s);
        if (G > 1 || sub == 0) {
          s_par[0][g * kD + ch] = a, s_par[1][g * kD + ch] = numbers ? reciprocal(s) : 0.f, s_par[2][g * kD + ch] = -s;
          store_meta(td.meta, (uint32_t)(g * H * kD + ch), s, a, meta16);
        }
      }
      group_sync(group);
      // ---- codes
      const int gp = (G == 1 ? 0 : warp / (kWarps / G)) * kD + 4 * p;
      uint8_t* o = td.codes + (uint32_t)t0 * row_stride + (uint32_t)(4 * p * BITS) / 8;
      uint64_t mn2[2][2], y2[2][2], yl2[2][2], ns2[2][2];  // per side: min, reciprocal, its rest, -scale of the four channels
      float y_min = 1.f;
#pragma unroll
      for (int side = 0; side < 2; ++side) {
        const float4 a = *reinterpret_cast<const float4*>(&s_par[0][gp + side * (kD / 2)]), b = *reinterpret_cast<const float4*>(&s_par[1][gp + side * (kD / 2)]),
                     c = *reinterpret_cast<const float4*>(&s_par[2][gp + side * (kD / 2)]);
        const uint64_t one2 = f2_pack(1.f, 1.f);
        mn2[side][0] = f2_pack(a.x, a.y), mn2[side][1] = f2_pack(a.z, a.w);
        y2[side][0] = f2_pack(b.x, b.y), y2[side][1] = f2_pack(b.z, b.w);
        ns2[side][0] = f2_pack(c.x, c.y), ns2[side][1] = f2_pack(c.z, c.w);
#pragma unroll
        for (int q = 0; q < 2; ++q) yl2[side][q] = f2_mul(y2[side][q], f2_fma(y2[side][q], ns2[side][q], one2));
        y_min = fminf(y_min, fminf(fminf(b.x, b.y), fminf(b.z, b.w)));
      }
      const bool odd = __any_sync(0xffffffffu, !(y_min > 0.f));
#pragma unroll 4
      for (int i = 0; i < kTok; ++i, o += 2 * row_stride) {
        uint64_t v[2][2];
        if (ROT) {
          float x[8];
          rotated(i, x);
          v[0][0] = f2_pack(x[0], x[1]), v[0][1] = f2_pack(x[2], x[3]), v[1][0] = f2_pack(x[4], x[5]), v[1][1] = f2_pack(x[6], x[7]);
        } else {
          const uint2 wl = words(i, 0), wh = words(i, 1);
          v[0][0] = unpack2<DT>(wl.x), v[0][1] = unpack2<DT>(wl.y), v[1][0] = unpack2<DT>(wh.x), v[1][1] = unpack2<DT>(wh.y);
        }
#pragma unroll
        for (int side = 0; side < 2; ++side) {
          uint32_t mq[4];
          code_pair(v[side][0], mn2[side][0], y2[side][0], yl2[side][0], ns2[side][0], mq[0], mq[1]);
          code_pair(v[side][1], mn2[side][1], y2[side][1], yl2[side][1], ns2[side][1], mq[2], mq[3]);
          if (BITS == 8) *reinterpret_cast<uint32_t*>(o + side * (kD / 2)) = pack4_u8(mq);
          else *reinterpret_cast<uint16_t*>(o + side * (kD / 4)) = (uint16_t)pack4_u4(mq);
        }
      }
      if (odd) redo_keys<DT, BITS, ROT>(tile, s_par, s_rot[ROT ? td.rot : 0], td.codes, row_stride, warp);
    };

    using std::integral_constant;
    if (td.kv) {
      if (td.bits == 8) values(integral_constant<int, 8>{});
      else values(integral_constant<int, 4>{});
    } else if (td.bits == 8) {
      if (td.rot >= 0) keys(integral_constant<int, 8>{}, integral_constant<bool, true>{});
      else keys(integral_constant<int, 8>{}, integral_constant<bool, false>{});
    } else {
      if (td.rot >= 0) keys(integral_constant<int, 4>{}, integral_constant<bool, true>{});
      else keys(integral_constant<int, 4>{}, integral_constant<bool, false>{});
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&s_empty[stage]);
    stage += kGroups;
    if (stage >= kStages) stage -= kStages;
    mine = (mine + 1) & 3;
  }
}

constexpr size_t kSmemBytes = kStages * kTileBytes;
constexpr int kSmallInline = (int)(kDescBlobSmall / sizeof(QuantJob));
static_assert(sizeof(InlineJobs<kQuantInline>) <= kDescBlobBytes, "argument size");

template <int DT, typename Jobs>
cudaError_t configure_one() {
  return cudaFuncSetAttribute(quantize_batch_kernel<DT, Jobs>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemBytes);
}
template <int DT>
cudaError_t configure_type() {
  cudaError_t e = configure_one<DT, InlineJobs<kSmallInline>>();
  if (e == cudaSuccess) e = configure_one<DT, InlineJobs<kQuantInline>>();
  if (e == cudaSuccess) e = configure_one<DT, const QuantJob*>();
  return e;
}

template <typename Jobs>
cudaError_t launch_with(const Jobs& jobs, const QuantBatch& b, const ModelDims& m, const double* inv_freq, uint32_t* status, int n_sm, bool pdl, bool stalled, cudaStream_t st) {
  // one CTA per SM
  const dim3 grid((unsigned)(b.n_tiles < (uint32_t)n_sm ? b.n_tiles : (uint32_t)n_sm)), block(kThreads);
  if (m.dtype == KVB_DT_BF16)
    return launch_pdl(pdl, quantize_batch_kernel<KVB_DT_BF16, Jobs>, grid, block, kSmemBytes, st, jobs, m, b.n_jobs, b.n_tiles, b.per_job, inv_freq, status, stalled);
  return launch_pdl(pdl, quantize_batch_kernel<KVB_DT_F16, Jobs>, grid, block, kSmemBytes, st, jobs, m, b.n_jobs, b.n_tiles, b.per_job, inv_freq, status, stalled);
}

template <int N>
cudaError_t launch_inline(const QuantJob* host_jobs, const QuantBatch& b, const ModelDims& m, const double* inv_freq, uint32_t* status, int n_sm, bool pdl, bool stalled, cudaStream_t st) {
  InlineJobs<N> jobs;
  memcpy(jobs.d, host_jobs, sizeof(QuantJob) * (size_t)b.n_jobs);
  return launch_with(jobs, b, m, inv_freq, status, n_sm, pdl, stalled, st);
}

}  // namespace

cudaError_t quantize_configure() {
  const cudaError_t e = configure_type<KVB_DT_BF16>();
  return e == cudaSuccess ? configure_type<KVB_DT_F16>() : e;
}

cudaError_t launch_quantize_inline(const QuantJob* host_jobs, const QuantBatch& b, const ModelDims& m, const double* inv_freq, uint32_t* status, int n_sm, bool pdl, bool stalled,
                                   cudaStream_t st) {
  if (b.n_jobs <= (uint32_t)kSmallInline) return launch_inline<kSmallInline>(host_jobs, b, m, inv_freq, status, n_sm, pdl, stalled, st);
  if (b.n_jobs <= (uint32_t)kQuantInline) return launch_inline<kQuantInline>(host_jobs, b, m, inv_freq, status, n_sm, pdl, stalled, st);
  return cudaErrorInvalidValue;
}

cudaError_t launch_quantize_table(const QuantJob* table, const QuantBatch& b, const ModelDims& m, const double* inv_freq, uint32_t* status, int n_sm, bool pdl, bool stalled,
                                  cudaStream_t st) {
  return launch_with(table, b, m, inv_freq, status, n_sm, pdl, stalled, st);
}

}  // namespace kvb
