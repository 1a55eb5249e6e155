// Cosine deviation (Algorithm 2, step 2): for every position t,
//     delta_t = 1 - mean over layers, KV heads (and K/V) of cos(stored row, fresh row).
//
// Pure streaming: every 256-byte (token, head) row of the stitched buffer and of the fresh
// tensor is read once with 16-byte loads, a half-warp per row, 8 elements per lane.  Each
// row pair yields ||a-b||^2, ||a||^2 and ||b||^2 (float32, warp-shuffle reduced), and
//     1 - cos = (||a-b||^2 - (||a|| - ||b||)^2) / (2 ||a|| ||b||),
//     ||a|| - ||b|| = (||a||^2 - ||b||^2) / (||a|| + ||b||),
// which has no cancellation for nearly equal rows (1 - dot/(|a||b|) in float32 does).
// The per-row terms are summed over layers, heads and K/V in 2^-40 fixed point with integer
// atomics, so the sum is exact and independent of the order CTAs run in.
//
// Bound by HBM reads.  One kernel per combination of sides, so that a side that is not wanted costs
// neither registers nor arithmetic and its place is taken by a second row.  One side: the next pass's
// four loads are in flight while a pass is worked on: 4224 positions, keys only, 36 layers of 2 heads
// (156 MB) 44.9 -> 25.3 us = 6.1 TB/s.  Both sides (40 registers, so the compiler issues a pass's loads
// where they are used): the same positions, 311 MB, call with selection 70.1 -> 63.6 us.
#include <cuda_bf16.h>
#include <cuda_fp16.h>

#include <type_traits>

#include "deviation_math.cuh"
#include "f32x2.cuh"
#include "kvb_internal.h"
#include "pdl.cuh"
#include "table_arg.cuh"

namespace kvb {
namespace {

constexpr int kThreads = 256;
// Positions of a tile: 64, and for both sides at most 128 (token, head) rows of either.  With 64 positions of 16 heads a CTA
// is so long that a last wave of a few of them weighs: both sides of 2048 positions, 36 layers, call with selection, 4 / 8 / 16
// heads 75.8 / 121 / 229 us, in tiles of 128 rows 58.5 / 97.7 / 177; 8192 positions 202 / 375 / 711 and 186 / 344 / 662.
__host__ __device__ constexpr int tile_tokens(int H, int which) { return which != 3 || H <= 2 ? 64 : 128 / H; }

// grid (tiles over all requests, L).  A tile is tile_tokens consecutive positions of one request.
template <int DT, int WHICH, typename Tab>
__global__ void __launch_bounds__(kThreads)
    deviation_kernel(const __grid_constant__ Tab table, int n_req, ModelDims m, unsigned long long* __restrict__ acc) {
  pdl_wait();  // the table, the buffer and the cleared sums may come from the kernels before this one
  const ReqDesc* const reqs = reinterpret_cast<const ReqDesc*>(table.base());
  // request of this tile: last r with tile_offset <= tile
  const int tile = blockIdx.x;
  int lo = 0, hi = n_req - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (reqs[mid].tile_offset <= tile) lo = mid; else hi = mid - 1;
  }
  const ReqDesc rq = reqs[lo];
  const int l = blockIdx.y;
  const int H = m.Hkv;
  const int t_begin = (tile - rq.tile_offset) * tile_tokens(H, WHICH);
  const int t_end = min(rq.T, t_begin + tile_tokens(H, WHICH));
  const int u_begin = t_begin * H, u_end = t_end * H;  // (token, head) rows of 256 bytes
  const size_t plane = (size_t)rq.T * H * 256;           // bytes of one [T][H][d] plane, d = 128
  const uint8_t* stK = rq.kv_buf + (size_t)(2 * l) * plane;
  const uint8_t* frK = rq.fresh + (size_t)(2 * l) * plane;

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int s = lane >> 4, ln = lane & 15;
  const int n_hw = (kThreads / 32) * 2;
  const bool pair_same_token = (H % 2) == 0;  // rows u, u+1 (u even) belong to one token

  // Lanes 0-7 of a half-warp end up with the sums of one row pair, lanes 8-15 with those of another: the keys and the values
  // of one row when both are wanted, two rows of the one side otherwise (a side that is not wanted costs nothing).
  const bool both = WHICH == 3;
  const uint8_t* const st = WHICH == 2 ? stK + plane : stK;
  const uint8_t* const fr = WHICH == 2 ? frK + plane : frK;
  const int step = both ? n_hw : 2 * n_hw;
  // the next pass's loads before this one's are used
  uint4 w[2][4];
  auto load = [&](int u0, uint4 (&x)[4]) {
    const int ua = u0 + s, ub = both ? ua : ua + n_hw;
    const size_t oa = (size_t)ua * 256 + (size_t)ln * 16, ob = both ? plane + oa : (size_t)ub * 256 + (size_t)ln * 16;
    const uint4 zero = make_uint4(0, 0, 0, 0);
    x[0] = x[1] = x[2] = x[3] = zero;
    if (ua < u_end) x[0] = __ldcs(reinterpret_cast<const uint4*>(st + oa)), x[1] = __ldcs(reinterpret_cast<const uint4*>(fr + oa));
    if (ub < u_end) x[2] = __ldcs(reinterpret_cast<const uint4*>(st + ob)), x[3] = __ldcs(reinterpret_cast<const uint4*>(fr + ob));
  };
  auto work = [&](int u0, const uint4 (&x)[4]) {
    const int ua = u0 + s, ub = both ? ua : ua + n_hw;
    float a[3], b[3];
    row_sums<DT>(x[0], x[1], a[0], a[1], a[2]);
    row_sums<DT>(x[2], x[3], b[0], b[1], b[2]);
    long long fx = pair_terms_fixed(a, b, ln, ua < u_end, ub < u_end);
    if (both) fx += __shfl_xor_sync(0xffffffffu, fx, 8);                // K + V of row u
    if (pair_same_token) fx += __shfl_xor_sync(0xffffffffu, fx, 16);    // both heads of the token
    const int u = (ln & 8) ? ub : ua;
    const bool writes = (both ? ln == 0 : (ln & 7) == 0) && (!pair_same_token || s == 0);
    if (writes && u < u_end) atomicAdd(&acc[rq.tok_offset + u / H], (unsigned long long)fx);
  };
  int u0 = u_begin + warp * 2;
  load(u0, w[0]);  // (rows beyond the tile are not read)
  for (; u0 < u_end; u0 += 2 * step) {
    load(u0 + step, w[1]);
    work(u0, w[0]);
    load(u0 + 2 * step, w[0]);
    work(u0 + step, w[1]);
  }
}

}  // namespace

int deviation_tile_tokens(int Hkv, int which) { return tile_tokens(Hkv, which); }

cudaError_t launch_deviation(const Table& table, int n_req, int total_tiles, const ModelDims& m, int which,
                             unsigned long long* acc, bool pdl, cudaStream_t st) {
  const dim3 grid((unsigned)total_tiles, (unsigned)m.L), block(kThreads);
  return with_table(table, [&](const auto& tab) {
    using Tab = std::decay_t<decltype(tab)>;
    auto launch = [&](auto kernel) { return launch_pdl(pdl, kernel, grid, block, 0, st, tab, n_req, m, acc); };
    if (m.dtype == KVB_DT_BF16)
      return which == 1 ? launch(deviation_kernel<KVB_DT_BF16, 1, Tab>) : which == 2 ? launch(deviation_kernel<KVB_DT_BF16, 2, Tab>) : launch(deviation_kernel<KVB_DT_BF16, 3, Tab>);
    return which == 1 ? launch(deviation_kernel<KVB_DT_F16, 1, Tab>) : which == 2 ? launch(deviation_kernel<KVB_DT_F16, 2, Tab>) : launch(deviation_kernel<KVB_DT_F16, 3, Tab>);
  });
}

}  // namespace kvb
