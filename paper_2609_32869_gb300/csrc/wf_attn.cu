// Decode-time multi-head attention of a few query rows per sequence against a
// per-sequence key/value cache laid out [slot][head][position][64] (bf16).
//
// attention_kernel serves the three attentions of the step (cross_walk_kernel,
// below, the third one for many sequences):
//  - mode 0, causal: the target's self-attention over its cache, query row j
//    of a block starting at position L sees positions [0, L+j] (verify block,
//    prompt, plain greedy step; Sec. 3.1 "one causal target pass");
//  - mode 1, block: the drafter's joint softmax over its history memory at
//    positions [0, L) and the 9 block positions [L, L+9), bidirectional inside
//    the block, with RoPE on queries and keys (Sec. 3.2, App. A.2);
//  - mode 2, cross: all encoder frames (cross-attention, Sec. 3.2).
//
// A CTA takes one (sequence, head, group of <= 16 query rows, block of 256
// keys).  Keys and values arrive by TMA, a block of 32 KB at once from the
// acoustic memory and 64 rows at a time, as many as hold a visible key, from a
// text cache (the caches are
// 3-D tensors (64, position, slot * heads), 128-byte swizzled in shared
// memory; rows past the cache are zero-filled by the copy, value rows past
// the visible keys are zeroed after it); each of the eight
// warps multiplies the 16 query rows against its 32 keys on the tensor cores
// (mma.sync m16n8k16, bf16 in, fp32 accumulate), keeps the row maxima and
// sums in fp32 and forms P V the same way.  Warps combine in order, and the
// blocks of a (sequence, head, group) are combined by the last CTA in block
// order.  Blocks and warps are aligned to absolute key positions and a key a
// query cannot see contributes an exact zero, so a query's result does not
// depend on how many other rows run with it.
#include <cmath>
#include <map>
#include <mutex>
#include <tuple>

#include "wf_device.cuh"
#include "wf_internal.h"

namespace wf {

constexpr int kKB = kAttnKeysPerCTA;  // 256 keys per CTA
constexpr int kQG = kAttnQGroup;      // 16 query rows per CTA
constexpr int kWarps = 8;             // each takes kKW consecutive keys of the block
constexpr int kThreadsA = 32 * kWarps;
constexpr int kKW = kKB / kWarps;     // 32 keys per warp
constexpr int kNT = kKW / 8;          // 8-key score tiles per warp
constexpr int kKS = kKW / 16;         // 16-key steps per warp
constexpr int kDPT = kQG * 64 / kThreadsA;  // output dims per thread in the combine
constexpr int kPartStride = 2 + 64;   // m, l, o[64]
// Scores are kept in base-2 units (times log2 e): every softmax weight, and
// every weight of the merges of partial results, is one exp2 (of the warps'
// weights those below 2^-126 are taken as 0).
constexpr int kSmemK = kKB * 128;     // bytes
constexpr int kSmemQ = kQG * 128;
// K, V, Q, then the warps' (m, l); the warps' O partials reuse the K tile.
// The K and V tiles start 1024-aligned (the copies swizzle by address).
constexpr int kSmemAttn = 1024 + 2 * kSmemK + kSmemQ + kWarps * kQG * 2 * 4 + 16;
static_assert(kWarps * kQG * 64 * 4 <= kSmemK, "O partials must fit in the key tile");
static_assert(kQG * 8 <= kThreadsA && kDPT * kThreadsA == kQG * 64, "thread mapping");
// A launch with fewer CTAs than SMs asks for enough shared memory that no two
// of its CTAs share an SM (it runs beside the neighbouring kernels' CTAs
// under programmatic dependent launch); a larger one packs three per SM.
constexpr int kSmemAttnSpread = 116 * 1024;

// kDPT consecutive output dims (scaled by inv) as bf16
__device__ __forceinline__ void store_row(bf16 *orow, const float (&v)[kDPT], float inv) {
  uint32_t w[kDPT / 2];
#pragma unroll
  for (int e = 0; e < kDPT / 2; ++e) w[e] = pack_bf16(v[2 * e] * inv, v[2 * e + 1] * inv);
  if constexpr (kDPT == 8) {
    *reinterpret_cast<uint4 *>(orow) = make_uint4(w[0], w[1], w[2], w[3]);
  } else {
    static_assert(kDPT == 4, "combine width");
    *reinterpret_cast<uint2 *>(orow) = make_uint2(w[0], w[1]);
  }
}
// Combine a query row's partials (m, l, o[64] per block) in block order into
// output dims d0..d0+3: blocks in groups of 8 with every load of a group in
// flight; a block past n_blocks adds exact zeros.
__device__ __forceinline__ void combine_blocks(const float *pg, int n_blocks, int d0, bf16 *orow) {
  float MM = -INFINITY;
  for (int u0 = 0; u0 < n_blocks; u0 += 8) {
    float mc[8];
#pragma unroll
    for (int u = 0; u < 8; ++u)
      mc[u] = u0 + u < n_blocks ? __ldcg(pg + static_cast<size_t>(u0 + u) * kQG * kPartStride) : -INFINITY;
#pragma unroll
    for (int u = 0; u < 8; ++u) MM = fmaxf(MM, mc[u]);
  }
  float LL = 0.f, oo[kDPT];
#pragma unroll
  for (int e = 0; e < kDPT; ++e) oo[e] = 0.f;
  for (int u0 = 0; u0 < n_blocks; u0 += 8) {
    float mc[8], lc[8], ov[8][kDPT];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      mc[u] = -INFINITY;
      lc[u] = 0.f;
#pragma unroll
      for (int e = 0; e < kDPT; ++e) ov[u][e] = 0.f;
      if (u0 + u < n_blocks) {
        const float *pe = pg + static_cast<size_t>(u0 + u) * kQG * kPartStride;
        mc[u] = __ldcg(pe);
        lc[u] = __ldcg(pe + 1);
#pragma unroll
        for (int e = 0; e < kDPT; ++e) ov[u][e] = __ldcg(pe + 2 + d0 + e);
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const float wt = (mc[u] == -INFINITY) ? 0.f : exp2f(mc[u] - MM);
      LL = __fmaf_rn(lc[u], wt, LL);
#pragma unroll
      for (int e = 0; e < kDPT; ++e) oo[e] = __fmaf_rn(ov[u][e], wt, oo[e]);
    }
  }
  store_row(orow, oo, 1.0f / LL);
}

__global__ void __launch_bounds__(kThreadsA, 3) attention_kernel(const __grid_constant__ CUtensorMap tmK,
                                                              const __grid_constant__ CUtensorMap tmV,
                                                              const AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_u32 = smem_u32(smem_raw);
  uint8_t *smem = smem_raw + (((raw_u32 + 1023u) & ~1023u) - raw_u32);
  uint8_t *sK = smem;
  uint8_t *sV = smem + kSmemK;
  uint8_t *sQ = smem + 2 * kSmemK;
  float *sm = reinterpret_cast<float *>(smem + 2 * kSmemK + kSmemQ);  // [kWarps][16]
  float *sl = sm + kWarps * kQG;                                     // [kWarps][16]
  // [kWarps][16][64]: the warps' O, in the key tile once every warp is done
  // with it (in the value tile for a looping CTA, whose next keys are by
  // then streaming into the key tile)
  float *so = reinterpret_cast<float *>(p.loop ? sV : sK);
  __shared__ int s_last;
  __shared__ uint64_t s_bar[2];  // [0] keys, [1] values

  const int blk = blockIdx.x;
  const int h = blockIdx.y % p.n_heads;
  const int qg = blockIdx.y / p.n_heads;
  const int i = blockIdx.z;
  const int tid = threadIdx.x, warp = warp_index(), lane = tid & 31;

  // Before griddepcontrol.wait only data the previous kernel cannot be
  // writing is touched: the active list and cache lengths change only between
  // steps (the kernels that precede an attention launch in a call all wait
  // for their predecessors before allowing it to start), the acoustic memory
  // only at prefill, and self-attention cache rows below L only in earlier
  // steps.  Those rows stream in while the producer of this layer's queries
  // (and of rows L..L+rps-1) finishes.

  const int slot = __ldcg(p.seq_slot + i);
  const int base = (p.mode == 2 || !p.pos_base) ? 0 : __ldcg(p.pos_base + slot);
  const int q0 = qg * kQG;
  const int nq = min(kQG, p.rps - q0);
  int n_keys;
  if (p.mode == 2)
    n_keys = p.ctx;
  else if (p.mode == 1)
    n_keys = base + p.rps;
  else
    n_keys = base + q0 + nq;  // keys visible to the last query of the group
  if (n_keys > p.ctx || (p.mode != 2 && base + p.rps > p.ctx)) {
    // the block would pass the cache: record it and leave the output untouched
    if (blk == 0 && tid == 0) set_error(p.err, WF_DEV_ERR_CAPACITY);
    return;
  }
  const int n_blocks = (n_keys + kKB - 1) / kKB;
  // In a cluster launch every CTA of a multi-block group takes part in the
  // merge; a block past the keys computes over masked keys only and yields
  // the exact empty partial (m = -inf, l = 0, o = 0).
  if (!p.loop && blk >= n_blocks && !(p.cluster && n_blocks > 1)) return;

  const int d_model = p.n_heads * 64;
  // the key blocks this CTA computes: its own, or (loop) all of its group's
  // in order, each leaving its partial as a CTA of its own would
  const int b_first = p.loop ? 0 : blk, b_end = p.loop ? n_blocks : blk + 1;
  const int group_id = (i * p.n_heads + h) * p.qgroups + qg;

  // ---- keys and values: TMA copies, a whole block at once of the acoustic
  // memory and 64 rows, as many as hold a visible key, of a text cache (whose
  // blocks are rarely full: 256-row copies read a short cache twice over).  A block holding rows that this
  // step's projection writes (positions from `fresh` on) loads after the
  // wait; a block of settled rows streams in while the producer of the
  // queries finishes.  A looping CTA requests each later block once the
  // previous one is done with the tiles.
  const int fresh = p.mode == 2 ? n_keys : base;
  const int cache_row = slot * p.n_heads + h;
  const int box = p.box;
  const uint32_t box_bytes = static_cast<uint32_t>(min(box, p.ctx)) * 128u;  // the maps' box
  auto issue_tile = [&](const CUtensorMap *tm, uint8_t *tile, uint64_t *bar, int b) {  // by the first warp
    const int n = (min(kKB, n_keys - b * kKB) + box - 1) / box;
    if (elect_one()) {
      if (b > b_first) fence_proxy_async();  // generic writes to the tile come before the copy
      mbar_arrive_expect_tx(bar, n * box_bytes);
      for (int c = 0; c < n; ++c) tma_load_3d(tile + c * box * 128, tm, 0, b * kKB + c * box, cache_row, bar);
    }
    __syncwarp();
  };
  auto issue_k = [&](int b) { issue_tile(&tmK, sK, &s_bar[0], b); };
  auto issue_v = [&](int b) { issue_tile(&tmV, sV, &s_bar[1], b); };
  auto issue = [&](int b) {
    issue_k(b);
    issue_v(b);
  };
  const bool first_keys = b_first * kKB < n_keys;
  const bool first_fresh = first_keys && fresh < n_keys && b_first * kKB + kKB > fresh;
  if (tid == 0) {
    mbar_init(&s_bar[0], 1);
    mbar_init(&s_bar[1], 1);
    fence_barrier_init();
    tma_prefetch_desc(&tmK);
    tma_prefetch_desc(&tmV);
  }
  __syncwarp();
  if (warp == 0 && first_keys && !first_fresh) issue(b_first);
  pdl_wait();
  pdl_launch_dependents();
  if (warp == 0 && first_fresh) issue(b_first);
  const long long spin = p.spin > 0 ? p.spin : kSpinLimitCycles;
  // ---- queries, pre-scaled by 1/8 = 1/sqrt(64) (exact in binary), RoPE in fp32
  if (tid < kQG * 8) {
    const int r = tid >> 3, ch = tid & 7;
    uint4 raw = make_uint4(0, 0, 0, 0), par = make_uint4(0, 0, 0, 0);
    if (r < nq) {
      const bf16 *qrow = p.q + static_cast<size_t>(i * p.rps + q0 + r) * d_model + h * 64;
      raw = *reinterpret_cast<const uint4 *>(qrow + ch * 8);
      if (p.rope_tab) par = *reinterpret_cast<const uint4 *>(qrow + ((ch * 8) ^ 32));
    }
    const bf16 *qv = reinterpret_cast<const bf16 *>(&raw);
    const bf16 *qp = reinterpret_cast<const bf16 *>(&par);
    float f[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      float v = bf2f(qv[e]);
      if (p.rope_tab && r < nq) {
        const int dd = ch * 8 + e;
        const float2 cs = __ldg(p.rope_tab + (base + q0 + r) * 32 + (dd & 31));
        const float other = bf2f(qp[e]);
        v = dd < 32 ? v * cs.x - other * cs.y : v * cs.x + other * cs.y;
      }
      f[e] = v * 0.125f;
    }
    uint4 o;
    o.x = pack_bf16(f[0], f[1]);
    o.y = pack_bf16(f[2], f[3]);
    o.z = pack_bf16(f[4], f[5]);
    o.w = pack_bf16(f[6], f[7]);
    *reinterpret_cast<uint4 *>(sQ + swz(r, ch)) = o;
  }
  // thread -> (row qi, dims d0..d0+kDPT-1) in the combines
  const int qi = tid / (64 / kDPT), d0 = (tid % (64 / kDPT)) * kDPT;
  for (int bi = b_first; bi < b_end; ++bi) {
  const int key0 = bi * kKB;
  const bool any_keys = key0 < n_keys;
  const uint32_t ph = static_cast<uint32_t>((bi - b_first) & 1);  // the tiles' copy of this block
  // (this block's keys were requested under the previous block's P V)
  if (bi > b_first && warp == 0) issue_v(bi);
  // keys first; the values keep streaming while the scores are formed.  After
  // a timeout thread 0 waits (bounded) for both copies before going on, so
  // no copy lands in a CTA that has exited.
  __syncthreads();
  if (any_keys && !mbar_wait(&s_bar[0], ph, p.err, spin) && tid == 0) {
    mbar_drain(&s_bar[0], ph);
    mbar_drain(&s_bar[1], ph);
  }

  // ---- per warp: 16 query rows x kKW keys on the tensor cores
  const int g = lane >> 2, c4 = lane & 3;
  const int kw = warp * kKW;  // first key of this warp within the block
  const bool any = key0 + kw < n_keys;  // (else the exact empty partial: m = -inf, l = 0)
  float mrow[2] = {-INFINITY, -INFINITY}, lrow[2] = {0.f, 0.f};
  float s[kNT][4], o[8][4];
  if (any) {
  // ---- RoPE on the warp's keys (drafter): dims i and i+32 rotate by pos * base^(-2i/64)
  if (p.rope_tab) {
#pragma unroll
    for (int t = 0; t < kKW * 4 / 32; ++t) {
      const int kr = kw + t * 8 + (lane >> 2), c = lane & 3;  // chunk c (dims 8c..8c+7) pairs with chunk c+4
      const int pos = key0 + kr;
      if (pos >= n_keys) continue;
      uint4 *lo = reinterpret_cast<uint4 *>(sK + swz(kr, c));
      uint4 *hi = reinterpret_cast<uint4 *>(sK + swz(kr, c + 4));
      uint4 a = *lo, b = *hi;
      bf16 *av = reinterpret_cast<bf16 *>(&a);
      bf16 *bv = reinterpret_cast<bf16 *>(&b);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float2 cs = __ldg(p.rope_tab + pos * 32 + c * 8 + e);
        const float x1 = bf2f(av[e]), x2 = bf2f(bv[e]);
        av[e] = __float2bfloat16(x1 * cs.x - x2 * cs.y);
        bv[e] = __float2bfloat16(x2 * cs.x + x1 * cs.y);
      }
      *lo = a;
      *hi = b;
    }
    __syncwarp();
  }
  const uint32_t q_u32 = smem_u32(sQ), k_u32 = smem_u32(sK);
#pragma unroll
  for (int nt = 0; nt < kNT; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {
    uint32_t a0, a1, a2, a3;
    {
      const int mi = lane >> 3;
      ldsm_x4(q_u32 + swz((mi & 1) * 8 + (lane & 7), 2 * ks + (mi >> 1)), a0, a1, a2, a3);
    }
#pragma unroll
    for (int np = 0; np < kKS; ++np) {
      uint32_t b0, b1, b2, b3;
      const int mi = lane >> 3;
      ldsm_x4(k_u32 + swz(kw + np * 16 + (mi >> 1) * 8 + (lane & 7), 2 * ks + (mi & 1)), b0, b1, b2,
              b3);
      mma_bf16(s[2 * np], a0, a1, a2, a3, b0, b1);
      mma_bf16(s[2 * np + 1], a0, a1, a2, a3, b2, b3);
    }
  }
  // row maxima and exponentials (rows g and g+8 of the group; rows past nq are
  // read by nobody), masked only where some row misses one of the keys
#pragma unroll
  for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) s[nt][e] *= kLog2e;  // base-2 logits
  if (key0 + kw + kKW > (p.mode == 0 ? min(n_keys, base + q0 + 1) : n_keys)) {
#pragma unroll
    for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const int pos = key0 + kw + nt * 8 + c4 * 2 + (e & 1);
        if (pos >= n_keys || (p.mode == 0 && pos > base + q0 + g + (e >> 1) * 8)) s[nt][e] = -INFINITY;
      }
  }
#pragma unroll
  for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
    for (int e = 0; e < 4; ++e) mrow[e >> 1] = fmaxf(mrow[e >> 1], s[nt][e]);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    mrow[r] = fmaxf(mrow[r], __shfl_xor_sync(0xffffffffu, mrow[r], 1));
    mrow[r] = fmaxf(mrow[r], __shfl_xor_sync(0xffffffffu, mrow[r], 2));
  }
  // (a row that sees none of these keys has no maximum: weights 0, not NaN)
  const float mfin[2] = {mrow[0] == -INFINITY ? 0.f : mrow[0], mrow[1] == -INFINITY ? 0.f : mrow[1]};
#pragma unroll
  for (int nt = 0; nt < kNT; ++nt) {
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float v = exp2f_fast(s[nt][e] - mfin[e >> 1]);
      s[nt][e] = v;
      lrow[e >> 1] += v;
    }
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    lrow[r] += __shfl_xor_sync(0xffffffffu, lrow[r], 1);
    lrow[r] += __shfl_xor_sync(0xffffffffu, lrow[r], 2);
  }
  }
  if (any_keys && !mbar_wait(&s_bar[1], ph, p.err, spin) && tid == 0) mbar_drain(&s_bar[1], ph);
  if (p.loop) {
    // every warp is done with the keys: a looping CTA requests the next block's
    __syncthreads();
    if (bi + 1 < b_end && warp == 0) issue_k(bi + 1);
  }
  if (any) {
  // the warp's values; rows past the visible keys (stale cache rows, rows past
  // the copies) become zeros, so P V adds exact zeros there
  const int z0 = n_keys - key0 - kw;
  if (z0 < kKW) {
    for (int idx = lane; idx < (kKW - z0) * 8; idx += 32)
      *reinterpret_cast<uint4 *>(sV + swz(kw + z0 + (idx >> 3), idx & 7)) = make_uint4(0u, 0u, 0u, 0u);
    __syncwarp();
  }
  const uint32_t v_u32 = smem_u32(sV);
  // O = P V (P rounded to bf16 as the A operand)
#pragma unroll
  for (int nd = 0; nd < 8; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;
#pragma unroll
  for (int kk = 0; kk < kKS; ++kk) {
    const uint32_t a0 = pack_bf16(s[2 * kk][0], s[2 * kk][1]);
    const uint32_t a1 = pack_bf16(s[2 * kk][2], s[2 * kk][3]);
    const uint32_t a2 = pack_bf16(s[2 * kk + 1][0], s[2 * kk + 1][1]);
    const uint32_t a3 = pack_bf16(s[2 * kk + 1][2], s[2 * kk + 1][3]);
#pragma unroll
    for (int dp = 0; dp < 4; ++dp) {
      uint32_t b0, b1, b2, b3;
      const int mi = lane >> 3;
      ldsm_x4_t(v_u32 + swz(kw + kk * 16 + (mi & 1) * 8 + (lane & 7), 2 * dp + (mi >> 1)), b0, b1,
                b2, b3);
      mma_bf16(o[2 * dp], a0, a1, a2, a3, b0, b1);
      mma_bf16(o[2 * dp + 1], a0, a1, a2, a3, b2, b3);
    }
  }
  }
  __syncthreads();  // every warp is done with the tile that now holds O
  // stage this warp's (m, l, O) for the in-order combine
  if (c4 == 0) {
    sm[warp * kQG + g] = mrow[0];
    sm[warp * kQG + g + 8] = mrow[1];
    sl[warp * kQG + g] = lrow[0];
    sl[warp * kQG + g + 8] = lrow[1];
  }
  // O rows of 64 floats, 8-float column groups XOR-swizzled by the row's
  // low two bits: a half-warp's fragment stores fall in distinct banks
  if (any) {
#pragma unroll
  for (int nd = 0; nd < 8; ++nd) {
    const int col = (nd ^ (g & 3)) * 8 + c4 * 2;
    *reinterpret_cast<float2 *>(so + (warp * kQG + g) * 64 + col) = make_float2(o[nd][0], o[nd][1]);
    *reinterpret_cast<float2 *>(so + (warp * kQG + g + 8) * 64 + col) = make_float2(o[nd][2], o[nd][3]);
  }
  }
  __syncthreads();

  // ---- combine the warps in order (a warp that saw no key of the row adds
  // exact zeros; one without any key left its O unwritten)
  static_assert(kDPT == 4, "one float4 of O per warp and thread");
  float M = -INFINITY, L = 0.f, acc[kDPT] = {0.f, 0.f, 0.f, 0.f};
  if (qi < nq) {
    float mw[kWarps];
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      mw[w] = sm[w * kQG + qi];
      M = fmaxf(M, mw[w]);
    }
    const float mf = M == -INFINITY ? 0.f : M;
#pragma unroll
    for (int w = 0; w < kWarps; ++w) {
      const float wt = exp2f_fast(mw[w] - mf);
      L = __fmaf_rn(sl[w * kQG + qi], wt, L);
      // dims d0..d0+3 stay contiguous under the swizzle (it flips bits 3 and 4)
      const float4 o4 = *reinterpret_cast<const float4 *>(so + (w * kQG + qi) * 64 + (d0 ^ ((qi & 3) << 3)));
      const bool none = mw[w] == -INFINITY;
      acc[0] = none ? acc[0] : __fmaf_rn(o4.x, wt, acc[0]);
      acc[1] = none ? acc[1] : __fmaf_rn(o4.y, wt, acc[1]);
      acc[2] = none ? acc[2] : __fmaf_rn(o4.z, wt, acc[2]);
      acc[3] = none ? acc[3] : __fmaf_rn(o4.w, wt, acc[3]);
    }
  }

  if (n_blocks == 1) {
    if (qi < nq) {
      const float inv = 1.0f / L;
      bf16 *orow = p.out + static_cast<size_t>(i * p.rps + q0 + qi) * d_model + h * 64 + d0;
      store_row(orow, acc, inv);
    }
    return;
  }

  if (p.cluster) {
    // ---- several key blocks in one cluster: each CTA leaves its partial in
    // its shared memory ([16][68]: m, l, -, -, o[64]); CTA 0 combines them in
    // block order over DSMEM with the same arithmetic as the global path.
    float *pb = reinterpret_cast<float *>(sV);
    if (d0 == 0) {
      pb[qi * 68] = M;
      pb[qi * 68 + 1] = L;
    }
#pragma unroll
    for (int e = 0; e < kDPT; ++e) pb[qi * 68 + 4 + d0 + e] = acc[e];
    cluster_sync();
    float MM = -INFINITY, LL = 0.f, oo[kDPT];
    if (blk == 0) {
      // every peer's (m, l, o) load in flight at once (at most 8 blocks), then
      // merged in block order; an absent block adds exact zeros
      const uint32_t pb_u32 = smem_u32(pb);
      float mc[8], lc[8];
      float4 o4[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        mc[u] = -INFINITY;
        lc[u] = 0.f;
        o4[u] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (u < p.n_chunks) {
          mc[u] = dsmem_ld_f32(dsmem_map(pb_u32 + 4u * (qi * 68), u));
          lc[u] = dsmem_ld_f32(dsmem_map(pb_u32 + 4u * (qi * 68 + 1), u));
          o4[u] = dsmem_ld_f32x4(dsmem_map(pb_u32 + 4u * (qi * 68 + 4 + d0), u));
        }
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) MM = fmaxf(MM, mc[u]);
#pragma unroll
      for (int e = 0; e < kDPT; ++e) oo[e] = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const float ov[4] = {o4[u].x, o4[u].y, o4[u].z, o4[u].w};
        const float wt = (mc[u] == -INFINITY) ? 0.f : exp2f(mc[u] - MM);
        LL = __fmaf_rn(lc[u], wt, LL);
#pragma unroll
        for (int e = 0; e < kDPT; ++e) oo[e] = __fmaf_rn(ov[e], wt, oo[e]);
      }
    }
    cluster_arrive();  // CTA 0 has read every partial; peers may exit
    cluster_wait();
    if (blk == 0 && qi < nq) {
      bf16 *orow = p.out + static_cast<size_t>(i * p.rps + q0 + qi) * d_model + h * 64 + d0;
      store_row(orow, oo, 1.0f / LL);
    }
    return;
  }

  // ---- several key blocks: partials to global, the last CTA combines in order
  float *part = p.part + (static_cast<size_t>(group_id) * p.n_chunks + bi) * kQG * kPartStride;
  if (qi < nq) {
    float *pe = part + qi * kPartStride;
    if (d0 == 0) {
      pe[0] = M;
      pe[1] = L;
    }
#pragma unroll
    for (int e = 0; e < kDPT; ++e) pe[2 + d0 + e] = acc[e];
  }
  // one fence per CTA: after the barrier thread 0 releases the whole CTA's
  // partial at GPU scope and counts it; the last CTA's thread 0 fences again
  // (acquire) before the barrier that releases its threads into the combine.
  // A looping CTA goes on to its next block once every thread is done with
  // this one (its partials are then visible to all its threads).
  __syncthreads();
  if (p.loop) continue;
  if (tid == 0) {
    __threadfence();
    const int last = atomicAdd(&p.counters[group_id], 1) == n_blocks - 1;
    if (last) __threadfence();
    s_last = last;
  }
  __syncthreads();
  if (!s_last) return;
  }  // key blocks
  // A block the query cannot see carries m = -inf, l = 0, o = 0 and gets
  // weight 0, so it adds exact zeros; the loads of all blocks are independent.
  if (qi < nq) {
    const float *pg = p.part + static_cast<size_t>(group_id) * p.n_chunks * kQG * kPartStride;
    combine_blocks(pg + qi * kPartStride, n_blocks, d0,
                   p.out + static_cast<size_t>(i * p.rps + q0 + qi) * d_model + h * 64 + d0);
  }
  if (tid == 0) p.counters[group_id] = 0;
}

// ------------------------------------------------ walking cross-attention --
// Cross-attention of many sequences: two persistent CTAs per SM, each walking
// an even share of all (sequence, head, query group, key block) units in group
// order.  One warp runs ahead copying keys and values into a ring of three
// 32 KB tiles, so that two tiles are on their way while eight warps compute on
// the third; another writes the next group's queries (scaled) into one of two
// tiles.  The keys' tile is free once the scores are formed; the values' tile
// takes the warps' O for the combine and is free after it.
//
// Arithmetic as above, operation for operation (a slice of 32 keys per warp,
// warps combined in order, blocks combined in order): partials go to global
// memory; the CTA that walks all blocks of a group combines them itself, a
// group cut by the end of a share is combined by whichever CTA finishes last.
//
// A bounded wait that runs out: the compute warps go through the same units and
// barriers, read at a unit's first barrier whether one of them gave up, and
// leave together; they count the blocks that they owe to groups shared with
// other CTAs, so that the counters return to zero.  The copying warp leaves
// last, after its copies in flight have landed.  What the CTA had not finished
// stays unwritten.
//
// Bound by HBM for many sequences.  Captured calls over 1500 frames, 20 heads,
// nine rows, keys and values from HBM, against one CTA per group: 32 sequences
// 55 -> 53 us, 96 sequences 137 -> 129 (5.9 TB/s), 16 sequences 31.3 -> 32.8
// with the counters' clearing that only a call pays for.  Inside a step, where
// its copies start under the query projection: 96 sequences 8.58 -> 8.30 ms, 32
// sampling (4 layers) 1037 -> 995 us, 16 (4 layers) 686 -> 675 us.  Rings of
// nine 64-row copies with the warps' O beside them measured 136 us at 96
// sequences; a warp per block without any merge of warps 145 us.
constexpr int kWkThreads = kThreadsA + 64;  // eight compute warps, the copying warp, the query warp
constexpr int kWkTiles = 3;
struct WalkUnit {
  int row0, h, nq, blk;  // first query row, head, queries, key block
  int group, mine, qbuf, end;  // mine: blocks of the group this CTA walked when this is its last one (else 0)
                               // end: the share's last unit
};
constexpr int kSmemWalk = 1024 + kWkTiles * kSmemK + 2 * kSmemQ + kWarps * kQG * 2 * 4 +
                          kWkTiles * static_cast<int>(sizeof(WalkUnit)) + (2 * kWkTiles + 4) * 8 + 16;

__device__ __forceinline__ void compute_barrier() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
// The CTA's end: the copying warp waits there for all others.
__device__ __forceinline__ void walk_end_barrier() { asm volatile("bar.sync 2, 320;" ::: "memory"); }
__device__ __forceinline__ void walk_end_arrive() { asm volatile("bar.arrive 2, 320;" ::: "memory"); }

__global__ void __launch_bounds__(kWkThreads, 2)
    cross_walk_kernel(const __grid_constant__ CUtensorMap tmK, const __grid_constant__ CUtensorMap tmV,
                          const AttnParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw_u32 = smem_u32(smem_raw);
  uint8_t *smem = smem_raw + (((raw_u32 + 1023u) & ~1023u) - raw_u32);
  uint8_t *sQ = smem + kWkTiles * kSmemK;                      // two tiles
  float *sm = reinterpret_cast<float *>(sQ + 2 * kSmemQ);      // [kWarps][16]
  float *sl = sm + kWarps * kQG;                               // [kWarps][16]
  WalkUnit *info = reinterpret_cast<WalkUnit *>(sl + kWarps * kQG);  // of the unit whose keys a tile holds
  uint64_t *full = reinterpret_cast<uint64_t *>(info + kWkTiles);
  uint64_t *empty = full + kWkTiles;
  uint64_t *qfree = empty + kWkTiles;  // [2] every compute warp has read the queries
  int *s_last = reinterpret_cast<int *>(qfree + 2);
  volatile int &s_gave_up = s_last[1];   // a compute warp's wait ran out
  volatile int &s_counted = s_last[2];   // groups shared with other CTAs whose blocks here were counted
  volatile int &s_arrivals = s_last[3];  // of the query warp on the tiles

  const int warp = warp_index(), lane = threadIdx.x & 31, tid = threadIdx.x;
  const int groups = p.n_seq * p.n_heads * p.qgroups;
  const long long total = static_cast<long long>(groups) * p.n_chunks;
  const int u_begin = static_cast<int>(total * blockIdx.x / gridDim.x);
  const int u_end = static_cast<int>(total * (blockIdx.x + 1) / gridDim.x);
  const int d_model = p.n_heads * 64;
  const long long spin = p.spin > 0 ? p.spin : kSpinLimitCycles;

  if (tid == 0) {
    for (int t = 0; t < kWkTiles; ++t) {
      mbar_init(&full[t], 2);  // its copies; the unit and its queries in place
      mbar_init(&empty[t], kWarps);
    }
    mbar_init(&qfree[0], kWarps);
    mbar_init(&qfree[1], kWarps);
    s_gave_up = 0;
    s_counted = 0;
    for (int t = 0; t < kWkTiles; ++t) info[t] = WalkUnit{};
    fence_barrier_init();
    fence_proxy_async();
  }
  __syncthreads();

  if (warp >= kWarps) {
    // ---------------- the two warps that run ahead over the units: the first
    // copies keys and values, the second writes what the compute warps need to
    // know of a unit and its queries.  Both step through the same tiles.
    const bool copies = warp == kWarps;
    int tile = 0;
    uint32_t eph = 1;  // (a fresh barrier passes the wait for the phase before its first)
    bool ok = true;
    auto next_tile = [&]() {
      if (++tile == kWkTiles) {
        tile = 0;
        eph ^= 1;
      }
    };
    int g = u_begin / p.n_chunks, blk = u_begin - g * p.n_chunks, u = u_begin;
    if (copies) {
      if (lane == 0) {
        tma_prefetch_desc(&tmK);
        tma_prefetch_desc(&tmV);
      }
      // the acoustic memory is settled: nothing here waits for the previous kernel
      const uint32_t bytes = static_cast<uint32_t>(min(kKB, p.ctx)) * 128u;
      int slot_next = u < u_end ? __ldcg(p.seq_slot + g / p.qgroups / p.n_heads) : 0;  // read a group ahead
      int n_copies = 0;
      for (; u < u_end && ok; ++g, blk = 0) {
        const int ih = g / p.qgroups, i = ih / p.n_heads, cache_row = slot_next * p.n_heads + ih - i * p.n_heads;
        bool ahead = false;
        for (; blk < p.n_chunks && u < u_end && ok; ++blk, ++u) {
          for (int kv = 0; kv < 2; ++kv) {
            if (!(ok = warp_mbar_wait(&empty[tile], eph, p.err, spin))) break;
            ++n_copies;
            if (elect_one()) {
              mbar_arrive_expect_tx(&full[tile], bytes);
              tma_load_3d(smem + tile * kSmemK, kv ? &tmV : &tmK, 0, blk * kKB, cache_row, &full[tile]);
            }
            __syncwarp();
            next_tile();
          }
          if (!ahead && g + 1 < groups) slot_next = __ldcg(p.seq_slot + (g + 1) / p.qgroups / p.n_heads);
          ahead = true;
        }
      }
      pdl_wait();
      walk_end_barrier();
      if (s_gave_up && lane == 0) {
        // No copy lands in a CTA that has exited.  Nobody else looks at the
        // tiles any more, so this warp makes up for arrivals of the query warp
        // that did not come.
        for (int c = max(0, n_copies - kWkTiles); c < n_copies; ++c) {
          if (c >= s_arrivals) mbar_arrive_cta(&full[c % kWkTiles]);
          mbar_drain(&full[c % kWkTiles], static_cast<uint32_t>(c / kWkTiles) & 1u);
        }
        // The blocks of shared groups (the first and the last of the share)
        // that the compute warps did not come to count.
        int counted = s_counted;
        for (int q = u_begin / p.n_chunks; q * p.n_chunks < u_end; ++q) {
          const int mine = min(u_end, (q + 1) * p.n_chunks) - max(u_begin, q * p.n_chunks);
          if (mine == p.n_chunks || --counted >= 0) continue;
          if (atomicAdd(&p.counters[q], mine) + mine == p.n_chunks) p.counters[q] = 0;
        }
      }
      return;
    }
    pdl_wait();  // the queries are the previous kernel's
    pdl_launch_dependents();
    uint4 raw[kQG * 8 / 32];  // the next group's queries, in flight
    auto load_queries = [&](int group) {
      const int ih = group / p.qgroups, i = ih / p.n_heads, h = ih - i * p.n_heads, q0 = (group - ih * p.qgroups) * kQG;
      const int nq = group < groups ? min(kQG, p.rps - q0) : 0;
#pragma unroll
      for (int t = 0; t < kQG * 8 / 32; ++t) {
        const int r = t * 4 + (lane >> 3), ch = lane & 7;
        raw[t] = make_uint4(0, 0, 0, 0);
        if (r < nq)
          raw[t] = *reinterpret_cast<const uint4 *>(p.q + static_cast<size_t>(i * p.rps + q0 + r) * d_model + h * 64 + ch * 8);
      }
    };
    load_queries(g);
    WalkUnit w = {};
    int n_groups = 0, n_arrivals = 0;
    for (; u < u_end && ok; ++g, blk = 0) {
      const int ih = g / p.qgroups, i = ih / p.n_heads, q0 = (g - ih * p.qgroups) * kQG;
      w.h = ih - i * p.n_heads;
      w.nq = min(kQG, p.rps - q0);
      w.row0 = i * p.rps + q0;
      w.group = g;
      for (int walked = 0; blk < p.n_chunks && u < u_end; ++blk, ++u) {
        if (!(ok = warp_mbar_wait(&empty[tile], eph, p.err, spin))) break;
        if (walked++ == 0) {
          // ---- queries, pre-scaled by 1/8 = 1/sqrt(64) (exact in binary)
          w.qbuf = n_groups & 1;
          if (!(ok = warp_mbar_wait(&qfree[w.qbuf], ((static_cast<uint32_t>(n_groups) >> 1) & 1u) ^ 1u, p.err, spin)))
            break;
          ++n_groups;
          uint8_t *q = sQ + w.qbuf * kSmemQ;
#pragma unroll
          for (int t = 0; t < kQG * 8 / 32; ++t) {
            const bf16 *qv = reinterpret_cast<const bf16 *>(&raw[t]);
            uint32_t o4[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) o4[e] = pack_bf16(bf2f(qv[2 * e]) * 0.125f, bf2f(qv[2 * e + 1]) * 0.125f);
            *reinterpret_cast<uint4 *>(q + swz(t * 4 + (lane >> 3), lane & 7)) = make_uint4(o4[0], o4[1], o4[2], o4[3]);
          }
        }
        w.blk = blk;
        w.end = u + 1 == u_end;
        w.mine = (blk == p.n_chunks - 1 || u + 1 == u_end) ? walked : 0;
        if (lane == 0) info[tile] = w;
        __syncwarp();
        if (lane == 0) mbar_arrive_cta(&full[tile]);  // unit and queries are in place
        ++n_arrivals;
        next_tile();
        // the values' tile has nothing to add
        if (!(ok = warp_mbar_wait(&empty[tile], eph, p.err, spin))) break;
        if (lane == 0) mbar_arrive_cta(&full[tile]);
        ++n_arrivals;
        next_tile();
        if (walked == 1) load_queries(g + 1);
      }
    }
    if (lane == 0) s_arrivals = n_arrivals;
    __syncwarp();
    walk_end_arrive();
    return;
  }

  // ---------------- compute warps
  const int qi = tid / (64 / kDPT), d0 = (tid % (64 / kDPT)) * kDPT;
  const int g = lane >> 2, c4 = lane & 3, mi = lane >> 3, kw = warp * kKW;
  int tile = 0;
  uint32_t fph = 0;
  auto step_tile = [&]() {
    if (++tile == kWkTiles) {
      tile = 0;
      fph ^= 1;
    }
  };
  pdl_wait();
  WalkUnit w;
  do {
    bool ok = warp_mbar_wait(&full[tile], fph, p.err, spin);  // (the same in all lanes)
    w = info[tile];
    uint8_t *sK = smem + tile * kSmemK;
    const int key0 = w.blk * kKB;
    const bool any = ok && key0 + kw < p.ctx;  // this warp's slice has a visible key
    float s[kNT][4];
    if (any) {
      const uint32_t q_u32 = smem_u32(sQ + w.qbuf * kSmemQ), k_u32 = smem_u32(sK);
#pragma unroll
      for (int nt = 0; nt < kNT; ++nt) s[nt][0] = s[nt][1] = s[nt][2] = s[nt][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < 4; ++ks) {
        uint32_t a0, a1, a2, a3;
        ldsm_x4(q_u32 + swz((mi & 1) * 8 + (lane & 7), 2 * ks + (mi >> 1)), a0, a1, a2, a3);
#pragma unroll
        for (int np = 0; np < kKS; ++np) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4(k_u32 + swz(kw + np * 16 + (mi >> 1) * 8 + (lane & 7), 2 * ks + (mi & 1)), b0, b1, b2, b3);
          mma_bf16(s[2 * np], a0, a1, a2, a3, b0, b1);
          mma_bf16(s[2 * np + 1], a0, a1, a2, a3, b2, b3);
        }
      }
    }
    __syncwarp();
    if (ok && lane == 0) {
      mbar_arrive_cta(&empty[tile]);
      if (w.mine) mbar_arrive_cta(&qfree[w.qbuf]);
    }
    step_tile();
    uint8_t *sV = smem + tile * kSmemK;
    float mrow[2] = {-INFINITY, -INFINITY}, lrow[2] = {0.f, 0.f};
    float o[8][4];
    if (any) {
      // row maxima and exponentials (rows g and g + 8 of the group; rows past
      // nq are read by nobody); only the last frames' slice has keys to mask
#pragma unroll
      for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) s[nt][e] *= kLog2e;  // base-2 logits
      if (key0 + kw + kKW > p.ctx) {
#pragma unroll
        for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            if (key0 + kw + nt * 8 + c4 * 2 + (e & 1) >= p.ctx) s[nt][e] = -INFINITY;
      }
#pragma unroll
      for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) mrow[e >> 1] = fmaxf(mrow[e >> 1], s[nt][e]);
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        mrow[r] = fmaxf(mrow[r], __shfl_xor_sync(0xffffffffu, mrow[r], 1));
        mrow[r] = fmaxf(mrow[r], __shfl_xor_sync(0xffffffffu, mrow[r], 2));
      }
      // (a row whose scores here are all -inf has no maximum: weights 0, not NaN)
      const float mfin[2] = {mrow[0] == -INFINITY ? 0.f : mrow[0], mrow[1] == -INFINITY ? 0.f : mrow[1]};
#pragma unroll
      for (int nt = 0; nt < kNT; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float v = exp2f_fast(s[nt][e] - mfin[e >> 1]);
          s[nt][e] = v;
          lrow[e >> 1] += v;
        }
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        lrow[r] += __shfl_xor_sync(0xffffffffu, lrow[r], 1);
        lrow[r] += __shfl_xor_sync(0xffffffffu, lrow[r], 2);
      }
    }
    if (ok) ok = warp_mbar_wait(&full[tile], fph, p.err, spin);
    if (any && ok) {
      // rows past the last frame become zeros, so P V adds exact zeros there
      const int z0 = p.ctx - key0 - kw;
      if (z0 < kKW) {
        for (int idx = lane; idx < (kKW - z0) * 8; idx += 32)
          *reinterpret_cast<uint4 *>(sV + swz(kw + z0 + (idx >> 3), idx & 7)) = make_uint4(0u, 0u, 0u, 0u);
        __syncwarp();
      }
      const uint32_t v_u32 = smem_u32(sV);
      // O = P V (P rounded to bf16 as the A operand)
#pragma unroll
      for (int nd = 0; nd < 8; ++nd) o[nd][0] = o[nd][1] = o[nd][2] = o[nd][3] = 0.f;
#pragma unroll
      for (int kk = 0; kk < kKS; ++kk) {
        const uint32_t a0 = pack_bf16(s[2 * kk][0], s[2 * kk][1]);
        const uint32_t a1 = pack_bf16(s[2 * kk][2], s[2 * kk][3]);
        const uint32_t a2 = pack_bf16(s[2 * kk + 1][0], s[2 * kk + 1][1]);
        const uint32_t a3 = pack_bf16(s[2 * kk + 1][2], s[2 * kk + 1][3]);
#pragma unroll
        for (int dp = 0; dp < 4; ++dp) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4_t(v_u32 + swz(kw + kk * 16 + (mi & 1) * 8 + (lane & 7), 2 * dp + (mi >> 1)), b0, b1, b2, b3);
          mma_bf16(o[2 * dp], a0, a1, a2, a3, b0, b1);
          mma_bf16(o[2 * dp + 1], a0, a1, a2, a3, b2, b3);
        }
      }
    }
    if (!ok) s_gave_up = 1;
    compute_barrier();  // every warp is done with the values, and with the last unit's sums
    // (the same for all warps: none sets it for a later unit before the next barrier)
    const int leave = s_gave_up;
    // stage this warp's (m, l, O) for the in-order combine: O over the values,
    // 8-float column groups XOR-swizzled by the row's low two bits
    float *so = reinterpret_cast<float *>(sV);
    if (c4 == 0) {
      sm[warp * kQG + g] = mrow[0];
      sm[warp * kQG + g + 8] = mrow[1];
      sl[warp * kQG + g] = lrow[0];
      sl[warp * kQG + g + 8] = lrow[1];
    }
    if (any) {
#pragma unroll
      for (int nd = 0; nd < 8; ++nd) {
        const int col = (nd ^ (g & 3)) * 8 + c4 * 2;
        *reinterpret_cast<float2 *>(so + (warp * kQG + g) * 64 + col) = make_float2(o[nd][0], o[nd][1]);
        *reinterpret_cast<float2 *>(so + (warp * kQG + g + 8) * 64 + col) = make_float2(o[nd][2], o[nd][3]);
      }
    }
    if (leave) break;
    compute_barrier();

    // ---- combine the warps in order (a warp without a visible key of the row
    // adds exact zeros)
    float M = -INFINITY, L = 0.f, acc[kDPT] = {0.f, 0.f, 0.f, 0.f};
    if (qi < w.nq) {
      float mw[kWarps];
#pragma unroll
      for (int v = 0; v < kWarps; ++v) {
        mw[v] = sm[v * kQG + qi];
        M = fmaxf(M, mw[v]);
      }
      const float mf = M == -INFINITY ? 0.f : M;
#pragma unroll
      for (int v = 0; v < kWarps; ++v) {
        const float wt = exp2f_fast(mw[v] - mf);  // (0 for -inf)
        const float4 o4 = *reinterpret_cast<const float4 *>(so + (v * kQG + qi) * 64 + (d0 ^ ((qi & 3) << 3)));
        L = __fmaf_rn(sl[v * kQG + qi], wt, L);
        const bool none = mw[v] == -INFINITY;  // (a slice without a key left its O unwritten)
        acc[0] = none ? acc[0] : __fmaf_rn(o4.x, wt, acc[0]);
        acc[1] = none ? acc[1] : __fmaf_rn(o4.y, wt, acc[1]);
        acc[2] = none ? acc[2] : __fmaf_rn(o4.z, wt, acc[2]);
        acc[3] = none ? acc[3] : __fmaf_rn(o4.w, wt, acc[3]);
      }
    }
    fence_proxy_async();  // the tile's generic writes and reads come before its next copy
    __syncwarp();
    if (lane == 0) mbar_arrive_cta(&empty[tile]);
    step_tile();

    bf16 *orow = p.out + static_cast<size_t>(w.row0 + qi) * d_model + w.h * 64 + d0;
    float *pg = p.part + static_cast<size_t>(w.group) * p.n_chunks * kQG * kPartStride;
    if (qi < w.nq) {
      float *pe = pg + (static_cast<size_t>(w.blk) * kQG + qi) * kPartStride;
      if (d0 == 0) *reinterpret_cast<float2 *>(pe) = make_float2(M, L);
      *reinterpret_cast<float2 *>(pe + 2 + d0) = make_float2(acc[0], acc[1]);
      *reinterpret_cast<float2 *>(pe + 4 + d0) = make_float2(acc[2], acc[3]);
    }
    if (!w.mine) continue;
    // ---- the CTA's last block of the group: combine, or leave it to the last CTA
    compute_barrier();
    if (w.mine < p.n_chunks) {
      if (tid == 0) {
        __threadfence();
        const int last = atomicAdd(&p.counters[w.group], w.mine) + w.mine == p.n_chunks;
        s_counted = s_counted + 1;
        if (last) {
          __threadfence();
          p.counters[w.group] = 0;
        }
        *s_last = last;
      }
      compute_barrier();
      if (!*s_last) continue;
    }
    if (qi < w.nq) combine_blocks(pg + qi * kPartStride, p.n_chunks, d0, orow);
  } while (!w.end);
  walk_end_arrive();
}

// (cos, sin) of pos * base^(-2i/64) for every position below max_pos, or below
// the last key of the call (n_seq > 0: the longest seq_slot / pos_base plus
// rps).  Double precision runs at 2 operations per cycle and SM, and a sine and
// cosine take ~100: the frequencies come from the host and two positions make
// a CTA, so that the SMs share the rest (10.4 us at 159 positions with the
// powers on the device and 16 positions a CTA).
constexpr int kRopeRows = 2;  // positions per CTA
struct RopeFreq {
  float inv[32];  // base^(-2i/64), rounded from double
};
static RopeFreq rope_freq(float base) {
  RopeFreq f;
  for (int i = 0; i < 32; ++i) f.inv[i] = static_cast<float>(std::pow(static_cast<double>(base), -2.0 * i / 64.0));
  return f;
}
__global__ void __launch_bounds__(32 * kRopeRows)
    rope_table_kernel(float2 *tab, int max_pos, const RopeFreq f, const int32_t *seq_slot, const int32_t *pos_base,
                      int n_seq, int rps) {
  const int pos = blockIdx.x * kRopeRows + threadIdx.x / 32, i = threadIdx.x % 32;
  bool used = n_seq == 0;
  for (int q = i; q < n_seq; q += 32) used = used || pos < pos_base[seq_slot[q]] + rps;
  if (!__any_sync(0xffffffffu, used) || pos >= max_pos) return;
  // the phase pos * inv_freq in FP32 (App. A.2)
  const float ang = __fmul_rn(static_cast<float>(pos), f.inv[i]);
  double sn, cs;
  sincos(static_cast<double>(ang), &sn, &cs);
  tab[pos * 32 + i] = make_float2(static_cast<float>(cs), static_cast<float>(sn));
}

size_t attn_partial_floats(int n_seq, int rps, int n_heads, int ctx) {
  const int qgroups = (rps + kQG - 1) / kQG;
  const int n_blocks = (ctx + kKB - 1) / kKB;
  return static_cast<size_t>(n_seq) * n_heads * qgroups * n_blocks * kQG * kPartStride;
}

int attn_counter_slots(int n_seq, int rps, int n_heads) {
  return n_seq * n_heads * ((rps + kQG - 1) / kQG);
}

// Tensor maps of the caches, encoded once per (cache, ctx, outer, box): 3-D
// (64 dims, ctx positions, outer = slot * heads + head) with a box of `box`
// positions of one (slot, head), 128-byte swizzled; positions past ctx read
// as zeros.
static const CUtensorMap *attn_tmap(const void *cache, int ctx, int outer, int box) {
  static std::mutex mu;
  static std::map<std::tuple<uintptr_t, int, int, int>, CUtensorMap *> maps;
  std::lock_guard<std::mutex> lock(mu);
  const auto key = std::make_tuple(reinterpret_cast<uintptr_t>(cache), ctx, outer, box);
  auto it = maps.find(key);
  if (it != maps.end()) return it->second;
  CUtensorMap *m = new CUtensorMap;
  if (!tmap_bf16_cache(m, cache, static_cast<uint64_t>(ctx), static_cast<uint64_t>(outer),
                       static_cast<uint32_t>(ctx < box ? ctx : box))) {
    delete m;
    return nullptr;
  }
  maps.emplace(key, m);
  return m;
}

cudaError_t attention_init() {
  static cudaError_t status = cudaErrorNotReady;
  static std::once_flag once;
  std::call_once(once, [] {
    status = cudaFuncSetAttribute(attention_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  kSmemAttnSpread);
    if (status == cudaSuccess)
      status = cudaFuncSetAttribute(cross_walk_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemWalk);
    if (status == cudaSuccess) status = prefer_max_shared(reinterpret_cast<const void *>(attention_kernel));
    if (status == cudaSuccess) status = prefer_max_shared(reinterpret_cast<const void *>(cross_walk_kernel));
  });
  return status;
}

// The form of a launch: small launches merge their blocks over DSMEM (no
// global round trip); large ones keep the global partials, where cluster
// placement costs more than it saves.  With at least two (sequence, head,
// query group)s per SM one CTA per group walks its key blocks in order,
// leaving the same partials and merging them itself (a single wave of CTAs, no
// counter), or, over the acoustic memory, where every group has as many
// blocks, persistent CTAs walk even shares of all blocks (cross_walk_kernel,
// with its measurements; it does not rotate, so a call with a RoPE table stays
// with one CTA per group).  All do the same arithmetic in the same order.
//
// One CTA per group, three per SM, stays the better form over the acoustic
// memory in two cases (us, one CTA per group / walking):
//  - its only wave is nearly full (370-456 of 456 places): calls over 1500
//    frames, 20 heads, 22 sequences of nine rows 34.6 / 41.1 (of 16, 70% full,
//    29.5 / 32.5, 3 of them the clearing of counters that only a call pays for);
//    a step, large widths, 4 layers: 22 sequences 708 / 722, 20 691 / 700, but 18
//    679 / 675, 16 664 / 651 and, with a second wave begun, 24 794 / 751;
//  - several query groups per head over keys and values that do not stay in L2:
//    a walking CTA comes back to them for the next group when they are gone.
//    Calls of 15 sequences of 33 rows 53.5 / 65.1, of 16 of 200 rows 228 / 270;
//    prefill of 13 prompts of 33 tokens (100 MB of keys and values a layer) 1,150
//    / 1,167; but calls of 10 of 33 rows (77 MB) 43.9 / 41.2.
constexpr double kLoopWaveFill = 0.81;
constexpr long long kWalkGroupsBytes = 88LL << 20;
struct AttnForm {
  int n_sm, qgroups, n_chunks, cluster, loop, walk;
  bool counters() const { return n_chunks > 1 && !cluster && !loop; }  // the form counts finished blocks
};
static AttnForm attn_form(int n_seq, int rps, int n_heads, int ctx, int mode, bool rope) {
  static const int n_sm = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    return n;
  }();
  AttnForm f;
  f.n_sm = n_sm;
  f.qgroups = (rps + kQG - 1) / kQG;
  f.n_chunks = (ctx + kKB - 1) / kKB;
  const long long groups = static_cast<long long>(n_seq) * n_heads * f.qgroups;
  f.cluster = (f.n_chunks > 1 && f.n_chunks <= 8 && groups * f.n_chunks <= n_sm) ? 1 : 0;
  const bool many = !f.cluster && f.n_chunks > 1 && n_sm > 0 && groups >= 2LL * n_sm;
  const long long places = 3LL * n_sm, kv_bytes = 256LL * n_seq * n_heads * ctx;
  const bool full_wave = groups <= places && groups >= kLoopWaveFill * places;
  const bool rereads = f.qgroups > 1 && kv_bytes > kWalkGroupsBytes;
  f.walk = (many && mode == 2 && !rope && !full_wave && !rereads && groups * f.n_chunks <= 0x3fffffff) ? 1 : 0;
  f.loop = (many && !f.walk) ? 1 : 0;
  return f;
}

cudaError_t launch_attention(const AttnParams &p0, cudaStream_t s, bool pdl) {
  AttnParams p = p0;
  AttnForm f = attn_form(p.n_seq, p.rps, p.n_heads, p.ctx, p.mode, p.rope_tab != nullptr);
  if (f.walk && (reinterpret_cast<uintptr_t>(p.part) & 7)) {  // its partials go out in pairs
    f.walk = 0;
    f.loop = 1;
  }
  p.qgroups = f.qgroups;
  p.n_chunks = f.n_chunks;
  p.cluster = f.cluster;
  p.loop = f.loop;
  const int n_sm = f.n_sm;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(p.loop ? 1 : p.n_chunks, p.n_heads * p.qgroups, p.n_seq);
  cfg.blockDim = dim3(kThreadsA, 1, 1);
  const long long ctas = static_cast<long long>(cfg.gridDim.x) * cfg.gridDim.y * cfg.gridDim.z;
  cfg.dynamicSmemBytes = ctas <= n_sm ? kSmemAttnSpread : kSmemAttn;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (p.cluster) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = p.n_chunks;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = 1;
    ++na;
  }
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  if (p.outer < 1) return cudaErrorInvalidValue;
  if (f.walk) {
    const CUtensorMap *wk = attn_tmap(p.kc, p.ctx, p.outer, kKB), *wv = attn_tmap(p.vc, p.ctx, p.outer, kKB);
    if (!wk || !wv) return cudaErrorInvalidValue;
    cfg.gridDim = dim3(2 * n_sm);
    cfg.blockDim = dim3(kWkThreads);
    cfg.dynamicSmemBytes = kSmemWalk;
    return cudaLaunchKernelEx(&cfg, cross_walk_kernel, *wk, *wv, p);
  }
  p.box = p.mode == 2 ? kKB : 64;
  const CUtensorMap *tk = attn_tmap(p.kc, p.ctx, p.outer, p.box), *tv = attn_tmap(p.vc, p.ctx, p.outer, p.box);
  if (!tk || !tv) return cudaErrorInvalidValue;
  return cudaLaunchKernelEx(&cfg, attention_kernel, *tk, *tv, p);
}

cudaError_t launch_rope_table(float2 *tab, int max_pos, float base, cudaStream_t s) {
  rope_table_kernel<<<(max_pos + kRopeRows - 1) / kRopeRows, 32 * kRopeRows, 0, s>>>(tab, max_pos, rope_freq(base), nullptr,
                                                                                          nullptr, 0, 0);
  return cudaGetLastError();
}

// Positions of a call's RoPE table: those of its cache, and over all frames
// (mode 2, queries at positions 0..RPS-1) its queries' too.
static int rope_rows(int mode, int rope, int RPS, int ctx) { return rope && mode == 2 && RPS > ctx ? RPS : ctx; }
static size_t attn_scratch_bytes(int n_seq, int RPS, int n_heads, int ctx, int rope_rows) {
  const size_t counters = static_cast<size_t>(attn_counter_slots(n_seq, RPS, n_heads)) * 4;
  return attn_partial_floats(n_seq, RPS, n_heads, ctx) * sizeof(float) + ((counters + 255) / 256) * 256 +
         static_cast<size_t>(rope_rows) * 32 * sizeof(float2) + 256;
}

// The kernel-level entry points: scratch holds the partials, the counters of
// finished blocks and the RoPE table of the call's positions.  Counters are
// cleared only for the form that counts; behind a table the attention is a
// dependent launch (the table kernel starts after everything before it).
static wf_status attention_call(const void *d_q, const void *d_kc, const void *d_vc, const int32_t *d_slot,
                                const int32_t *d_base, int32_t n_seq, int32_t RPS, int32_t n_heads, int32_t ctx,
                                int32_t mode, int32_t rope, float rope_base, void *d_out, void *scratch,
                                cudaStream_t s) {
  AttnParams p = {};
  p.q = static_cast<const bf16 *>(d_q);
  p.kc = static_cast<const bf16 *>(d_kc);
  p.vc = static_cast<const bf16 *>(d_vc);
  p.out = static_cast<bf16 *>(d_out);
  p.seq_slot = d_slot;
  p.pos_base = d_base;
  p.n_seq = n_seq;
  p.rps = RPS;
  p.n_heads = n_heads;
  p.ctx = ctx;
  p.mode = mode;
  p.outer = kAttnOuterBound;
  const size_t pf = attn_partial_floats(n_seq, RPS, n_heads, ctx);
  const size_t counters = static_cast<size_t>(attn_counter_slots(n_seq, RPS, n_heads)) * 4;
  p.part = static_cast<float *>(scratch);
  p.counters = reinterpret_cast<int32_t *>(static_cast<char *>(scratch) + pf * sizeof(float));
  if (attn_form(n_seq, RPS, n_heads, ctx, mode, rope != 0).counters() &&
      cudaMemsetAsync(p.counters, 0, counters, s) != cudaSuccess)
    return WF_ERR_CUDA;
  if (rope) {
    float2 *tab = reinterpret_cast<float2 *>(static_cast<char *>(scratch) + pf * sizeof(float) +
                                             ((counters + 255) / 256) * 256);
    const int rows = rope_rows(mode, rope, RPS, ctx);
    rope_table_kernel<<<(rows + kRopeRows - 1) / kRopeRows, 32 * kRopeRows, 0, s>>>(
        tab, rows, rope_freq(rope_base), d_slot, d_base, mode == 2 ? 0 : n_seq, RPS);
    if (cudaGetLastError() != cudaSuccess) return WF_ERR_CUDA;
    p.rope_tab = tab;
  }
  return launch_attention(p, s, rope != 0) == cudaSuccess ? WF_OK : WF_ERR_CUDA;
}

}  // namespace wf

extern "C" size_t wf_attention_scratch_bytes(int32_t n_seq, int32_t RPS, int32_t n_heads,
                                             int32_t ctx) {
  if (n_seq <= 0 || RPS <= 0 || n_heads <= 0 || ctx <= 0) return 0;
  return wf::attn_scratch_bytes(n_seq, RPS, n_heads, ctx, wf::rope_rows(2, 1, RPS, ctx));
}

extern "C" wf_status wf_attention(const void *d_q, const void *d_kc, const void *d_vc,
                                  const int32_t *d_slot, const int32_t *d_base, int32_t n_seq,
                                  int32_t RPS, int32_t n_heads, int32_t ctx, int32_t mode,
                                  int32_t rope, float rope_base, void *d_out, void *d_scratch,
                                  size_t scratch_bytes, void *stream) {
  if (!d_q || !d_kc || !d_vc || !d_slot || !d_out || n_seq <= 0 || RPS <= 0 || n_heads <= 0 ||
      ctx <= 0 || mode < 0 || mode > 2)
    return WF_ERR_INVALID;
  if (mode != 2 && !d_base) return WF_ERR_INVALID;
  if (scratch_bytes < wf::attn_scratch_bytes(n_seq, RPS, n_heads, ctx, wf::rope_rows(mode, rope, RPS, ctx)) || !d_scratch)
    return WF_ERR_CAPACITY;
  if (wf::attention_init() != cudaSuccess) return WF_ERR_CUDA;
  return wf::attention_call(d_q, d_kc, d_vc, d_slot, d_base, n_seq, RPS, n_heads, ctx, mode, rope, rope_base, d_out,
                            d_scratch, static_cast<cudaStream_t>(stream));
}

// ---------------------------------------------------------------------------
// wf_attention_noalloc: the same attention for callers that cannot allocate
// device memory.
//
// Some callers have no way to obtain scratch: code that runs while a CUDA
// graph is being captured in a mode that forbids cudaMalloc, plugins hosted
// by a framework that owns every device allocation, and latency-critical
// loops where an allocation (which can synchronise the device) is not
// acceptable.  For them the partial sums and counters live in one file-scope
// device array of kNoAllocScratchBytes, which every GPU that loads this
// library holds until the process exits.  The first call on a device looks
// the array's device address up (cudaGetSymbolAddress), which can load the
// library's module; make that first call before any stream capture.  All
// calls share the array: calls that can overlap on the GPU (different
// streams, or without ordering between them) race on it and must not be
// issued.  The counters are cleared on every call of a form that counts
// finished blocks; the partial sums need no clearing.
namespace {
constexpr size_t kNoAllocScratchBytes = size_t(8) << 20;  // 8 MiB
static __device__ __align__(256) unsigned char g_noalloc_scratch[kNoAllocScratchBytes];
constexpr int kNoAllocMaxDevices = 64;
std::mutex g_noalloc_mu;
void *g_noalloc_ptr[kNoAllocMaxDevices] = {};
}  // namespace

extern "C" wf_status wf_attention_noalloc(const void *d_q, const void *d_kc, const void *d_vc,
                                          const int32_t *d_slot, const int32_t *d_base,
                                          int32_t n_seq, int32_t RPS, int32_t n_heads,
                                          int32_t ctx, int32_t mode, int32_t rope,
                                          float rope_base, void *d_out, void *stream) {
  if (!d_q || !d_kc || !d_vc || !d_slot || !d_out || n_seq <= 0 || RPS <= 0 || n_heads <= 0 ||
      ctx <= 0 || mode < 0 || mode > 2)
    return WF_ERR_INVALID;
  if (mode != 2 && !d_base) return WF_ERR_INVALID;
  const size_t need = wf::attn_scratch_bytes(n_seq, RPS, n_heads, ctx, wf::rope_rows(mode, rope, RPS, ctx));
  if (need > kNoAllocScratchBytes) return WF_ERR_CAPACITY;
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess) return WF_ERR_CUDA;
  if (dev < 0 || dev >= kNoAllocMaxDevices) return WF_ERR_UNSUPPORTED;
  void *scratch = nullptr;
  {
    std::lock_guard<std::mutex> lock(g_noalloc_mu);
    if (!g_noalloc_ptr[dev]) {
      void *ptr = nullptr;
      if (cudaGetSymbolAddress(&ptr, g_noalloc_scratch) != cudaSuccess || !ptr) return WF_ERR_CUDA;
      g_noalloc_ptr[dev] = ptr;
    }
    scratch = g_noalloc_ptr[dev];
  }
  if (wf::attention_init() != cudaSuccess) return WF_ERR_CUDA;
  return wf::attention_call(d_q, d_kc, d_vc, d_slot, d_base, n_seq, RPS, n_heads, ctx, mode, rope, rope_base, d_out,
                            scratch, static_cast<cudaStream_t>(stream));
}
