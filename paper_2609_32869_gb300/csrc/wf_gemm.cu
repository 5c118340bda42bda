// Skinny-M bf16 GEMM on the sm_103a tensor cores (tcgen05 + TMEM + TMA).
//
// Every projection of the decode step is Y = X W^T with few token rows
// (M = 9 per sequence: the anchor and K = 8 proposals, Sec. 3.1) against a
// large weight matrix, so the weights stream from HBM once and set the time.
// The kernel computes a 128 x BT tile of D = W_tile X_tile^T ("swap-AB"): the
// 128 weight rows fill the MMA's M side, the token tile (a multiple of 16,
// <= 128) its N side.  Weight and token tiles stream into shared memory by
// TMA (128-byte swizzle) through an mbarrier ring; one thread issues
// tcgen05.mma into a TMEM accumulator; eight warps read it back with
// tcgen05.ld for a fused epilogue (bias, GELU, residual add, taps or key/value
// cache scatter; the output head runs in wf_gemm_wide.cu).
//
// K is split into a fixed number of chunks per (N, K) shape so that ~150 CTAs
// stream weights even for a single sequence.  The S split CTAs of a tile form
// a thread-block cluster; after the MMAs each pushes its fp32 partials over
// distributed shared memory to the CTAs that finish the rows, which add them
// in split order, so results are deterministic and independent of M, and no
// partial ever travels through global memory.  Past wide_min_rows() the pushes
// (~16 bytes per cycle and SM) cost more than they save and pairs of SMs run
// the projection instead (wf_gemm_wide.cu).
//
// With programmatic dependent launch the weight tiles of the first pipeline
// stages are requested before griddepcontrol.wait: they do not depend on the
// previous kernel, so their HBM latency overlaps its tail.
#include <cuda.h>
#include <cudaTypedefs.h>
#include <mutex>
#include <map>
#include <tuple>
#include <algorithm>

#include "wf_device.cuh"
#include "wf_gemm_epi.cuh"
#include "wf_internal.h"

namespace wf {

constexpr int kBlockN = 128;   // weight rows per tile (MMA M)
constexpr int kThreads = 256;  // 8 warps: two per TMEM lane quarter
constexpr int kBlockK = 64;    // K per pipeline stage (one 128-byte swizzle atom)
constexpr int kStageA = kBlockN * kBlockK * 2;  // 16 KB
// Shared memory a CTA plans for: two CTAs fit on an SM, so one CTA's
// epilogue overlaps the other's weight stream.
constexpr int kSmemBudget = 110 * 1024;
constexpr int kMaxBT = 128;                // token rows per tile (MMA N)
constexpr size_t kSmemPerSM = 228 * 1024;  // shared memory of one SM
constexpr uint32_t kGroupBytes = 128 * 4 * 4;  // one split's partials of four token rows
// Token rows above which pairs of SMs (wf_gemm_wide.cu) take a projection from
// the cluster split-K.  A pair goes through all of K for its tile, K / 64 steps
// one after the other; a cluster shares K out and pays with pushes that grow
// with the rows.  Many weight tiles let the pairs cover the GPU early.  A launch
// of its own (no programmatic dependence) shows a pair's whole chain, so there
// the line lies higher the longer K is and the fewer CTAs the clusters have in
// all; behind a dependent launch the chain's weights are under way before the
// previous kernel ends, and the line does not move.  Launches of a captured
// graph, us (cluster / pairs), weights from HBM at the large widths, from L2 at
// the tiny ones:
//   3840 x 1280   45 rows  7.5 /  7.4   97 rows  9.7 /  7.6
//   5120 x 1280   45 rows  8.0 /  7.7   97 rows 10.3 /  8.2
//   2560 x 1280   72 rows  6.8 /  7.2   97 rows  7.8 /  7.3
//   384 x 384     90 rows  5.3 /  5.4   97 rows  5.8 /  5.3  (1152, 1536 x 384 alike)
//   1280 x 1280   97 rows  7.7 /  7.8  108 rows  7.7 /  7.8  126 rows  8.6 / 7.8
//   1280 x 5120   97 rows 12.4 / 13.5  108 rows 13.2 / 13.5  126 rows 14.5 / 13.5
//   1280 x 6400  108 rows 10.7 / 15.4  180 rows 12.7 / 15.4  252 rows 15.5 / 15.5
//   384 x 1920    97 rows  7.3 /  9.1  180 rows  7.4 /  9.1  252 rows  8.6 / 9.1
//   384 x 1536    97 rows  6.9 /  8.1  180 rows  6.5 /  8.2  252 rows  7.8 / 8.2
//   768 x 3072   180 rows  9.2 / 10.4  216 rows 11.0 / 10.6  (clusters of 16)
//   1024 x 4096   97 rows 11.3 / 11.9  126 rows 13.3 / 11.8  (128 CTAs)
// A step of 12 sequences (108 rows, large widths, 4 layers) takes 656 us with a
// lone launch's lines, 638 with 96; one of 20 (180 rows, tiny) 451 and 444.
constexpr int kWideMinM = 96;
constexpr int kWideMinMFewRows = 40;  // many weight tiles
constexpr int kWideFewRowsN = 3840;
// lone launches: few weight tiles and a long K; a longer one whose clusters
// leave SMs idle (two token tiles; clusters of 16 push most per row)
constexpr int kWideMinMLongK = 112;
constexpr int kWideLongKN = 1280;
constexpr int kWideLongK = 1280;
constexpr int kWideMinMRoom = 256;
constexpr int kWideMinMRoom16 = 192;
constexpr int kWideRoomK = 1536;
constexpr int kWideRoomCtas = 104;

static int wide_min_rows(int N, int K, int splits, bool pdl) {
  if (N >= kWideFewRowsN) return kWideMinMFewRows;
  if (pdl) return kWideMinM;
  if (K >= kWideRoomK && (N + kBlockN - 1) / kBlockN * splits <= kWideRoomCtas)
    return splits < 16 ? kWideMinMRoom : kWideMinMRoom16;
  return N <= kWideLongKN && K >= kWideLongK ? kWideMinMLongK : kWideMinM;
}

// Epilogue of 16 consecutive token columns t0..t0+15 for output feature n.
// acc[] holds the 16 accumulated values; every global load of the chunk (the
// residual) is issued before its stores so the latencies overlap.
template <int EPI>
__device__ __forceinline__ void epi_chunk(const GemmParams &p, int t0, int n, float bn,
                                          const float (&acc)[16], const int2 *tok) {
  if (n >= p.N) return;
  if constexpr (EPI == EPI_F32) {
#pragma unroll
    for (int jj = 0; jj < 16; ++jj)
      if (t0 + jj < p.M) p.out_f32[static_cast<size_t>(t0 + jj) * p.ld_out + n] = acc[jj] + bn;
  } else if constexpr (EPI == EPI_BF16) {
#pragma unroll
    for (int jj = 0; jj < 16; ++jj)
      if (t0 + jj < p.M)
        p.out_bf16[static_cast<size_t>(t0 + jj) * p.ld_out + n] = __float2bfloat16(acc[jj] + bn);
  } else if constexpr (EPI == EPI_GELU) {
#pragma unroll
    for (int jj = 0; jj < 16; ++jj)
      if (t0 + jj < p.M)
        p.out_bf16[static_cast<size_t>(t0 + jj) * p.ld_out + n] =
            __float2bfloat16(gelu_erf(acc[jj] + bn));
  } else if constexpr (EPI == EPI_RESID) {
    float r[16];
#pragma unroll
    for (int jj = 0; jj < 16; ++jj)
      r[jj] = (t0 + jj < p.M) ? p.resid[static_cast<size_t>(t0 + jj) * p.ld_resid + n] : 0.f;
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) {
      if (t0 + jj >= p.M) continue;
      const float nr = r[jj] + (acc[jj] + bn);
      p.resid[static_cast<size_t>(t0 + jj) * p.ld_resid + n] = nr;
      if (p.tap0) p.tap0[static_cast<size_t>(t0 + jj) * p.ld_tap + n] = __float2bfloat16(nr);
      if (p.tap1) p.tap1[static_cast<size_t>(t0 + jj) * p.ld_tap + n] = __float2bfloat16(nr);
    }
  } else if constexpr (EPI == EPI_KV) {
    if (n < p.q_cols) {
#pragma unroll
      for (int jj = 0; jj < 16; ++jj)
        if (t0 + jj < p.M)
          p.out_bf16[static_cast<size_t>(t0 + jj) * p.ld_out + n] = __float2bfloat16(acc[jj] + bn);
      return;
    }
    const int c = n - p.q_cols;
    const int which = c / p.d_model;
    const int hd = c - which * p.d_model;
    const int h = hd >> 6, dd = hd & 63;
    bf16 *dst = which == 0 ? p.kc : p.vc;
#pragma unroll
    for (int jj = 0; jj < 16; ++jj) {
      if (t0 + jj >= p.M) continue;
      const int2 sp = tok[jj];  // (slot, position) of this token row
      if (sp.y >= p.ctx) {
        set_error(p.err, WF_DEV_ERR_CAPACITY);
        continue;
      }
      dst[((static_cast<size_t>(sp.x) * p.n_heads + h) * p.ctx + sp.y) * 64 + dd] =
          __float2bfloat16(acc[jj] + bn);
    }
  }
}

template <int EPI>
__global__ void __launch_bounds__(kThreads) gemm_tc_kernel(const __grid_constant__ CUtensorMap tmW,
                                                      const __grid_constant__ CUtensorMap tmX,
                                                      const GemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t *smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  const int BT = p.BT, stages = p.stages, kps = p.kps;
  const uint32_t stageB = static_cast<uint32_t>(BT) * kBlockK * 2;
  uint8_t *sA = smem;
  uint8_t *sB = smem + static_cast<size_t>(stages) * kStageA;
  uint64_t *full = reinterpret_cast<uint64_t *>(smem + p.pipe_bytes);
  uint64_t *empty = full + stages;
  uint64_t *done = empty + stages;
  uint64_t *inbox_bar = done + 1;  // split-K: the partials of this CTA's token groups arrived
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 2);
  // per-token (slot, position) for EPI_KV
  int2 *tok = reinterpret_cast<int2 *>(smem + p.pipe_bytes + (2 * stages + 2) * 8 + 32);
  // split-K: where the partials of each group of four token rows go (the
  // cluster addresses of the slot and of its owner's inbox barrier)
  uint2 *dest = reinterpret_cast<uint2 *>(tok + BT);
  // a bounded wait of this CTA gave up (in the 32 bytes reserved after the
  // barriers, beside the TMEM address; the kernel has no static shared memory)
  volatile int &s_timed_out = *reinterpret_cast<int *>(tmem_slot + 1);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int tt = blockIdx.x, ntile = blockIdx.y, split = blockIdx.z;
  const int n0 = ntile * kBlockN, t0 = tt * BT, kit0 = split * kps;

  if (threadIdx.x == 0) {
    s_timed_out = 0;
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmX);
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    mbar_init(inbox_bar, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  __syncwarp();
  if (warp == 2) tmem_alloc(tmem_slot, p.tmem_cols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_launch_dependents();

  // Weight tiles of the first stages do not depend on the previous kernel:
  // request them before the dependency wait.
  // Copies and MMAs are issued by one elected lane of code that the whole warp
  // runs: under a lane comparison each of them took ~430 cycles.
  const int npre = kps < stages ? kps : stages;
  const uint32_t tx = kStageA + stageB;
  if (warp == 0) {
    for (int i = 0; i < npre; ++i) {
      if (elect_one()) {
        mbar_arrive_expect_tx(&full[i], tx);
        tma_load_2d(sA + static_cast<size_t>(i) * kStageA, &tmW, (kit0 + i) * kBlockK, n0, &full[i]);
      }
    }
  }
  int issued = npre;  // k-steps whose tiles the producer (warp 0) has requested
  if (warp == 0) {
    // ---------------- TMA producer
    pdl_wait();  // token rows come from the previous kernel
    for (int i = 0; i < npre; ++i)
      if (elect_one()) tma_load_2d(sB + static_cast<size_t>(i) * stageB, &tmX, (kit0 + i) * kBlockK, t0, &full[i]);
    int s = 0;
    uint32_t ph = 0;
    for (int it = npre; it < kps; ++it) {  // (only when npre == stages)
      if (!warp_mbar_wait(&empty[s], ph, p.err, p.spin)) {
        s_timed_out = 1;
        break;
      }
      issued = it + 1;
      if (elect_one()) {
        mbar_arrive_expect_tx(&full[s], tx);
        tma_load_2d(sA + static_cast<size_t>(s) * kStageA, &tmW, (kit0 + it) * kBlockK, n0, &full[s]);
        tma_load_2d(sB + static_cast<size_t>(s) * stageB, &tmX, (kit0 + it) * kBlockK, t0, &full[s]);
      }
      if (++s == stages) {
        s = 0;
        ph ^= 1;
      }
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer.  A 16-deep K step is 32 bytes: +2 in the
    // descriptors' start-address field (shared address >> 4, 14 bits; shared
    // memory is below 256 KB, so the field never carries).
    const uint32_t idesc = umma_idesc_bf16(kBlockN, BT);
    const uint64_t a_base = umma_desc_sw128(smem_u32(sA)), b_base = umma_desc_sw128(smem_u32(sB));
    int s = 0;
    uint32_t ph = 0;
    for (int it = 0; it < kps; ++it) {
      if (!warp_mbar_wait(&full[s], ph, p.err, p.spin)) {
        s_timed_out = 1;
        break;
      }
      tc_fence_after();
      if (elect_one()) {
        const uint64_t ad = a_base + static_cast<uint64_t>((s * kStageA) >> 4);
        const uint64_t bd = b_base + static_cast<uint64_t>((s * stageB) >> 4);
#pragma unroll
        for (int kk = 0; kk < kBlockK / 16; ++kk)
          umma_bf16(tmem, ad + 2 * kk, bd + 2 * kk, idesc, (it | kk) != 0 ? 1u : 0u);
        umma_commit(&empty[s]);
      }
      __syncwarp();
      if (++s == stages) {
        s = 0;
        ph ^= 1;
      }
    }
    if (elect_one()) umma_commit(done);
  }
  __syncwarp();

  // ---------------- epilogue: warp w owns TMEM lanes [32w, 32w+32) = weight rows
  pdl_wait();
  if constexpr (EPI == EPI_KV) {
    for (int j = threadIdx.x; j < BT; j += blockDim.x) {
      const int t = t0 + j;
      int2 sp = make_int2(0, 0x7fffffff);
      if (t < p.M) {
        const int i = t / p.rows_per_seq, jr = t - i * p.rows_per_seq;
        sp.x = p.seq_slot[i];
        sp.y = (p.pos_base ? p.pos_base[sp.x] : 0) + jr;
      }
      tok[j] = sp;
    }
  }
  // Inputs of the four-feature epilogue that do not depend on this GEMM's
  // result load while the MMAs run: the bias of the lane's four features and,
  // for a residual update, the first row this warp will own.
  const int cols = max(0, min(BT, p.M - t0));
  // split-K: the tile's groups of four token rows, and those this CTA finishes
  const int S = p.splits, n_grp = (cols + 3) / 4;
  const int g_lo = n_grp * split / S, g_hi = n_grp * (split + 1) / S;
  if (S > 1) {
    const int g_max = (n_grp + S - 1) / S;
    if (threadIdx.x == 0)
      mbar_arrive_expect_tx(inbox_bar, static_cast<uint32_t>(S * (g_hi - g_lo)) * kGroupBytes);
    for (int g = threadIdx.x; g < n_grp; g += kThreads) {
      const int owner = ((g + 1) * S - 1) / n_grp, lg = g - n_grp * owner / S;
      dest[g] = make_uint2(dsmem_map(smem_u32(smem) + static_cast<uint32_t>(split * g_max + lg) * kGroupBytes, owner),
                           dsmem_map(smem_u32(inbox_bar), owner));
    }
  }
  float b4[4] = {0.f, 0.f, 0.f, 0.f};
  // (split-K: a warp's first group of four rows)
  float4 pre[4];
  if (S > 1 || p.stats_out) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int nn = n0 + 4 * lane + i;
      b4[i] = (p.bias && nn < p.N) ? bf2f(p.bias[nn]) : 0.f;
    }
  }
  auto load_group = [&](int g) {  // the residual rows of group g
    if constexpr (EPI == EPI_RESID) {
#pragma unroll
      for (int k = 0; k < 4; ++k)
        pre[k] = 4 * g + k < cols
                     ? *reinterpret_cast<const float4 *>(p.resid + static_cast<size_t>(t0 + 4 * g + k) * p.ld_resid +
                                                         n0 + 4 * lane)
                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  if (S > 1 && g_lo + warp < g_hi) load_group(g_lo + warp);
  __syncthreads();
  bool ok = mbar_wait(done, 0, p.err, p.spin);
  if (!ok) s_timed_out = 1;
  tc_fence_after();
  __syncwarp();
  // warp w reads TMEM lane quarter w % 4 (weight rows 32 (w % 4) ..) and the
  // token-column chunks [c_lo, c_hi) of its half of the tile
  const int quarter = warp & 3, half = warp >> 2;
  const int n = n0 + quarter * 32 + lane;
  const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16);
  const int n_chunks = BT / 16, c_per = (n_chunks + 1) / 2;
  const int c_lo = half * c_per, c_hi = min(n_chunks, c_lo + c_per);

  if (p.splits == 1 && !p.stats_out) {
    const float bn = (p.bias && n < p.N) ? bf2f(p.bias[n]) : 0.f;
    for (int c = c_lo; c < c_hi; ++c) {
      float v[16];
      tmem_ld16(trow + c * 16, v);
      if (ok) epi_chunk<EPI>(p, t0 + c * 16, n, bn, v, tok + c * 16);
    }
  } else {
    // Four-feature epilogue: a warp owns token rows (lane l: features
    // 4l..4l+3), so a row's LayerNorm statistics over this 128-feature tile
    // are two warp reductions.
    const int stat_tiles = p.N / kBlockN;
    auto finish_row = [&](int tl, const float4 &acc, bool valid, const float4 &old) {
      float fin[4] = {0.f, 0.f, 0.f, 0.f};
      if (valid) epi_quad<EPI>(p, t0 + tl, n0 + 4 * lane, acc, b4, old, tok + tl, fin);
      if (p.stats_out) {
        const float mean = warp_sum((fin[0] + fin[1]) + (fin[2] + fin[3])) * (1.0f / 128.f);
        const float d0 = fin[0] - mean, d1 = fin[1] - mean, d2 = fin[2] - mean, d3 = fin[3] - mean;
        const float m2 = warp_sum((d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3));
        if (lane == 0 && valid)
          p.stats_out[static_cast<size_t>(t0 + tl) * stat_tiles + ntile] = make_float2(mean, m2);
      }
    };
    const int r = quarter * 32 + lane;
    float *tile = reinterpret_cast<float *>(smem);
    if (S > 1) {
      // Split-K: every CTA pushes its fp32 partials of each group of four
      // token rows into the inbox of the CTA that finishes the group (over the
      // pipeline buffers, free once all CTAs' MMAs are done), 16 bytes (four
      // tokens of one feature) per asynchronous store; the inbox's barrier
      // counts the bytes.  The owner adds the S partials in split order from
      // its own shared memory.  From the last MMA to the CTA's end this takes
      // 1400 cycles at 9 rows and 4200 at 64 (1280 x 1280); pulling over DSMEM
      // between two release / acquire cluster barriers took 4300 and 6000.
      cluster_arrive_relaxed();
      cluster_wait();
      const int pos = (r & ~3) | ((r + (r >> 3)) & 3);  // conflict-free for the owner's reads
      for (int c = c_lo; c < c_hi; ++c) {
        float v[16];
        tmem_ld16_issue(trow + c * 16, v);
        tmem_ld_wait(v);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int g = c * 4 + k;
          if (g >= n_grp) break;
          const uint2 d = dest[g];
          dsmem_push_f32x4(d.x + 16u * pos, make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]), d.y);
        }
      }
      if (!mbar_wait(inbox_bar, 0, p.err, p.spin)) {
        ok = false;
        s_timed_out = 1;
        // partials on their way into this CTA must land before it leaves
        mbar_drain(inbox_bar, 0);
      }
      __syncwarp();
      const int g_max = (n_grp + S - 1) / S;
      for (int g = g_lo + warp; g < g_hi; g += kThreads / 32) {
        if (g != g_lo + warp) load_group(g);
        const float4 *in = reinterpret_cast<const float4 *>(smem + static_cast<size_t>(g - g_lo) * kGroupBytes);
        float4 acc[4];  // feature 4 lane + i, its four tokens
#pragma unroll
        for (int i = 0; i < 4; ++i) acc[i] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 4
        for (int sp = 0; sp < S; ++sp) {
          const float4 *src = in + static_cast<size_t>(sp * g_max) * (kGroupBytes / 16);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 v = src[4 * lane + ((i + (lane >> 1)) & 3)];
            acc[i].x += v.x;
            acc[i].y += v.y;
            acc[i].z += v.z;
            acc[i].w += v.w;
          }
        }
        const float4 row[4] = {make_float4(acc[0].x, acc[1].x, acc[2].x, acc[3].x),
                               make_float4(acc[0].y, acc[1].y, acc[2].y, acc[3].y),
                               make_float4(acc[0].z, acc[1].z, acc[2].z, acc[3].z),
                               make_float4(acc[0].w, acc[1].w, acc[2].w, acc[3].w)};
#pragma unroll
        for (int k = 0; k < 4; ++k)
          if (4 * g + k < cols) finish_row(4 * g + k, row[k], ok, pre[k]);
      }
    } else {
      for (int c = c_lo; c < c_hi; ++c) {
        float v[16];
        tmem_ld16(trow + c * 16, v);
#pragma unroll
        for (int jj = 0; jj < 16; ++jj) tile[(c * 16 + jj) * kBlockN + r] = v[jj];
      }
      __syncthreads();
      for (int tl = warp; tl < cols; tl += kThreads / 32) {
        float4 old = make_float4(0.f, 0.f, 0.f, 0.f);
        if constexpr (EPI == EPI_RESID)
          old = *reinterpret_cast<const float4 *>(p.resid + static_cast<size_t>(t0 + tl) * p.ld_resid + n0 + 4 * lane);
        finish_row(tl, *reinterpret_cast<const float4 *>(tile + tl * kBlockN + 4 * lane), ok, old);
      }
    }
  }

  // After a timeout, copies this CTA requested may still be landing and
  // MMAs it issued may still be running: wait for both (bounded) before the
  // CTA frees its TMEM and leaves.  Otherwise every copy was consumed by the
  // MMA thread and the MMAs completed before the epilogue read TMEM.
  __syncthreads();
  if (threadIdx.x == 0 && s_timed_out) {
    for (int q = max(0, issued - stages); q < issued; ++q)
      mbar_drain(&full[q % stages], static_cast<uint32_t>(q / stages) & 1u);
    mbar_drain(done, 0u);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) tmem_dealloc(tmem, p.tmem_cols);
}

// --------------------------------------------------------------- host ----
static PFN_cuTensorMapEncodeTiled_v12000 encode_fn() {
  static PFN_cuTensorMapEncodeTiled_v12000 fn = nullptr;
  static std::once_flag once;
  std::call_once(once, [] {
    void *ptr = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &ptr, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(ptr);
  });
  return fn;
}

const CUtensorMap *tmap_bf16_2d(const void *ptr, uint64_t rows, uint64_t cols, uint32_t box_rows) {
  static std::mutex mu;
  static std::map<std::tuple<uintptr_t, uint64_t, uint64_t, uint32_t>, CUtensorMap *> cache;
  std::lock_guard<std::mutex> lock(mu);
  auto key = std::make_tuple(reinterpret_cast<uintptr_t>(ptr), rows, cols, box_rows);
  auto it = cache.find(key);
  if (it != cache.end()) return it->second;
  auto fn = encode_fn();
  if (!fn) return nullptr;
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || (cols * 2) % 16 || box_rows == 0 || box_rows > 256)
    return nullptr;
  CUtensorMap *m = new CUtensorMap;
  cuuint64_t gdim[2] = {cols, rows};
  cuuint64_t gstride[1] = {cols * 2};
  cuuint32_t box[2] = {static_cast<cuuint32_t>(kBlockK), box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), gdim, gstride,
                  box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    delete m;
    return nullptr;
  }
  cache.emplace(key, m);
  return m;
}

// 3-D view of a row-major [rows][cols] bf16 matrix as (64 columns, row,
// 64-column block) with strides (cols * 2 bytes, 128 bytes): a box of
// {64, 8, kblocks} is 8 consecutive rows by kblocks * 64 columns, landing in
// shared memory as [kblock][8 rows][128 B] with 128-byte swizzling (one
// swizzle atom per k-block), in a single copy.
bool tmap_bf16_units(CUtensorMap *m, const void *ptr, uint64_t rows, uint64_t cols, uint32_t kblocks) {
  auto fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(ptr) & 15) || cols % 64 || kblocks == 0 || kblocks > 256 ||
      kblocks > cols / 64)
    return false;
  cuuint64_t gdim[3] = {64, rows, cols / 64};
  cuuint64_t gstride[2] = {cols * 2, 128};
  cuuint32_t box[3] = {64, 8, kblocks};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), gdim, gstride, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tmap_bf16_rows(CUtensorMap *m, const void *ptr, uint32_t rows, uint64_t cols, uint64_t ld, uint32_t kblocks) {
  auto fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(ptr) & 15) || cols % 64 || (ld * 2) % 16 || ld < cols || rows == 0 ||
      rows > 256 || kblocks == 0 || kblocks > 256 || kblocks > cols / 64)
    return false;
  cuuint64_t gdim[3] = {64, rows, cols / 64};
  cuuint64_t gstride[2] = {ld * 2, 128};
  cuuint32_t box[3] = {64, rows, kblocks};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), gdim, gstride, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

bool tmap_bf16_cache(CUtensorMap *m, const void *ptr, uint64_t ctx, uint64_t outer, uint32_t box_rows) {
  auto fn = encode_fn();
  if (!fn || (reinterpret_cast<uintptr_t>(ptr) & 15) || ctx == 0 || outer == 0 || box_rows == 0 || box_rows > 256 ||
      box_rows > ctx)
    return false;
  cuuint64_t gdim[3] = {64, ctx, outer};
  cuuint64_t gstride[2] = {128, ctx * 128};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void *>(ptr), gdim, gstride, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

void gemm_token_tiling(int M, int *BT, int *n_tt) {
  const int nt = (M + kMaxBT - 1) / kMaxBT;
  const int per = (M + nt - 1) / nt;
  *n_tt = nt;
  *BT = ((per + 15) / 16) * 16;
}

int gemm_splits(int N, int K) {
  const int n_tiles = (N + kBlockN - 1) / kBlockN;
  const int k_iters = K / kBlockK;
  int best = 1;
  for (int s = 1; s <= k_iters && s <= 16; ++s) {
    if (k_iters % s) continue;
    if (n_tiles * s > 160) break;
    if (k_iters / s < 2) break;
    best = s;
  }
  return best;
}

template <int EPI>
static cudaError_t cluster_fits(int splits, size_t smem, dim3 grid) {
  static std::mutex mu;
  static std::map<std::pair<int, size_t>, int> seen;
  std::lock_guard<std::mutex> lock(mu);
  auto key = std::make_pair(splits, smem);
  auto it = seen.find(key);
  if (it == seen.end()) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = 1;
    attr.val.clusterDim.y = 1;
    attr.val.clusterDim.z = splits;
    cfg.attrs = &attr;
    cfg.numAttrs = 1;
    int n = 0;
    cudaError_t e = cudaOccupancyMaxActiveClusters(&n, gemm_tc_kernel<EPI>, &cfg);
    if (e != cudaSuccess) return e;
    it = seen.emplace(key, n).first;
  }
  return it->second > 0 ? cudaSuccess : cudaErrorInvalidConfiguration;
}

template <int EPI>
static cudaError_t launch_typed(const CUtensorMap *tw, const CUtensorMap *tx, const GemmParams &p,
                                size_t smem, cudaStream_t s, bool pdl) {
  const bool clustered = p.splits > 1;
  const dim3 grid(p.n_tt, (p.N + kBlockN - 1) / kBlockN, clustered ? p.splits : 1);
  if (clustered) {
    cudaError_t e = cluster_fits<EPI>(p.splits, smem, grid);
    if (e != cudaSuccess) return e;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  int na = 0;
  if (clustered) {
    attr[na].id = cudaLaunchAttributeClusterDimension;
    attr[na].val.clusterDim.x = 1;
    attr[na].val.clusterDim.y = 1;
    attr[na].val.clusterDim.z = p.splits;
    ++na;
  }
  if (pdl) {
    attr[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = attr;
  cfg.numAttrs = na;
  return cudaLaunchKernelEx(&cfg, gemm_tc_kernel<EPI>, *tw, *tx, p);
}

cudaError_t gemm_init() {
  static cudaError_t status = cudaErrorNotReady;
  static std::once_flag once;
  std::call_once(once, [] {
    const int lim = 227 * 1024;
    status = cudaFuncSetAttribute(gemm_tc_kernel<EPI_F32>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (status == cudaSuccess)
      status = cudaFuncSetAttribute(gemm_tc_kernel<EPI_BF16>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (status == cudaSuccess)
      status = cudaFuncSetAttribute(gemm_tc_kernel<EPI_GELU>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (status == cudaSuccess)
      status = cudaFuncSetAttribute(gemm_tc_kernel<EPI_RESID>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    if (status == cudaSuccess)
      status = cudaFuncSetAttribute(gemm_tc_kernel<EPI_KV>, cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
    // split-K clusters of up to 16 CTAs
    const void *fns[] = {reinterpret_cast<const void *>(gemm_tc_kernel<EPI_F32>),
                         reinterpret_cast<const void *>(gemm_tc_kernel<EPI_BF16>),
                         reinterpret_cast<const void *>(gemm_tc_kernel<EPI_GELU>),
                         reinterpret_cast<const void *>(gemm_tc_kernel<EPI_RESID>),
                         reinterpret_cast<const void *>(gemm_tc_kernel<EPI_KV>)};
    for (const void *f : fns)
      if (status == cudaSuccess)
        status = cudaFuncSetAttribute(f, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    for (const void *f : fns)
      if (status == cudaSuccess) status = prefer_max_shared(f);
  });
  return status;
}

// Tiling, split and shared-memory plan of one launch; false if it does not fit.
static bool plan_gemm(GemmParams &p, size_t *smem_out) {
  if (p.M <= 0 || p.N <= 0 || p.K <= 0 || p.K % kBlockK) return false;
  gemm_token_tiling(p.M, &p.BT, &p.n_tt);
  if (p.splits < 1) p.splits = 1;
  const int k_iters = p.K / kBlockK;
  if (k_iters % p.splits) return false;
  p.kps = k_iters / p.splits;
  const size_t stageA = kStageA, stageB = static_cast<size_t>(p.BT) * kBlockK * 2;
  const size_t red = static_cast<size_t>(p.BT) * sizeof(int2) +
                     (p.splits > 1 ? static_cast<size_t>(p.BT / 4) * sizeof(uint2) : 0);
  uint32_t cols = 32;
  while (cols < static_cast<uint32_t>(p.BT)) cols <<= 1;
  p.tmem_cols = cols;
  if (red + stageA + stageB > kSmemBudget) return false;
  int stages = static_cast<int>((kSmemBudget - red) / (stageA + stageB));
  if (stages > p.kps) stages = p.kps;
  if (stages > 16) stages = 16;
  size_t pipe = stages * (stageA + stageB);
  p.stages = stages;
  // the staged epilogues reuse the pipeline buffers for a [BT][128] fp32 tile
  if (p.stats_out) pipe = std::max<size_t>(pipe, 512 * static_cast<size_t>(p.BT));
  if (p.splits > 1)  // inbox: every split's partials of the CTA's share of the token groups
    pipe = std::max<size_t>(pipe, static_cast<size_t>(p.splits) * ((p.BT / 4 + p.splits - 1) / p.splits) * kGroupBytes);
  size_t smem = 1024 + pipe + (2 * stages + 2) * 8 + 32 + 16 + red;
  // A CTA blocks in tcgen05.alloc while co-resident CTAs hold the SM's 512
  // TMEM columns; CTAs of one cluster wait for each other, so no more CTAs
  // may fit on an SM (by shared memory) than can hold TMEM at once.
  const int tmem_ctas = 512 / static_cast<int>(cols);
  if (tmem_ctas < 4)
    smem = std::max<size_t>(smem, kSmemPerSM / (tmem_ctas + 1) + 1);
  if (smem > 227 * 1024) return false;
  p.pipe_bytes = static_cast<int>(pipe);
  *smem_out = smem;
  return true;
}

cudaError_t launch_gemm(const void *X, const void *W, GemmParams p, cudaStream_t s, bool pdl) {
  if (p.spin <= 0) p.spin = kSpinLimitCycles;
  const bool quad = p.splits > 1 || p.stats_out;  // the staged (four-feature) epilogue
  if (!X || (p.epi == EPI_HEAD && p.stats_out)) return cudaErrorInvalidValue;
  if ((p.stats_out || p.epi == EPI_RESID) && p.N % kBlockN) return cudaErrorInvalidValue;
  if (p.epi == EPI_RESID && (p.ld_resid % 4 || (reinterpret_cast<uintptr_t>(p.resid) & 15)))
    return cudaErrorInvalidValue;
  if (quad && p.epi == EPI_KV && (p.N % 4 || p.q_cols % 4 || p.d_model % 4 || p.ld_out % 4))
    return cudaErrorInvalidValue;
  if (quad && p.epi == EPI_RESID && (p.tap0 || p.tap1) && p.ld_tap % 4) return cudaErrorInvalidValue;
  // Past wide_min_rows() pairs of SMs on 256-row weight tiles (same bits).
  // They write four features at a time whatever the split, so a key/value
  // scatter with odd strides stays here.  They run the output head at any
  // number of rows.
  const bool quads = p.epi != EPI_KV || !(p.N % 4 || p.q_cols % 4 || p.d_model % 4 || p.ld_out % 4);
  const int wide_m = wide_min_rows(p.N, p.K, std::max(1, p.splits), pdl);
  if (p.epi == EPI_HEAD || (p.M > wide_m && quads)) return launch_gemm_wide(X, W, p, s, pdl);
  size_t smem = 0;
  if (!plan_gemm(p, &smem)) return cudaErrorInvalidValue;
  const CUtensorMap *tw = tmap_bf16_2d(W, p.N, p.K, kBlockN);
  const CUtensorMap *tx = tmap_bf16_2d(X, p.M, p.K, p.BT);
  if (!tw || !tx) return cudaErrorInvalidValue;
  switch (p.epi) {
    case EPI_F32: return launch_typed<EPI_F32>(tw, tx, p, smem, s, pdl);
    case EPI_BF16: return launch_typed<EPI_BF16>(tw, tx, p, smem, s, pdl);
    case EPI_GELU: return launch_typed<EPI_GELU>(tw, tx, p, smem, s, pdl);
    case EPI_RESID: return launch_typed<EPI_RESID>(tw, tx, p, smem, s, pdl);
    case EPI_KV: return launch_typed<EPI_KV>(tw, tx, p, smem, s, pdl);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace wf

// ------------------------------------------------------- C entry points --
extern "C" size_t wf_gemm_scratch_bytes(int32_t M, int32_t N, int32_t K) {
  // split-K partials are reduced on chip (cluster shared memory): no scratch
  (void)M;
  (void)N;
  (void)K;
  return 0;
}

extern "C" wf_status wf_gemm_bf16(const void *d_x, const void *d_w, const void *d_b, float *d_y,
                                  int32_t M, int32_t N, int32_t K, void *d_scratch,
                                  size_t scratch_bytes, void *stream) {
  (void)d_scratch;
  (void)scratch_bytes;
  if (!d_x || !d_w || !d_y || M <= 0 || N <= 0 || K <= 0) return WF_ERR_INVALID;
  if (K % 64) return WF_ERR_UNSUPPORTED;
  wf::GemmParams p = {};
  p.M = M;
  p.N = N;
  p.K = K;
  p.epi = wf::EPI_F32;
  p.bias = static_cast<const wf::bf16 *>(d_b);
  p.out_f32 = d_y;
  p.ld_out = N;
  p.splits = wf::gemm_splits(N, K);
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (wf::gemm_init() != cudaSuccess) return WF_ERR_CUDA;
  return wf::launch_gemm(d_x, d_w, p, s, false) == cudaSuccess ? WF_OK : WF_ERR_CUDA;
}
