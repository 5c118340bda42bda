// Projections of many token rows on pairs of SMs (tcgen05 cta_group::2).
//
// The skinny-M kernel of wf_gemm.cu gives every 128 x BT tile to one CTA; at
// hundreds of rows each CTA then pulls its whole weight slab and token slab
// through L2 for a small tile, and the pushes of its split-K partials grow with
// the rows.  Here two CTAs (one cluster) share a tile of 256 weight rows by BT
// tokens: each holds its own 128 weight rows and half of the tokens in shared
// memory, the even CTA issues one 256-row MMA for both, so a CTA fetches
// 128 + BT/2 operand rows for 128 x BT outputs.  The grid is persistent (one
// pair per two SMs, tiles dealt round robin, token tiles of one weight tile
// next to each other so the weights leave HBM once), with two TMEM
// accumulators: eight epilogue warps work on one while the MMAs fill the
// other.
//
// What bounds it depends on the shape (clocks inside the kernel, cycles of 0.5
// ns, means over the CTAs; 864 rows within a step of 96 sequences).  A launch
// starts with ~2,700 to its first tile of operands and ends 4,000-5,000 after
// its last MMA (TMEM reads, staging, stores); between them:
//  - fc2, one tile of 80 k-steps: ~225 a step of 20 KB, the copies' rate of ~90
//    bytes per cycle and SM; 16,000-18,000 of ~25,000 (prefetching the weights
//    into L2 first takes the same engine and measured 5-15% slower);
//  - out, cross out, cross query, 20 steps: ~6,500 of 14,000, so launch and
//    epilogue weigh more than the copies;
//  - fc1, two tiles a pair with GELU: 34,700, of them 11,300 in which the MMAs
//    wait for the epilogue to free an accumulator, 4,400 for copies, and 12,000
//    of epilogue after the last MMA;
//  - acoustic K/V (24000 rows, 12 tiles a pair, 256 tokens): ~600 a step of 32 KB
//    for 512 of MMAs; the MMAs wait for copies two thirds of the time, for the
//    epilogue a tenth.
// Measured against one CTA per tile that went through the chunks of its K in
// turn, at 864 rows (one launch, cold): out / cross out / fc2 36 -> 15 us on average, fc1 39 -> 23, QKV 37 -> 19,
// cross query 18 -> 11; acoustic K/V of 8 requests (12000 x 2560 x 1280)
// 139 -> 75 us; 837 x 1280 x 5120 back to back 47 -> 18 us.  Stages of 128
// columns instead of 64 (fewer barrier rounds, a shallower ring) measured 10%
// slower there, and every single token tile of 64, 96 or 128 rows 2-5% slower
// over a 96-sequence step than the choice of gemm_wide_plan.
// The output head (51866 x 1280) runs here at any number of rows: against one
// CTA per 128 ids and token tile, whose epilogue folded (max, sum, argmax,
// Gumbel) records through five shuffles per step, 33 -> 28 us at 9 rows (one
// read of the weights is 20), 61 -> 30 at 144, 304 -> 86 at 864, and sampling
// 288 rows 205 -> 86.
//
// Arithmetic: K is cut into the same `splits` chunks as the cluster split-K of
// wf_gemm.cu, each chunk accumulates on its own in TMEM, and the chunks are
// added in order from zero in fp32 (in registers), so a row's bits do not
// depend on which of the two kernels ran it.
//
// Roles per CTA: warp 0 requests its CTA's tiles by TMA; warp 1
// of the even CTA issues the MMAs; warp 2 owns TMEM; warps 4 and on run the
// epilogue, two or four per TMEM lane quarter, each with its group of the
// token columns.
#include <mutex>

#include "wf_device.cuh"
#include "wf_gemm_epi.cuh"
#include "wf_internal.h"

namespace wf {

constexpr int kWideEpiWarp = 4;      // first epilogue warp
constexpr int kWideBK = 64;               // K per stage (one 128-byte swizzle atom)
constexpr int kWideA = 128 * kWideBK * 2;  // weight tile: [128 rows][128 B]
constexpr int kWideMaxStages = 10;
constexpr int kWideStage = 64 * 128 * 4;  // two staging buffers per column group, 64 token rows in all
// Epilogue warps: two per TMEM lane quarter, four for the output head, whose
// per-id arithmetic needs the latency hiding (51866 ids, one launch, cold:
// sampling 288 rows 116 us with eight warps, 86 with sixteen; greedy 864 rows
// with their logits 116 and 86).
template <int EPI>
constexpr int kWideEpiWarps = EPI == EPI_HEAD ? 16 : 8;
template <int EPI>
constexpr int kWideThreads = 32 * (4 + kWideEpiWarps<EPI>);
constexpr int kWideAcc = 256;        // TMEM columns per accumulator
constexpr uint32_t kWideTmem = 512;

// mbarrier and table space after the pipeline and staging buffers
constexpr int kWideBars = (2 * kWideMaxStages + 5) * 8;
constexpr int kWideTok = 2 * 256 * 8;  // (slot, position) per token row, two tiles
constexpr int kWideFixed = 1024 + kWideStage + kWideTok + kWideBars + 32;

__device__ __forceinline__ void group_barrier(int hg) {  // the four epilogue warps of a column group
  asm volatile("bar.sync %0, 128;" ::"r"(1 + hg) : "memory");
}

// ---- output head: R token rows over a 128-id vocabulary tile.  Lane l
// holds ids 4l..4l+3 of each row; `masked` has a bit for each of them that is
// suppressed or past the vocabulary.  Reductions over the warp run on integer
// keys in the order of the floats (redux.sync), lowest id on ties; the
// rows go through each stage together so that its latencies overlap.

// The warp's best key and the lowest id of the lanes that hold it.
__device__ __forceinline__ uint32_t warp_argmax(uint32_t key, int id, int *arg) {
  const uint32_t b = __reduce_max_sync(0xffffffffu, key);
  *arg = static_cast<int>(__reduce_min_sync(0xffffffffu, key == b && b != 0u ? static_cast<uint32_t>(id) : 0x7fffffffu));
  return b;
}

// Greedy: maximum and lowest id attaining it.
template <int R>
__device__ __forceinline__ void head_rows_greedy(const float4 (&z4)[R], uint32_t masked, int id0, HeadRec (&r)[R]) {
#pragma unroll
  for (int k = 0; k < R; ++k) {
    const float z[4] = {masked & 1u ? -INFINITY : z4[k].x, masked & 2u ? -INFINITY : z4[k].y,
                        masked & 4u ? -INFINITY : z4[k].z, masked & 8u ? -INFINITY : z4[k].w};
    const float m = fmaxf(fmaxf(z[0], z[1]), fmaxf(z[2], z[3]));  // (NaN only if all are)
    const int id = z[0] == m ? 0 : z[1] == m ? 1 : z[2] == m ? 2 : 3;
    r[k] = HeadRec{};
    r[k].m = key_value(warp_argmax(order_key(m), id0 + id, &r[k].arg));
    r[k].gm = -INFINITY;
    r[k].garg = 0x7fffffff;
  }
}

// Sampling: maximum and sum of exponentials of x = z / T (for the log-sum-exp)
// and the Gumbel-max draw, argmax x - log(-log u).  The four ids of a lane
// share one Philox block.  The draw's order is that of the exponential race
// exp(x) / -log(u), which needs three fast special functions per id; only ids
// within kRaceTol of the warp's best are scored exactly (one lane, nearly
// always), so the draw is that of the exact scores of every id.  (An id whose x is 20 below
// the tile's maximum cannot win, as u lies in [2^-24, 1 - 2^-24]; above that
// the exponent's magnitude stays below 29 in base 2 and its four roundings make
// the fast exponential good to 2^-17.)  The exact scores are rounded to fp32
// themselves, two of them by up to two units in the last place of x together:
// past |x| = kRaceMaxX every id is scored.
// ss[k]: (slot and block row, step) of row k.
template <int R>
__device__ __forceinline__ void head_rows_sample(const GemmParams &p, const float4 (&z4)[R], uint32_t masked, int id0,
                                                 const int2 *ss, HeadRec (&r)[R]) {
  float z[R][4], u[R][4], e[R][4], w[R][4], zmax[R], sum[R];
  const float c = fminf(__fdiv_rn(kLog2e, p.temperature), 3.402823466e38f);
#pragma unroll
  for (int k = 0; k < R; ++k) {
    z[k][0] = masked & 1u ? -INFINITY : z4[k].x;
    z[k][1] = masked & 2u ? -INFINITY : z4[k].y;
    z[k][2] = masked & 4u ? -INFINITY : z4[k].z;
    z[k][3] = masked & 8u ? -INFINITY : z4[k].w;
    zmax[k] = key_value(
        __reduce_max_sync(0xffffffffu, order_key(fmaxf(fmaxf(z[k][0], z[k][1]), fmaxf(z[k][2], z[k][3])))));
  }
#pragma unroll
  for (int k = 0; k < R; ++k) {
    const Philox4 o = philox4x32_10(static_cast<uint32_t>(id0) >> 2, static_cast<uint32_t>(ss[k].x) >> 24,
                                    static_cast<uint32_t>(ss[k].y),
                                    (p.tag << 24) | (static_cast<uint32_t>(ss[k].x) & 0xFFFFFFu),
                                    static_cast<uint32_t>(p.seed), static_cast<uint32_t>(p.seed >> 32));
    sum[k] = 0.f;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      // word_to_open_uniform's (w >> 9 + 1/2) / 2^23, without a conversion: exact
      u[k][i] = __uint_as_float((o.x[i] >> 9) | 0x3f800000u) - 0.999999940395355224609375f;
      w[k][i] = neg_log2_estimate(u[k][i]);
      e[k][i] = (masked >> i) & 1u ? 0.f : exp2f_fast((z[k][i] - zmax[k]) * c);
      sum[k] += e[k][i];
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1)
#pragma unroll
    for (int k = 0; k < R; ++k) sum[k] += __shfl_xor_sync(0xffffffffu, sum[k], off);
  float best[R];
#pragma unroll
  for (int k = 0; k < R; ++k) {
    r[k] = HeadRec{};
    r[k].arg = 0x7fffffff;
    r[k].m = __fdiv_rn(zmax[k], p.temperature);  // = max x: division by T > 0 is monotonic
    r[k].s = zmax[k] == -INFINITY ? 0.f : sum[k];
    // the lane's best e / w by cross products (0 in place of NaN), then the
    // warp's: nonnegative floats are ordered like their bits
    float be = 0.f, bw = 1.f;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (e[k][i] * bw > be * w[k][i]) {
        be = e[k][i];
        bw = w[k][i];
      }
    best[k] = __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(__fdividef(be, bw))));
  }
  // Exact scores of the candidates: each lane's first one of every row
  // together, further ones (rare) after.
  uint32_t cand[R] = {}, gkey[R] = {};
  int gid[R] = {};
  auto take = [&](int k) {  // score row k's lowest candidate of this lane
    const int i = __ffs(static_cast<int>(cand[k])) - 1;
    const float zi = i == 0 ? z[k][0] : i == 1 ? z[k][1] : i == 2 ? z[k][2] : z[k][3];
    const float ui = i == 0 ? u[k][0] : i == 1 ? u[k][1] : i == 2 ? u[k][2] : u[k][3];
    const float x = __fdiv_rn(zi, p.temperature) - logf(-logf(ui));
    const uint32_t key = i < 0 ? 0u : order_key((masked >> i) & 1u ? -INFINITY : x);
    if (key > gkey[k]) {
      gkey[k] = key;
      gid[k] = id0 + i;
    }
    cand[k] &= cand[k] - 1;
  };
  uint32_t more = 0;
#pragma unroll
  for (int k = 0; k < R; ++k) {
    // without a maximum below kRaceMaxX every id is scored; a masked id scores
    // -inf, so that a row without any other id has one
    const bool all = !(fabsf(r[k].m) <= kRaceMaxX);
    const float floor = best[k] - best[k] * kRaceTol;
    cand[k] = masked;
    gid[k] = 0x7fffffff;
    gkey[k] = 0u;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (all || e[k][i] >= floor * w[k][i]) cand[k] |= 1u << i;
    take(k);
    more |= cand[k];
  }
  while (__any_sync(0xffffffffu, more)) {
    more = 0;
#pragma unroll
    for (int k = 0; k < R; ++k) {
      take(k);
      more |= cand[k];
    }
  }
#pragma unroll
  for (int k = 0; k < R; ++k) r[k].gm = key_value(warp_argmax(gkey[k], gid[k], &r[k].garg));
}

// HC: 16-column chunks of a column group kept in registers (the sum over the K
// chunks); 0: no split (p.splits == 1), the epilogue reads TMEM directly.
template <int EPI, int HC>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kWideThreads<EPI>, 1)
    gemm_wide_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX,
                     const GemmParams p) {
  constexpr int kEW = kWideEpiWarps<EPI>, kGroups = kEW / 4;
  constexpr int kSlice = 32 / kGroups;  // token rows per staging buffer
  constexpr int kR = kSlice / 4;        // of them a warp's
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t *smem = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  const int BT = p.BT, stages = p.stages;
  const uint32_t stageB = static_cast<uint32_t>(BT) * kWideBK;  // [BT / 2 rows][128 B]
  const uint32_t stage_bytes = kWideA + stageB;
  float *stg = reinterpret_cast<float *>(smem + stages * stage_bytes);
  int2 *tok = reinterpret_cast<int2 *>(reinterpret_cast<uint8_t *>(stg) + kWideStage);
  uint64_t *full = reinterpret_cast<uint64_t *>(reinterpret_cast<uint8_t *>(tok) + kWideTok);
  // (even CTA: the stage's tiles of both CTAs landed)
  uint64_t *empty = full + kWideMaxStages;   // the MMAs that read the stage completed
  uint64_t *accf = empty + kWideMaxStages;   // accumulator holds a finished chunk
  uint64_t *acce = accf + 2;                 // even CTA: all epilogue warps of the pair are done with it
  uint64_t *done = acce + 2;                 // even CTA: every MMA completed
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done + 1);
  volatile int &s_timed_out = *reinterpret_cast<int *>(tmem_slot + 1);
  // the other CTA's timeout flag and requested k-steps, written by it at its end
  volatile uint32_t *s_peer = tmem_slot + 2;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int pair = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;
  const int nk = p.kps * p.splits;  // k-steps (stages) of a tile
  const int tiles = p.n_ptiles;

  if (threadIdx.x == 0) {
    s_timed_out = 0;
    tma_prefetch_desc(&tmW);
    tma_prefetch_desc(&tmX);
    for (int s = 0; s < stages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&accf[a], 1);
      mbar_init(&acce[a], 2 * kEW);
    }
    mbar_init(done, 1);
    fence_barrier_init();
    fence_proxy_async();
  }
  __syncwarp();
  if (warp == 2) tmem_alloc_pair(tmem_slot, kWideTmem);
  tc_fence_before();
  cluster_sync();  // barriers of both CTAs initialised, TMEM allocated
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_launch_dependents();

  int issued = 0;  // stages whose tiles this CTA requested
  if (warp == 0) {
    // ---------------- TMA producer: this CTA's 128 weight rows and BT/2 token
    // rows; both CTAs' copies complete on the even CTA's barrier, which
    // expects them all.  The first tile's weights do not depend on the
    // previous kernel.
    const uint32_t full_u32 = dsmem_map(smem_u32(full), 0);
    auto load_w = [&](int st, int row, int s) {
      if (elect_one()) {
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * stage_bytes);
        tma_load_2d_pair(smem + s * stage_bytes, &tmW, st * kWideBK, row, full_u32 + 8 * s);
      }
    };
    auto load_x = [&](int st, int row, int s) {
      if (elect_one())
        tma_load_2d_pair(smem + s * stage_bytes + kWideA, &tmX, st * kWideBK, row, full_u32 + 8 * s);
    };
    // stage and phase step along: runtime divisions here would cost more than
    // the copies' issue
    const int npre = min(nk, stages);
    int s = 0;
    uint32_t ph = 1;  // a fresh barrier passes the wait for the phase before its first
    bool ok = true;
    for (int tile = pair; tile < tiles && ok; tile += n_pairs) {
      const int nt = tile / p.n_tt;
      const int wrow = nt * 256 + rank * 128, xrow = (tile - nt * p.n_tt) * BT + rank * (BT / 2);
      int st = 0;
      if (tile == pair) {
        for (; st < npre; ++st) load_w(st, wrow, st);
        pdl_wait();
        for (st = 0; st < npre; ++st) load_x(st, xrow, st);
        issued = npre;
        if ((s = npre) == stages) {
          s = 0;
          ph = 0;
        }
      }
      for (; st < nk; ++st) {
        if (!warp_mbar_wait(&empty[s], ph, p.err, p.spin)) {
          ok = false;
          break;
        }
        load_w(st, wrow, s);
        load_x(st, xrow, s);
        ++issued;
        if (++s == stages) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    // every stage read before the CTA leaves (the even CTA's commits arrive here)
    for (int i = 0; i < stages && ok; ++i) {
      ok = warp_mbar_wait(&empty[s], ph, p.err, p.spin);
      if (++s == stages) {
        s = 0;
        ph ^= 1;
      }
    }
    if (!ok) s_timed_out = 1;
  } else if (warp == 1 && rank == 0) {
    // ---------------- MMA issuer for the pair
    const uint32_t idesc = umma_idesc_bf16(256, BT);
    const uint64_t base = umma_desc_sw128(smem_u32(smem));
    int s = 0, q = 0;  // stage; chunk counter over all tiles
    uint32_t ph = 0;
    bool ok = true;
    for (int tile = pair; tile < tiles && ok; tile += n_pairs) {
      for (int r = 0; r < p.splits && ok; ++r, ++q) {
        if (q >= 2 && !warp_mbar_wait(&acce[q & 1], static_cast<uint32_t>((q >> 1) - 1) & 1u, p.err, p.spin)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t dacc = tmem + (q & 1) * kWideAcc;
        for (int kin = 0; kin < p.kps; ++kin) {
          if (!warp_mbar_wait(&full[s], ph, p.err, p.spin)) {
            ok = false;
            break;
          }
          tc_fence_after();
          if (elect_one()) {
            const uint64_t ad = base + static_cast<uint64_t>((s * stage_bytes) >> 4);
            const uint64_t bd = ad + static_cast<uint64_t>(kWideA >> 4);
#pragma unroll
            for (int kk = 0; kk < kWideBK / 16; ++kk)
              umma_bf16_pair(dacc, ad + 2 * kk, bd + 2 * kk, idesc, (kin | kk) != 0 ? 1u : 0u);
            umma_commit_pair(&empty[s], 3);
          }
          __syncwarp();
          if (++s == stages) {
            s = 0;
            ph ^= 1;
          }
        }
        if (ok && elect_one()) umma_commit_pair(&accf[q & 1], 3);
        __syncwarp();
      }
    }
    if (!ok) s_timed_out = 1;
    if (elect_one()) umma_commit_pair(done, 1);
  } else if (warp >= kWideEpiWarp) {
    // ---------------- epilogue: warp -> lane quarter (its TMEM rows), column group
    const int ew = warp - kWideEpiWarp, quarter = warp & 3, hg = ew >> 2;
    const int gcols = BT / kGroups;  // columns of this warp's group
    const int n_sl = gcols / kSlice;
    const uint32_t trow = tmem + (static_cast<uint32_t>(quarter * 32) << 16) + hg * gcols;
    const uint32_t acce_u32[2] = {dsmem_map(smem_u32(&acce[0]), 0), dsmem_map(smem_u32(&acce[1]), 0)};
    const int feat = quarter * 32 + lane;  // this thread's feature of the 128
    float *buf0 = stg + hg * 2 * kSlice * 128;
    const int stat_tiles = p.N / 128;
    bool ok = true;  // the same in all lanes: the head's reductions take the whole warp
    int q = 0;
    pdl_wait();
    int par = 0, n_written = 0;
    // The next tile's row table -- EPI_KV: (slot * heads * positions +
    // position, 1), or (0, 0) past the cache; a sampling head: (slot and row of
    // the block in the top byte, step) -- and its bias or masked ids, read while
    // the current tile is worked on (their dependent loads cost 4500 cycles a
    // tile in its path).
    int2 next_tok = make_int2(0, 0);
    bf16 next_b[4];
    uint32_t next_masked = 0;
    auto look_ahead = [&](int tile) {
      if (tile >= tiles) return;
      const int nt = tile / p.n_tt, n0 = (nt * 2 + rank) * 128, th = (tile - nt * p.n_tt) * BT + hg * gcols;
      if constexpr (EPI == EPI_KV || EPI == EPI_HEAD) {
        const int j = (ew & 3) * 32 + lane, t = th + j;
        next_tok = make_int2(0, 0);
        if (j < gcols && t < p.M && (EPI == EPI_KV || p.temperature > 0.f)) {
          const int i = t / p.rows_per_seq, jr = t - i * p.rows_per_seq, slot = p.seq_slot[i];
          if constexpr (EPI == EPI_KV) {
            const int pos = (p.pos_base ? p.pos_base[slot] : 0) + jr;
            if (pos < p.ctx) next_tok = make_int2(slot * p.n_heads * p.ctx + pos, 1);
          } else {
            next_tok = make_int2(slot | jr << 24, p.step[slot]);
          }
        }
      }
      next_masked = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int nn = n0 + 4 * lane + i;
        if constexpr (EPI == EPI_HEAD) next_masked |= (nn >= p.N || (p.suppress && p.suppress[nn])) ? 1u << i : 0u;
        else next_b[i] = (p.bias && nn < p.N) ? p.bias[nn] : __float2bfloat16(0.f);
      }
    };
    look_ahead(pair);
    for (int tile = pair; tile < tiles; tile += n_pairs, par ^= 1) {
      const int ntile = (tile / p.n_tt) * 2 + rank, n0 = ntile * 128;
      const int th = (tile % p.n_tt) * BT + hg * gcols;  // first token row of the group
      int2 *tk = tok + par * 256 + hg * (256 / kGroups);
      // this tile's row table and bias were read under the previous tile; the
      // first slice's barrier publishes the table
      float b4[4] = {0.f, 0.f, 0.f, 0.f};
      uint32_t masked = 0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        if constexpr (EPI == EPI_HEAD) masked = next_masked;
        else b4[i] = bf2f(next_b[i]);
      }
      if constexpr (EPI == EPI_KV || EPI == EPI_HEAD) {
        const int j = (ew & 3) * 32 + lane;
        if (j < gcols) tk[j] = next_tok;
      }
      look_ahead(tile + n_pairs);
      // EPI_KV: where this thread's four features go, from a row's table entry
      bf16 *kv_q = nullptr, *kv_c = nullptr;
      if constexpr (EPI == EPI_KV) {
        const int n = n0 + 4 * lane;
        if (n < p.q_cols) {
          kv_q = p.out_bf16 + n;
        } else if (n < p.N) {
          const int c = n - p.q_cols, which = c / p.d_model, hd = c - which * p.d_model;
          kv_c = (which == 0 ? p.kc : p.vc) + static_cast<size_t>(hd >> 6) * p.ctx * 64 + (hd & 63);
        }
      }
      // the residual rows of a slice (this warp's four), loaded ahead of use
      float4 old[kR];
      auto load_old = [&](int sl) {
        if constexpr (EPI == EPI_RESID) {
#pragma unroll
          for (int k = 0; k < kR; ++k) {
            const int t = th + sl * kSlice + quarter * kR + k;
            old[k] = (t < p.M && n0 < p.N)
                         ? *reinterpret_cast<const float4 *>(p.resid + static_cast<size_t>(t) * p.ld_resid + n0 + 4 * lane)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
          }
        }
      };
      load_old(0);
      float acc[HC > 0 ? HC * 16 : 1];
      if constexpr (HC > 0) {
        // add the chunks in order from zero, two 16-column loads in flight
        for (int r = 0; r < p.splits; ++r, ++q) {
          if (ok) ok = warp_mbar_wait(&accf[q & 1], static_cast<uint32_t>(q >> 1) & 1u, p.err, p.spin);
          __syncwarp();
          tc_fence_after();
          const uint32_t src = trow + (q & 1) * kWideAcc;
#pragma unroll
          for (int c = 0; c < HC; c += 2) {
            float v[32];
            if (c < n_sl) tmem_ld16_issue(src + c * 16, v);
            if (c + 1 < n_sl) tmem_ld16_issue(src + c * 16 + 16, v + 16);
            if (c < n_sl) {
              tmem_ld_wait(v);
#pragma unroll
              for (int e = 0; e < 16; ++e) acc[c * 16 + e] = (r == 0 ? 0.f : acc[c * 16 + e]) + v[e];
            }
            if (c + 1 < HC && c + 1 < n_sl) {
              tmem_ld_wait(v + 16);
#pragma unroll
              for (int e = 0; e < 16; ++e) acc[(c + 1) * 16 + e] = (r == 0 ? 0.f : acc[(c + 1) * 16 + e]) + v[16 + e];
            }
          }
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(acce_u32[q & 1]);
        }
      } else {
        if (ok) ok = warp_mbar_wait(&accf[q & 1], static_cast<uint32_t>(q >> 1) & 1u, p.err, p.spin);
        __syncwarp();
        tc_fence_after();
      }
      if (!ok) s_timed_out = 1;

      // slices of token rows through shared memory: a warp then owns whole
      // rows (lane l: features 4l..4l+3), so stores are full lines and the
      // row's LayerNorm statistics over the 128 features are warp reductions
      auto slice = [&](int sl, const float *src) {
        // the two buffers alternate over all slices, whatever a tile's number
        // of them: a slice's barrier says that the one before has been read
        float *buf = buf0 + (n_written++ & 1) * kSlice * 128;
#pragma unroll
        for (int jj = 0; jj < kSlice; ++jj) buf[jj * 128 + feat] = src[jj];
        group_barrier(hg);
        if constexpr (EPI == EPI_HEAD) {
          const int j0 = quarter * kR, tl0 = sl * kSlice + j0;
          if (!ok || th + tl0 >= p.M || n0 >= p.N) return;
          float4 z4[kR];
          HeadRec r[kR];
#pragma unroll
          for (int k = 0; k < kR; ++k) z4[k] = *reinterpret_cast<const float4 *>(buf + (j0 + k) * 128 + 4 * lane);
          if (p.logits) {
#pragma unroll
            for (int k = 0; k < kR; ++k) {
              if (th + tl0 + k >= p.M) break;
              float *lrow = p.logits + static_cast<size_t>(th + tl0 + k) * p.N + n0;
#pragma unroll
              for (int i = 0; i < 4; ++i)
                if (n0 + i * 32 + lane < p.N) lrow[i * 32 + lane] = buf[(j0 + k) * 128 + i * 32 + lane];
            }
          }
          if (p.temperature > 0.f) head_rows_sample(p, z4, masked, n0 + 4 * lane, tk + tl0, r);
          else head_rows_greedy(z4, masked, n0 + 4 * lane, r);
#pragma unroll
          for (int k = 0; k < kR; ++k)
            if (lane == k && th + tl0 + k < p.M)
              p.recs[static_cast<size_t>(th + tl0 + k) * ((p.N + 127) / 128) + ntile] = r[k];
          return;
        }
        float4 cur[kR];
        if constexpr (EPI == EPI_RESID) {
#pragma unroll
          for (int k = 0; k < kR; ++k) cur[k] = old[k];
          if (sl + 1 < n_sl) load_old(sl + 1);
        }
#pragma unroll
        for (int k = 0; k < kR; ++k) {
          const int jr = quarter * kR + k, tl = sl * kSlice + jr, t = th + tl;
          const bool valid = ok && t < p.M && n0 < p.N;
          const float4 a4 = *reinterpret_cast<const float4 *>(buf + jr * 128 + 4 * lane);
          const float v[4] = {a4.x + b4[0], a4.y + b4[1], a4.z + b4[2], a4.w + b4[3]};
          float fin[4] = {v[0], v[1], v[2], v[3]};
          if constexpr (EPI == EPI_RESID) {
            fin[0] = cur[k].x + v[0];
            fin[1] = cur[k].y + v[1];
            fin[2] = cur[k].z + v[2];
            fin[3] = cur[k].w + v[3];
            if (valid) {
              *reinterpret_cast<float4 *>(p.resid + static_cast<size_t>(t) * p.ld_resid + n0 + 4 * lane) =
                  make_float4(fin[0], fin[1], fin[2], fin[3]);
              const uint2 h = pack4_bf16(fin);
              if (p.tap0) *reinterpret_cast<uint2 *>(p.tap0 + static_cast<size_t>(t) * p.ld_tap + n0 + 4 * lane) = h;
              if (p.tap1) *reinterpret_cast<uint2 *>(p.tap1 + static_cast<size_t>(t) * p.ld_tap + n0 + 4 * lane) = h;
            }
          } else if constexpr (EPI == EPI_KV) {
            if (valid) {
              if (kv_q) {
                *reinterpret_cast<uint2 *>(kv_q + static_cast<size_t>(t) * p.ld_out) = pack4_bf16(fin);
              } else if (kv_c) {
                const int2 at = tk[tl];
                if (at.y) *reinterpret_cast<uint2 *>(kv_c + static_cast<size_t>(at.x) * 64) = pack4_bf16(fin);
                else set_error(p.err, WF_DEV_ERR_CAPACITY);
              }
            }
          } else if (valid) {
            float w4[4] = {v[0], v[1], v[2], v[3]};
            epi_quad_out<EPI>(p, t, n0 + 4 * lane, w4, tk + tl, fin);
          }
          if (p.stats_out) {
            const float mean = warp_sum((fin[0] + fin[1]) + (fin[2] + fin[3])) * (1.0f / 128.f);
            const float d0 = fin[0] - mean, d1 = fin[1] - mean, d2 = fin[2] - mean, d3 = fin[3] - mean;
            const float m2 = warp_sum((d0 * d0 + d1 * d1) + (d2 * d2 + d3 * d3));
            if (lane == 0 && valid)
              p.stats_out[static_cast<size_t>(t) * stat_tiles + ntile] = make_float2(mean, m2);
          }
        }
      };
      if constexpr (HC > 0) {
#pragma unroll
        for (int c = 0; c < HC; ++c)
          if (c < n_sl) slice(c, acc + c * 16);
      } else {
        const uint32_t src = trow + (q & 1) * kWideAcc;
        for (int c = 0; c < n_sl; ++c) {
          float v[kSlice];
          tmem_ld<kSlice>(src + c * kSlice, v);
          if (c + 1 == n_sl) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive_cluster(acce_u32[q & 1]);
          }
          slice(c, v);
        }
        ++q;
      }
    }
  }
  __syncwarp();

  // After a timeout, copies either CTA requested may still be landing and
  // MMAs the even CTA issued may still be running: the even CTA waits for
  // both (bounded) before either leaves.  It makes up on its barriers for
  // k-steps that only one of the two requested.  Otherwise the producers saw
  // every stage read.
  __syncthreads();
  if (threadIdx.x == 0) {
    const uint32_t peer = dsmem_map(smem_u32(tmem_slot + 2), rank ^ 1);
    dsmem_st_u32(peer, static_cast<uint32_t>(s_timed_out));
    dsmem_st_u32(peer + 4, static_cast<uint32_t>(issued));
  }
  __syncwarp();
  tc_fence_before();
  cluster_sync();
  if (s_timed_out | static_cast<int>(s_peer[0])) {
    if (rank == 0 && threadIdx.x == 0) {
      const int theirs = static_cast<int>(s_peer[1]), last = max(issued, theirs);
      for (int g = max(0, last - stages); g < last; ++g) {
        const int s = g % stages;
        if (g >= issued) mbar_arrive_expect_tx(&full[s], stage_bytes);
        else if (g >= theirs) mbar_complete_tx(&full[s], stage_bytes);
        mbar_drain(&full[s], static_cast<uint32_t>(g / stages) & 1u);
      }
      mbar_drain(done, 0u);
    }
    __syncwarp();
    cluster_sync();
  }
  if (warp == 2) tmem_dealloc_pair(tmem, kWideTmem);
}

// --------------------------------------------------------------- host ----
template <int EPI, int HC>
static cudaError_t wide_attr() {
  const void *f = reinterpret_cast<const void *>(gemm_wide_kernel<EPI, HC>);
  cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  return e == cudaSuccess ? prefer_max_shared(f) : e;
}

static cudaError_t gemm_wide_init() {
  static cudaError_t status = cudaErrorNotReady;
  static std::once_flag once;
  std::call_once(once, [] {
    status = wide_attr<EPI_F32, 4>();
    if (status == cudaSuccess) status = wide_attr<EPI_BF16, 4>();
    if (status == cudaSuccess) status = wide_attr<EPI_GELU, 4>();
    if (status == cudaSuccess) status = wide_attr<EPI_RESID, 4>();
    if (status == cudaSuccess) status = wide_attr<EPI_KV, 4>();
    if (status == cudaSuccess) status = wide_attr<EPI_KV, 0>();
    if (status == cudaSuccess) status = wide_attr<EPI_F32, 0>();
    if (status == cudaSuccess) status = wide_attr<EPI_HEAD, 0>();
  });
  return status;
}

// Token tile, ring depth and grid of a launch; false if the kernel does not
// take the shape.
static bool gemm_wide_plan(GemmParams &p, size_t *smem, int *pairs) {
  if (p.M <= 0 || p.N <= 0 || p.K <= 0 || p.K % 64) return false;
  if (p.splits < 1 || p.epi == EPI_HEAD) p.splits = 1;
  const int k_iters = p.K / 64;
  if (k_iters % p.splits) return false;
  p.kps = k_iters / p.splits;
  static const int n_sm = [] {
    int dev = 0, n = 0;
    if (cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
      return 0;
    return n;
  }();
  if (n_sm < 2) return false;
  const bool direct = p.splits == 1 && (p.epi == EPI_KV || p.epi == EPI_F32 || p.epi == EPI_HEAD);
  const int max_bt = direct ? 256 : 128, n_nt = (p.N + 255) / 256, slots = n_sm / 2;
  // The token tile with the least estimated time: per tile the larger of its
  // MMAs and its operand fetch over the k-steps plus an epilogue that grows with
  // the tile, times the tiles of the busiest pair.  The estimate only ranks the
  // tiles of one shape (the choice is better than any single tile, see above): it
  // leaves out what they share, takes 64 bytes per cycle and SM where an
  // unhindered copy loop reaches ~90, and one epilogue for all kinds.
  long long best = 0;
  p.BT = 0;
  for (int bt = 32; bt <= max_bt; bt += 32) {
    const int n_tt = (p.M + bt - 1) / bt;
    const long long tiles = static_cast<long long>(n_tt) * n_nt;
    const long long waves = (tiles + slots - 1) / slots;
    const long long fetch = (128 + bt / 2) * 2, mma = 2 * bt;
    const long long steps = k_iters * (fetch > mma ? fetch : mma);
    // (a head's epilogue of a tile runs under the next tile's MMAs)
    const long long head = (p.temperature > 0.f ? 70 : 20) * bt;
    const long long cost = p.epi == EPI_HEAD ? waves * (steps > head ? steps : head) + head : waves * (steps + 12 * bt);
    if (p.BT == 0 || cost < best) {
      best = cost;
      p.BT = bt;
      p.n_tt = n_tt;
    }
  }
  if (p.BT == 0) return false;
  p.n_ptiles = p.n_tt * n_nt;
  *pairs = p.n_ptiles < slots ? p.n_ptiles : slots;
  const size_t stage = kWideA + static_cast<size_t>(p.BT) * kWideBK;
  int st = static_cast<int>((227 * 1024 - kWideFixed) / stage);
  if (st > kWideMaxStages) st = kWideMaxStages;
  p.stages = st;
  *smem = kWideFixed + st * stage;
  return st >= 2;
}

template <int EPI, int HC>
static cudaError_t wide_launch(const CUtensorMap *tw, const CUtensorMap *tx, const GemmParams &p, size_t smem,
                               int pairs, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(kWideThreads<EPI>);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemm_wide_kernel<EPI, HC>, *tw, *tx, p);
}

cudaError_t launch_gemm_wide(const void *X, const void *W, GemmParams p, cudaStream_t s, bool pdl) {
  size_t smem = 0;
  int pairs = 0;
  cudaError_t e = gemm_wide_init();
  if (e != cudaSuccess) return e;
  if (!X || !gemm_wide_plan(p, &smem, &pairs)) return cudaErrorInvalidValue;
  const CUtensorMap *tw = tmap_bf16_2d(W, p.N, p.K, 128);
  const CUtensorMap *tx = tmap_bf16_2d(X, p.M, p.K, p.BT / 2);
  if (!tw || !tx) return cudaErrorInvalidValue;
  const bool direct = p.splits == 1;
  switch (p.epi) {
    case EPI_F32:
      return direct ? wide_launch<EPI_F32, 0>(tw, tx, p, smem, pairs, s, pdl)
                    : wide_launch<EPI_F32, 4>(tw, tx, p, smem, pairs, s, pdl);
    case EPI_BF16: return wide_launch<EPI_BF16, 4>(tw, tx, p, smem, pairs, s, pdl);
    case EPI_GELU: return wide_launch<EPI_GELU, 4>(tw, tx, p, smem, pairs, s, pdl);
    case EPI_RESID: return wide_launch<EPI_RESID, 4>(tw, tx, p, smem, pairs, s, pdl);
    case EPI_KV:
      return direct ? wide_launch<EPI_KV, 0>(tw, tx, p, smem, pairs, s, pdl)
                    : wide_launch<EPI_KV, 4>(tw, tx, p, smem, pairs, s, pdl);
    case EPI_HEAD: return wide_launch<EPI_HEAD, 0>(tw, tx, p, smem, pairs, s, pdl);
  }
  return cudaErrorInvalidValue;
}

}  // namespace wf
