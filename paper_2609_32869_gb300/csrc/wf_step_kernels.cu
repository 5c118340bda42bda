// Row-wise kernels of the decode step: block embeddings (Eq. 2 for the
// drafter; token + learned position for the target), LayerNorm, the
// cross-tile reduction of the output head, the per-sequence accept/rollback
// rule (Sec. 3.1, App. A.1, A.4) and per-slot state bookkeeping.
#include <mutex>

#include "wf_device.cuh"
#include "wf_internal.h"

namespace wf {

static cudaError_t launch_ex(const void *fn, dim3 grid, dim3 block, void **args, cudaStream_t s,
                             bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelExC(&cfg, fn, args);
}

// ------------------------------------------------------------ embedding --
// Target rows: x = Emb(tok) + PosEmb(L + j).  Drafter rows (Eq. 2): row 0 is
// Emb(anchor), rows 1..K are the mask vector m; no position embedding (the
// drafter marks positions with RoPE).
__global__ void embed_kernel(const EmbedParams p) {
  pdl_wait();
  pdl_launch_dependents();
  const int r = blockIdx.x;
  const int i = r / p.rps, j = r - i * p.rps;
  const int slot = p.seq_slot[i];
  int tok = -1;
  if (p.src == TOK_PROMPT) {
    tok = p.prompt[i * p.P + j];
  } else if (j == 0) {
    tok = p.anchor[slot];
  } else if (!p.drafter) {
    const int src = p.forced ? p.forced[slot * p.K + j - 1] : p.cand_in[slot * p.K + j - 1];
    tok = src;
    if (threadIdx.x == 0) p.cand_out[slot * p.K + j - 1] = src;
  }
  const bool use_mask = p.drafter && j > 0;
  if (!use_mask && (tok < 0 || tok >= p.vocab)) {
    if (threadIdx.x == 0) set_error(p.err, WF_DEV_ERR_TOKEN);
    tok = tok < 0 ? 0 : p.vocab - 1;
  }
  const int pos = (p.drafter || !p.L) ? 0 : ((p.src == TOK_PROMPT ? 0 : p.L[slot]) + j);
  float *x = p.x + static_cast<size_t>(r) * p.d;
  // thread tid holds feature 128k + tid of every 128-feature tile k
  const int tiles = p.d >> 7;
  // every load before the first store: the row's latencies overlap (11 us a
  // launch when each tile's stores stood between its loads and the next's)
  float v[kMaxStatTiles];
  bf16 emb[kMaxStatTiles], pe[kMaxStatTiles], gn[kMaxStatTiles], bn[kMaxStatTiles];
  const bf16 *src = use_mask ? p.mask_emb : p.tok_emb + static_cast<size_t>(tok) * p.d;
  const bf16 *psrc = use_mask || p.drafter ? nullptr : p.pos_emb + static_cast<size_t>(pos) * p.d;
#pragma unroll
  for (int k = 0; k < kMaxStatTiles; ++k) {
    if (k >= tiles) continue;
    const int e = k * 128 + threadIdx.x;
    emb[k] = src[e];
    if (psrc) pe[k] = psrc[e];
    if (p.xg) gn[k] = p.g_next[e];
    if (p.xg && r == 0) bn[k] = p.b_next[e];
  }
#pragma unroll
  for (int k = 0; k < kMaxStatTiles; ++k) {
    if (k >= tiles) continue;
    const int e = k * 128 + threadIdx.x;
    float val = bf2f(emb[k]);
    if (psrc) val += bf2f(pe[k]);
    v[k] = val;
    x[e] = val;
    if (p.xg) {
      p.xg[static_cast<size_t>(r + 2) * p.d + e] = __float2bfloat16(val * bf2f(gn[k]));
      if (r == 0) {
        p.xg[e] = gn[k];
        p.xg[static_cast<size_t>(p.d) + e] = bn[k];
      }
    }
  }
  if (p.part_out) {  // the whole row's (sum x, sum x^2), summed in a fixed order
    __shared__ float red2[4][2];
    float s1 = 0.f, s2 = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxStatTiles; ++k)
      if (k < tiles) {
        s1 += v[k];
        s2 = __fmaf_rn(v[k], v[k], s2);
      }
    s1 = warp_sum(s1);
    s2 = warp_sum(s2);
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
      red2[w][0] = s1;
      red2[w][1] = s2;
    }
    __syncthreads();
    if (threadIdx.x == 0)
      p.part_out[static_cast<size_t>(r) * p.part_stride] =
          make_float2((red2[0][0] + red2[1][0]) + (red2[2][0] + red2[3][0]),
                      (red2[0][1] + red2[1][1]) + (red2[2][1] + red2[3][1]));
  }
  if (!p.stats_out) return;
  // per-tile (mean, M2) of the row for the next LayerNorm
  __shared__ float red[4][kMaxStatTiles];
  __shared__ float mean_s[kMaxStatTiles];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kMaxStatTiles; ++k) {
    if (k >= tiles) continue;
    const float sum = warp_sum(v[k]);
    if (lane == 0) red[warp][k] = sum;
  }
  __syncthreads();
  if (threadIdx.x < tiles) {
    const int k = threadIdx.x;
    mean_s[k] = ((red[0][k] + red[1][k]) + (red[2][k] + red[3][k])) * (1.0f / 128.f);
  }
  __syncthreads();
#pragma unroll
  for (int k = 0; k < kMaxStatTiles; ++k) {
    if (k >= tiles) continue;
    const float dv = v[k] - mean_s[k];
    const float sq = warp_sum(dv * dv);
    if (lane == 0) red[warp][k] = sq;
  }
  __syncthreads();
  if (threadIdx.x < tiles) {
    const int k = threadIdx.x;
    p.stats_out[static_cast<size_t>(r) * tiles + k] =
        make_float2(mean_s[k], (red[0][k] + red[1][k]) + (red[2][k] + red[3][k]));
  }
}

cudaError_t launch_embed(const EmbedParams &p0, cudaStream_t s, bool pdl) {
  EmbedParams p = p0;
  void *args[] = {&p};
  return launch_ex(reinterpret_cast<const void *>(embed_kernel), dim3(p.n_seq * p.rps), dim3(128),
                   args, s, pdl);
}

// ------------------------------------------------------------ LayerNorm --
// One warp per row; lane l owns the float4 chunks l, l+32, ... of the row.
// The row's statistics come from the kernel that wrote it (per 128-feature
// tile, merged in tile order), so this kernel and the GEMMs that normalise
// their own token operand produce identical bits.  Every load is issued
// before any arithmetic so the latencies overlap.
__global__ void __launch_bounds__(128) layernorm_kernel(const float *__restrict__ x,
                                                        const float2 *__restrict__ stats,
                                                        int in_stride, int in_off,
                                                        const bf16 *__restrict__ g,
                                                        const bf16 *__restrict__ b,
                                                        bf16 *__restrict__ y, int rows, int d,
                                                        float eps) {
  pdl_wait();
  pdl_launch_dependents();
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int lane = threadIdx.x & 31;
  if (warp >= rows) return;
  const size_t row = static_cast<size_t>(warp) * in_stride + in_off;
  const float4 *xr = reinterpret_cast<const float4 *>(x + row * d);
  const uint2 *gr = reinterpret_cast<const uint2 *>(g);
  const uint2 *br = reinterpret_cast<const uint2 *>(b);
  const int chunks = d >> 7;
  float4 v[kMaxStatTiles];
  uint2 gv[kMaxStatTiles], bv[kMaxStatTiles];
#pragma unroll
  for (int k = 0; k < kMaxStatTiles; ++k) {
    if (k < chunks) {
      v[k] = xr[k * 32 + lane];
      gv[k] = gr[k * 32 + lane];
      bv[k] = br[k * 32 + lane];
    }
  }
  float2 ms;
  if (stats) {
    ms = merge_tile_stats(stats + row * chunks, chunks, eps);
  } else {  // the row's own mean and variance (two passes over the registers)
    float sum = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxStatTiles; ++k)
      if (k < chunks) sum += (v[k].x + v[k].y) + (v[k].z + v[k].w);
    const float mean = warp_sum(sum) / static_cast<float>(d);
    float q = 0.f;
#pragma unroll
    for (int k = 0; k < kMaxStatTiles; ++k) {
      if (k < chunks) {
        const float a = v[k].x - mean, b = v[k].y - mean, c = v[k].z - mean, e = v[k].w - mean;
        q += (a * a + b * b) + (c * c + e * e);
      }
    }
    ms = make_float2(mean, rsqrtf(warp_sum(q) / static_cast<float>(d) + eps));
  }
  uint2 *yr = reinterpret_cast<uint2 *>(y + static_cast<size_t>(warp) * d);
#pragma unroll
  for (int k = 0; k < kMaxStatTiles; ++k) {
    if (k < chunks) {
      const __nv_bfloat162 g01 = *reinterpret_cast<const __nv_bfloat162 *>(&gv[k].x);
      const __nv_bfloat162 g23 = *reinterpret_cast<const __nv_bfloat162 *>(&gv[k].y);
      const __nv_bfloat162 b01 = *reinterpret_cast<const __nv_bfloat162 *>(&bv[k].x);
      const __nv_bfloat162 b23 = *reinterpret_cast<const __nv_bfloat162 *>(&bv[k].y);
      const __nv_bfloat162 o01 =
          __floats2bfloat162_rn(ln_apply(v[k].x, ms, __low2float(g01), __low2float(b01)),
                                ln_apply(v[k].y, ms, __high2float(g01), __high2float(b01)));
      const __nv_bfloat162 o23 =
          __floats2bfloat162_rn(ln_apply(v[k].z, ms, __low2float(g23), __low2float(b23)),
                                ln_apply(v[k].w, ms, __high2float(g23), __high2float(b23)));
      uint2 o;
      o.x = *reinterpret_cast<const uint32_t *>(&o01);
      o.y = *reinterpret_cast<const uint32_t *>(&o23);
      yr[k * 32 + lane] = o;
    }
  }
}

cudaError_t launch_layernorm(const float *x, const float2 *stats, int in_stride, int in_off,
                             const bf16 *g, const bf16 *b, bf16 *y, int rows, int d, float eps,
                             cudaStream_t s, bool pdl) {
  if (d % 128 || d / 128 > kMaxStatTiles) return cudaErrorInvalidValue;
  void *args[] = {&x, &stats, &in_stride, &in_off, &g, &b, &y, &rows, &d, &eps};
  const int threads = 128;
  const int blocks = (rows * 32 + threads - 1) / threads;
  return launch_ex(reinterpret_cast<const void *>(layernorm_kernel), dim3(blocks), dim3(threads),
                   args, s, pdl);
}

// ---------------------------------------------------------- head reduce --
// Combine the per-tile records of each row: argmax (or Gumbel-max draw) with
// the lowest id on ties, and when sampling the log-sum-exp.  One CTA per row,
// every record of a thread in flight at once (a warp per row that folded its
// records one by one took 14 us, all of it load latency).  The order of the
// sum depends on the vocabulary only.
constexpr int kRedThreads = 128;
constexpr int kRedUnroll = 4;  // records per thread and round: 512 tiles, 65536 ids
__global__ void __launch_bounds__(kRedThreads) head_reduce_kernel(const HeadReduceParams p) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ float s_best[kRedThreads / 32], s_m[kRedThreads / 32], s_s[kRedThreads / 32];
  __shared__ int s_id[kRedThreads / 32];
  const int row = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const HeadRec *rr = p.recs + static_cast<size_t>(row) * p.n_tiles;
  float best = -INFINITY, m = -INFINITY, sum = 0.f;
  int id = 0x7fffffff;
  for (int t0 = tid; t0 < p.n_tiles; t0 += kRedThreads * kRedUnroll) {
    float rm[kRedUnroll], rs[kRedUnroll], rg[kRedUnroll];
    int ri[kRedUnroll];
#pragma unroll
    for (int i = 0; i < kRedUnroll; ++i) {
      const int t = t0 + i * kRedThreads;
      rm[i] = rg[i] = -INFINITY;
      rs[i] = 0.f;
      ri[i] = 0x7fffffff;
      if (t < p.n_tiles) {
        rm[i] = rr[t].m;
        rs[i] = rr[t].s;
        rg[i] = p.sampling ? rr[t].gm : rm[i];
        ri[i] = p.sampling ? rr[t].garg : rr[t].arg;
      }
    }
#pragma unroll
    for (int i = 0; i < kRedUnroll; ++i) {
      if (rg[i] > best || (rg[i] == best && ri[i] < id)) {
        best = rg[i];
        id = ri[i];
      }
      if (p.sampling) {
        const float M = fmaxf(m, rm[i]);
        if (M != -INFINITY)
          sum = (m == -INFINITY ? 0.f : sum * __expf(m - M)) + (rm[i] == -INFINITY ? 0.f : rs[i] * __expf(rm[i] - M));
        m = M;
      }
    }
  }
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float b2 = __shfl_xor_sync(0xffffffffu, best, off);
    const int i2 = __shfl_xor_sync(0xffffffffu, id, off);
    if (b2 > best || (b2 == best && i2 < id)) {
      best = b2;
      id = i2;
    }
  }
  if (p.sampling) {
    const float M = key_value(__reduce_max_sync(0xffffffffu, order_key(m)));
    sum = warp_sum(m == -INFINITY ? 0.f : sum * __expf(m - M));
    m = M;
  }
  if (lane == 0) {
    s_best[warp] = best;
    s_id[warp] = id;
    s_m[warp] = m;
    s_s[warp] = sum;
  }
  __syncthreads();
  if (tid == 0) {
    float M = -INFINITY, S = 0.f;
    for (int w = 0; w < kRedThreads / 32; ++w) {
      if (w > 0 && (s_best[w] > best || (s_best[w] == best && s_id[w] < id))) {
        best = s_best[w];
        id = s_id[w];
      }
      M = fmaxf(M, s_m[w]);
    }
    for (int w = 0; w < kRedThreads / 32; ++w) S += s_m[w] == -INFINITY ? 0.f : s_s[w] * __expf(s_m[w] - M);
    HeadOut out;
    out.arg = out.garg = id;  // the one its reader asks for (greedy or sampling)
    out.m = p.sampling ? M : best;
    out.lse = p.sampling ? M + logf(S) : 0.f;
    p.out[row] = out;
    if (p.cand) {
      const int i = row / p.rps, j = row - i * p.rps;
      if (j >= 1 && j <= p.K) p.cand[p.seq_slot[i] * p.K + j - 1] = id;
    }
  }
}

cudaError_t launch_head_reduce(const HeadReduceParams &p0, cudaStream_t s, bool pdl) {
  HeadReduceParams p = p0;
  void *args[] = {&p};
  return launch_ex(reinterpret_cast<const void *>(head_reduce_kernel), dim3(p.rows), dim3(kRedThreads), args, s, pdl);
}

// --------------------------------------------------------------- accept --
// One CTA per active sequence (greedy) or a cluster of kAccCluster (sampling).  Greedy (Sec. 3.1): keep proposals while they
// equal the target's argmax, then emit the target's token (correction, or
// bonus after K agreements).  Sampling (Sec. 3.1, App. A.4): accept c_i when
// u_i < p_i(c_i)/q_i(c_i) in FP32; at the first rejection draw from the
// normalised residual (p_i - q_i)_+ by Gumbel-max; after a full block emit
// the bonus drawn from the target.  An accepted EOS ends the transcript
// without a bonus; with R tokens left at most R-1 proposals are live; the
// cache keeps L+1+a positions (App. A.1).  One thread per proposal forms its
// decision and one reads them in order; the residual draw splits the
// vocabulary over the cluster, and each CTA takes one of the normalisers of
// forced proposal distributions.  The draw is bound by its arithmetic: one CTA
// that scored every id (three logarithms and a Philox block each) took 250 us
// at 51866 ids.  Here a Philox block serves its four ids, and a warp ranks them
// by the exponential race r / -log u (r the residual, exactly as scored) and
// scores only ids within kRaceTol of its best so far, so the draw is the exact
// scores' argmax: 26 us at 32 sequences.
constexpr int kAccThreads = 256;
constexpr int kAccCluster = 8;

// The CTA's maximum (value, lowest id on ties) of (v, arg) over its threads.
__device__ __forceinline__ void block_argmax(float &v, int &arg, float *sv, int *sa) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float v2 = __shfl_xor_sync(0xffffffffu, v, off);
    const int a2 = __shfl_xor_sync(0xffffffffu, arg, off);
    if (v2 > v || (v2 == v && a2 < arg)) {
      v = v2;
      arg = a2;
    }
  }
  __syncthreads();
  if (lane == 0) {
    sv[warp] = v;
    sa[warp] = arg;
  }
  __syncthreads();
  v = sv[0];
  arg = sa[0];
  for (int w = 1; w < kAccThreads / 32; ++w)
    if (sv[w] > v || (sv[w] == v && sa[w] < arg)) {
      v = sv[w];
      arg = sa[w];
    }
}
// log sum exp over the CTA of per-thread (max, sum of exp(x - max)).
__device__ __forceinline__ float block_lse(float m, float sum, float *sm, float *ss) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) {
    const float m2 = __shfl_xor_sync(0xffffffffu, m, off);
    const float s2 = __shfl_xor_sync(0xffffffffu, sum, off);
    const float M = fmaxf(m, m2);
    sum = (M == -INFINITY) ? 0.f : sum * expf(m - M) + s2 * expf(m2 - M);
    m = M;
  }
  __syncthreads();
  if (lane == 0) {
    sm[warp] = m;
    ss[warp] = sum;
  }
  __syncthreads();
  float M = -INFINITY, S = 0.f;
  for (int w = 0; w < kAccThreads / 32; ++w) {
    const float M2 = fmaxf(M, sm[w]);
    S = (M2 == -INFINITY) ? 0.f : S * expf(M - M2) + ss[w] * expf(sm[w] - M2);
    M = M2;
  }
  return M + logf(S);
}

template <int C>  // CTAs per sequence
__global__ void __launch_bounds__(kAccThreads) accept_kernel(const AcceptParams p) {
  pdl_wait();
  pdl_launch_dependents();
  __shared__ float s_v[kAccThreads / 32], s_w[kAccThreads / 32];
  __shared__ int s_a[kAccThreads / 32];
  __shared__ float s_qlse[8];
  __shared__ int s_em[16], s_cand[8], s_acc[8];
  __shared__ int s_state[4];  // emitted count, accepted a, stopped, rejected row (0: none)
  __shared__ float s_cv[C];   // the cluster's best scores and their ids (-1: nothing to draw from)
  __shared__ int s_ca[C];
  const int Kp1 = p.K + 1;
  const int tid = threadIdx.x;
  const int rank = C > 1 ? static_cast<int>(blockIdx.x % C) : 0, i = blockIdx.x / C, n_ctas = gridDim.x / C;
  // slots outside the active list emit nothing this step
  if (rank == 0) {
    for (int sl = i; sl < p.max_batch; sl += n_ctas) {
      bool mine = false;
      for (int q = tid; q < p.n_seq; q += kAccThreads) mine = mine || p.seq_slot[q] == sl;
      if (!__syncthreads_or(mine)) {
        for (int j = tid; j < Kp1; j += kAccThreads) p.out_tokens[sl * Kp1 + j] = -1;
        if (tid == 0) p.out_count[sl] = 0;
      }
    }
  }
  if (i >= p.n_seq) return;
  const int slot = p.seq_slot[i];
  const int finished_before = p.done[slot], R = p.remaining[slot], step = p.step[slot], L0 = p.L[slot];
  if (C > 1) cluster_sync();  // every CTA has read the state that CTA 0 rewrites
  if (finished_before) {
    if (rank == 0) {
      for (int j = tid; j < Kp1; j += kAccThreads) p.out_tokens[slot * Kp1 + j] = -1;
      if (tid == 0) p.out_count[slot] = 0;
    }
    return;
  }
  const bool sampling = p.temperature > 0.f;
  int k = p.greedy_step ? 0 : min(p.K, R - 1);
  if (k < 0) k = 0;
  const int r0 = i * p.rps;
  const float *fq = p.forced_q ? p.forced_q + static_cast<size_t>(slot) * p.K * p.vocab : nullptr;
  // normalisers of the forced proposal distributions softmax(q / T)
  if (sampling && fq) {
    for (int c = rank; c < k; c += C) {
      const float *row = fq + static_cast<size_t>(c) * p.vocab;
      float m = -INFINITY, sum = 0.f;
      for (int v = tid; v < p.vocab; v += kAccThreads) {
        if (p.suppress && p.suppress[v]) continue;
        const float x = __fdiv_rn(row[v], p.temperature);
        if (x > m) {
          sum = sum * expf(m - x) + 1.f;
          m = x;
        } else {
          sum += expf(x - m);
        }
      }
      const float l = block_lse(m, sum, s_v, s_w);
      if (tid < C) {
        if (C > 1) dsmem_st_u32(dsmem_map(smem_u32(&s_qlse[c]), tid), __float_as_uint(l));
        else s_qlse[c] = l;
      }
    }
    if (C > 1) cluster_sync();
    else __syncthreads();
  }
  // proposal c = tid + 1: accepted?
  if (tid < k) {
    const int c = tid + 1, cand = p.cand[slot * p.K + tid];
    bool acc;
    if (!sampling) {
      acc = cand == p.tout[r0 + tid].arg;
    } else if (cand < 0 || cand >= p.vocab) {
      // no such id (the embedding has recorded it): probability 0, so rejected.
      // All proposals are looked at together, also those behind a rejection.
      acc = false;
    } else {
      const int rt = r0 + c - 1, rd = r0 + c;  // drafter row c holds mask position c
      const float lse_t = p.tout[rt].lse;
      const float lse_d = fq ? s_qlse[c - 1] : p.dout[rd].lse;
      const float zd = fq ? fq[static_cast<size_t>(c - 1) * p.vocab + cand]
                          : p.dlogits[static_cast<size_t>(rd) * p.vocab + cand];
      const float xt = __fdiv_rn(p.tlogits[static_cast<size_t>(rt) * p.vocab + cand], p.temperature);
      const float xd = __fdiv_rn(zd, p.temperature);
      const bool sup = p.suppress && p.suppress[cand];
      const float pc = sup ? 0.f : expf(xt - lse_t);
      const float qc = sup ? 0.f : expf(xd - lse_d);
      Philox4 o = philox4x32_10(0, c, step, (kTagAccept << 24) | (slot & 0xFFFFFF),
                                static_cast<uint32_t>(p.seed), static_cast<uint32_t>(p.seed >> 32));
      const float u = word_to_uniform(o.x[0]);
      acc = u < __fdiv_rn(pc, qc);
    }
    s_cand[tid] = cand;
    s_acc[tid] = acc;
  }
  __syncthreads();
  if (tid == 0) {
    int n_em = 0, a = 0, stop = 0, rej = 0;
    bool finished = false;
    for (int c = 1; c <= k; ++c) {
      if (!s_acc[c - 1]) {
        if (sampling) {  // the residual draw below supplies the token
          rej = c;
          finished = true;
        }
        break;
      }
      s_em[n_em++] = s_cand[c - 1];
      a = c;
      if (s_cand[c - 1] == p.eos) {
        stop = 1;
        finished = true;
        break;
      }
    }
    if (!finished) {  // correction (greedy mismatch) or bonus
      const HeadOut &ho = p.tout[r0 + a];
      const int t = sampling ? ho.garg : ho.arg;
      s_em[n_em++] = t;
      stop = t == p.eos;
    }
    s_state[0] = n_em;
    s_state[1] = a;
    s_state[2] = stop;
    s_state[3] = rej;
  }
  __syncthreads();
  const int rej = s_state[3];
  if (rej) {
    // residual (p - q)_+ of row rej by Gumbel-max over log r; if it is empty
    // (rounding only) the token is drawn from the target itself
    const int rt = r0 + rej - 1, rd = r0 + rej;
    const float *xt = p.tlogits + static_cast<size_t>(rt) * p.vocab;
    const float *xd = fq ? fq + static_cast<size_t>(rej - 1) * p.vocab
                         : p.dlogits + static_cast<size_t>(rd) * p.vocab;
    const float lse_t = p.tout[rt].lse;
    const float lse_d = fq ? s_qlse[rej - 1] : p.dout[rd].lse;
    // this CTA's ids: whole groups of four (one Philox block each)
    const int groups = (p.vocab + 3) / 4;
    const int g0 = static_cast<int>(static_cast<long long>(groups) * rank / C);
    const int g1 = static_cast<int>(static_cast<long long>(groups) * (rank + 1) / C);
    const int warp = tid >> 5, lane = tid & 31;
    float best = -INFINITY;
    int barg = 0x7fffffff;
    // pass 0: the residual; pass 1 (if no CTA found any residual): the target
    for (int pass = 0; pass < 2; ++pass) {
      bool any = false;
      float wbest = 0.f;  // the warp's best r / w so far
      for (int gb = g0 + warp * 32; gb < g1; gb += kAccThreads) {
        const int gq = gb + lane;
        float rr[4], uu[4], est[4], top = 0.f;
        const Philox4 o = philox4x32_10(static_cast<uint32_t>(gq), static_cast<uint32_t>(rej),
                                        static_cast<uint32_t>(step), (kTagResidual << 24) | (slot & 0xFFFFFF),
                                        static_cast<uint32_t>(p.seed), static_cast<uint32_t>(p.seed >> 32));
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const int v = 4 * gq + e;
          const bool live = gq < g1 && v < p.vocab && !(p.suppress && p.suppress[v]);
          float r = live ? 1.f : 0.f;
          if (live && pass == 0) {
            const float pt = expf(__fdiv_rn(xt[v], p.temperature) - lse_t);
            const float qd = expf(__fdiv_rn(xd[v], p.temperature) - lse_d);
            r = fmaxf(pt - qd, 0.f);
          }
          rr[e] = r;
          uu[e] = word_to_open_uniform(o.x[e]);
          est[e] = __fdividef(r, neg_log2_estimate(uu[e]));
          top = fmaxf(top, est[e]);
        }
        wbest = fmaxf(wbest, __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(top))));
        // (the screen needs scores in the normal range; pass 1 scores all)
        const float floor = pass == 0 && wbest > 1e-30f ? wbest - wbest * kRaceTol : 0.f;
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          if (!(rr[e] > 0.f)) continue;
          any = true;
          if (est[e] < floor) continue;
          const int v = 4 * gq + e;
          const float x = pass == 0 ? logf(rr[e]) : __fdiv_rn(xt[v], p.temperature);
          const float sc = x + -logf(-logf(uu[e]));
          if (sc > best || (sc == best && v < barg)) {
            best = sc;
            barg = v;
          }
        }
      }
      any = __syncthreads_or(any);
      block_argmax(best, barg, s_v, s_a);
      if (C == 1) {
        if (any) break;
        continue;
      }
      // every CTA learns every CTA's best
      if (tid < C) {
        dsmem_st_u32(dsmem_map(smem_u32(&s_cv[rank]), tid), __float_as_uint(best));
        dsmem_st_u32(dsmem_map(smem_u32(&s_ca[rank]), tid), any ? static_cast<uint32_t>(barg) : 0xffffffffu);
      }
      cluster_sync();
      bool found = false;
      best = -INFINITY;
      barg = 0x7fffffff;
      for (int q = 0; q < C; ++q) {
        if (s_ca[q] < 0) continue;
        found = true;
        if (s_cv[q] > best || (s_cv[q] == best && s_ca[q] < barg)) {
          best = s_cv[q];
          barg = s_ca[q];
        }
      }
      if (found) break;
      cluster_sync();  // the exchange is read before the second pass rewrites it
    }
    if (tid == 0) {
      s_em[s_state[0]++] = barg;
      s_state[2] = barg == p.eos;
    }
  }
  if (rank != 0) return;
  __syncthreads();
  const int n_em = s_state[0], a = s_state[1];
  for (int j = tid; j < Kp1; j += kAccThreads) p.out_tokens[slot * Kp1 + j] = j < n_em ? s_em[j] : -1;
  if (tid == 0) {
    p.out_count[slot] = n_em;
    const int newL = L0 + 1 + a;
    p.L[slot] = newL;
    p.anchor[slot] = s_em[n_em - 1];
    const int left = R - n_em;
    p.remaining[slot] = left;
    p.step[slot] = step + 1;
    bool done = s_state[2] || left <= 0;
    if (!done && newL + Kp1 > p.max_ctx) {
      set_error(p.err, WF_DEV_ERR_CAPACITY);
      done = true;
    }
    p.done[slot] = done ? 1 : 0;
  }
}

cudaError_t launch_accept(const AcceptParams &p0, cudaStream_t s, bool pdl) {
  AcceptParams p = p0;
  if (p.K > 8) return cudaErrorInvalidValue;
  const int n = p.n_seq > 0 ? p.n_seq : 1;
  if (!(p.temperature > 0.f) || p.greedy_step) {
    void *args[] = {&p};
    return launch_ex(reinterpret_cast<const void *>(accept_kernel<1>), dim3(n), dim3(kAccThreads), args, s, pdl);
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n * kAccCluster);
  cfg.blockDim = dim3(kAccThreads);
  cfg.stream = s;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kAccCluster;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, accept_kernel<kAccCluster>, p);
}

// ---------------------------------------------------------------- state --
__global__ void state_kernel(const StateParams p) {
  pdl_wait();
  pdl_launch_dependents();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= p.n) return;
  const int slot = p.slots[i];
  if (slot < 0 || slot >= p.max_batch) return;
  if (p.op == 0) {  // begin prefill: empty cache, step 0
    p.L[slot] = 0;
    p.step[slot] = 0;
    p.done[slot] = 0;
  } else if (p.op == 1) {  // finish prefill: the first token becomes the anchor
    const HeadOut &ho = p.hout[i];
    const int first = p.sampling ? ho.garg : ho.arg;
    const int left = p.budget[i] - 1;
    p.L[slot] = p.P;
    p.anchor[slot] = first;
    p.remaining[slot] = left;
    p.step[slot] = 1;
    p.done[slot] = (first == p.eos || left <= 0) ? 1 : 0;
    p.snap_L[slot] = p.P;
    p.snap_anchor[slot] = first;
    p.snap_remaining[slot] = left;
    if (p.first) p.first[i] = first;
    p.active[p.active_offset + i] = slot;
    if (i == 0) *p.n_active_dev = p.active_offset + p.n;
  } else if (p.op == 2) {  // rewind to the post-prefill snapshot
    p.L[slot] = p.snap_L[slot];
    p.anchor[slot] = p.snap_anchor[slot];
    p.remaining[slot] = p.snap_remaining[slot];
    p.step[slot] = 1;
    p.done[slot] = (p.snap_remaining[slot] <= 0) ? 1 : 0;
  }
}

cudaError_t launch_state(const StateParams &p0, cudaStream_t s, bool pdl) {
  StateParams p = p0;
  void *args[] = {&p};
  return launch_ex(reinterpret_cast<const void *>(state_kernel), dim3((p.n + 127) / 128), dim3(128),
                   args, s, pdl);
}

// Active list = slots whose done flag is clear, ascending.
__global__ void compact_kernel(const int32_t *done, int max_batch, int32_t *active,
                               int32_t *n_active) {
  if (threadIdx.x == 0) {
    int c = 0;
    for (int s = 0; s < max_batch; ++s)
      if (!done[s]) active[c++] = s;
    *n_active = c;
  }
}

cudaError_t step_kernels_init() {
  static cudaError_t status = cudaErrorNotReady;
  static std::once_flag once;
  std::call_once(once, [] {
    const void *fns[] = {reinterpret_cast<const void *>(embed_kernel), reinterpret_cast<const void *>(layernorm_kernel),
                         reinterpret_cast<const void *>(head_reduce_kernel), reinterpret_cast<const void *>(accept_kernel<1>),
                         reinterpret_cast<const void *>(accept_kernel<kAccCluster>),
                         reinterpret_cast<const void *>(state_kernel), reinterpret_cast<const void *>(compact_kernel)};
    status = cudaSuccess;
    for (const void *f : fns)
      if (status == cudaSuccess) status = prefer_max_shared(f);
  });
  return status;
}

cudaError_t launch_compact(const int32_t *done, int max_batch, int32_t *active,
                           int32_t *n_active_dev, cudaStream_t s) {
  compact_kernel<<<1, 32, 0, s>>>(done, max_batch, active, n_active_dev);
  return cudaGetLastError();
}

}  // namespace wf
