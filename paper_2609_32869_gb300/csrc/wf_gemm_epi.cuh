// Epilogue arithmetic shared by the tcgen05 projection kernels: four output
// features of one token row at a time.
#pragma once
#include "wf_device.cuh"
#include "wf_internal.h"

namespace wf {

// Four floats as four bf16 (round to nearest even) in one 8-byte word.
__device__ __forceinline__ uint2 pack4_bf16(const float (&v)[4]) {
  __nv_bfloat162 h[2] = {__floats2bfloat162_rn(v[0], v[1]), __floats2bfloat162_rn(v[2], v[3])};
  return *reinterpret_cast<const uint2 *>(h);
}
// Non-residual epilogues of four features: GELU, then fp32, bf16 or the
// query / key / value split with the cache scatter.
template <int EPI>
__device__ __forceinline__ void epi_quad_out(const GemmParams &p, int t, int n, float (&v)[4],
                                             const int2 *tok_local, float (&fin)[4]) {
  if constexpr (EPI == EPI_GELU) {
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = gelu_erf(v[i]);
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) fin[i] = v[i];
  const bool whole = n + 3 < p.N && (p.ld_out & 3) == 0;
  if constexpr (EPI == EPI_F32) {
    float *o = p.out_f32 + static_cast<size_t>(t) * p.ld_out + n;
    if (whole && (reinterpret_cast<uintptr_t>(p.out_f32) & 15) == 0) {
      *reinterpret_cast<float4 *>(o) = make_float4(v[0], v[1], v[2], v[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (n + i < p.N) o[i] = v[i];
    }
  } else if constexpr (EPI == EPI_BF16 || EPI == EPI_GELU) {
    bf16 *o = p.out_bf16 + static_cast<size_t>(t) * p.ld_out + n;
    if (whole) {
      *reinterpret_cast<uint2 *>(o) = pack4_bf16(v);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (n + i < p.N) o[i] = __float2bfloat16(v[i]);
    }
  } else if constexpr (EPI == EPI_KV) {
    // N, q_cols and d_model are multiples of 4 (checked at launch)
    if (n >= p.N) return;
    if (n < p.q_cols) {
      *reinterpret_cast<uint2 *>(p.out_bf16 + static_cast<size_t>(t) * p.ld_out + n) = pack4_bf16(v);
      return;
    }
    const int c = n - p.q_cols;
    const int which = c / p.d_model;
    const int hd = c - which * p.d_model;
    const int2 sp = *tok_local;
    if (sp.y >= p.ctx) {
      set_error(p.err, WF_DEV_ERR_CAPACITY);
      return;
    }
    bf16 *dst = which == 0 ? p.kc : p.vc;
    *reinterpret_cast<uint2 *>(
        dst + ((static_cast<size_t>(sp.x) * p.n_heads + (hd >> 6)) * p.ctx + sp.y) * 64 + (hd & 63)) =
        pack4_bf16(v);
  }
}

// Epilogue of four consecutive output features n..n+3 of token row t (the
// staged path).  `old` is the residual row's current value (EPI_RESID).
// fin[] returns the final values (the updated residual for EPI_RESID) for the
// LayerNorm statistics.  Four consecutive features never straddle a head or
// the key/value boundary (multiples of 4), so each store is one vector.
template <int EPI>
__device__ __forceinline__ void epi_quad(const GemmParams &p, int t, int n, const float4 &a,
                                         const float (&b4)[4], const float4 &old,
                                         const int2 *tok_local, float (&fin)[4]) {
  float v[4] = {a.x + b4[0], a.y + b4[1], a.z + b4[2], a.w + b4[3]};
  if constexpr (EPI == EPI_RESID) {
    // N % 128 == 0 and ld_resid % 4 == 0 (checked at launch): one float4
    float4 *r = reinterpret_cast<float4 *>(p.resid + static_cast<size_t>(t) * p.ld_resid + n);
    const float4 nr = make_float4(old.x + v[0], old.y + v[1], old.z + v[2], old.w + v[3]);
    *r = nr;
    fin[0] = nr.x;
    fin[1] = nr.y;
    fin[2] = nr.z;
    fin[3] = nr.w;
    const uint2 h = pack4_bf16(fin);
    if (p.tap0) *reinterpret_cast<uint2 *>(p.tap0 + static_cast<size_t>(t) * p.ld_tap + n) = h;
    if (p.tap1) *reinterpret_cast<uint2 *>(p.tap1 + static_cast<size_t>(t) * p.ld_tap + n) = h;
  } else {
    epi_quad_out<EPI>(p, t, n, v, tok_local, fin);
  }
}

}  // namespace wf
