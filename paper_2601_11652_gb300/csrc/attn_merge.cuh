// attn_merge.cuh -- merge of the split partials of one (request, KV head, row group), shared by the
// attention kernels: O = sum_c O_c 2^(m_c - m) / sum_c l_c 2^(m_c - m).
#pragma once

#include "attn.cuh"
#include "sm100_ptx.cuh"

namespace wisp {

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<uint32_t *>(&v);
}

// CPL (2 or 4) consecutive floats of a partial, and as many outputs scaled by inv.
template <int CPL>
__device__ __forceinline__ void ld_cols(const float *src, float (&v)[CPL]) {
  if (CPL == 4) {
    const float4 t = __ldcg(reinterpret_cast<const float4 *>(src));
    v[0] = t.x;
    v[1] = t.y;
    v[CPL - 2] = t.z;
    v[CPL - 1] = t.w;
  } else {
    const float2 t = __ldcg(reinterpret_cast<const float2 *>(src));
    v[0] = t.x;
    v[1] = t.y;
  }
}
template <int CPL>
__device__ __forceinline__ void st_cols(uint16_t *dst, const float (&v)[CPL], float inv) {
  if (CPL == 4)
    *reinterpret_cast<uint2 *>(dst) = make_uint2(pack_bf16(v[0] * inv, v[1] * inv), pack_bf16(v[CPL - 2] * inv, v[CPL - 1] * inv));
  else
    *reinterpret_cast<uint32_t *>(dst) = pack_bf16(v[0] * inv, v[1] * inv);
}
template <int CPL>
__device__ __forceinline__ void st_cols(float *dst, const float (&v)[CPL], float inv) {
  if (CPL == 4)
    *reinterpret_cast<float4 *>(dst) = make_float4(v[0] * inv, v[1] * inv, v[CPL - 2] * inv, v[CPL - 1] * inv);
  else
    *reinterpret_cast<float2 *>(dst) = make_float2(v[0] * inv, v[1] * inv);
}

// By warp `wq` of `nw`.  The chunks' partials lie a fixed stride apart.  A warp takes two rows at a time: a
// lane holds one chunk's (m, l) of each, the warp reduces the rows' maximum and denominator, and then
// every lane adds its columns of the chunks' O with the chunk's weight broadcast by a shuffle, four
// chunks of both rows in flight.  (With one thread per row walking the chunks' (m, l), the merge took
// about 90 us of a request's 114 us at 16 chunks: serial chains of L2 loads.)
template <int D, typename T>
__device__ __forceinline__ void merge_chunks(const AttnParams &p, const WorkItem &w, int g, int chunks, int wq, int nw) {
  const int lane = threadIdx.x & 31;
  const float *base = p.partials + w.pbase;
  const int stride = ((w.rg ? w.row0 / w.rg : w.rows) * (D + 2) + 3) / 4 * 4;  // (groups before the last have equal rows)
  constexpr int CPL = D / 32;  // columns per lane
  T *og = static_cast<T *>(p.out);
  for (int j0 = 2 * wq; j0 < w.rows; j0 += 2 * nw) {
    const int j1 = min(j0 + 1, w.rows - 1);  // an odd last row is merged twice, alike
    float m0 = -INFINITY, m1 = -INFINITY;
    for (int c = lane; c < chunks; c += 32) {
      const float *pm = base + (int64_t)c * stride + w.rows * D;
      m0 = fmaxf(m0, __ldcg(pm + j0));
      m1 = fmaxf(m1, __ldcg(pm + j1));
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      m0 = fmaxf(m0, __shfl_xor_sync(0xffffffffu, m0, o));
      m1 = fmaxf(m1, __shfl_xor_sync(0xffffffffu, m1, o));
    }
    float den0 = 0.0f, den1 = 0.0f, a0[CPL], a1[CPL];
#pragma unroll
    for (int q = 0; q < CPL; ++q) a0[q] = a1[q] = 0.0f;
    for (int c0 = 0; c0 < chunks; c0 += 32) {
      float w0 = 0.0f, w1 = 0.0f;  // lane: chunk c0 + lane
      if (c0 + lane < chunks) {
        const float *pm = base + (int64_t)(c0 + lane) * stride + w.rows * D;
        const float mc0 = __ldcg(pm + j0), mc1 = __ldcg(pm + j1);
        w0 = mc0 == -INFINITY ? 0.0f : ptx::ex2(mc0 - m0);
        w1 = mc1 == -INFINITY ? 0.0f : ptx::ex2(mc1 - m1);
        den0 = fmaf(__ldcg(pm + w.rows + j0), w0, den0);
        den1 = fmaf(__ldcg(pm + w.rows + j1), w1, den1);
      }
      const int nc = min(32, chunks - c0);
#pragma unroll 1
      for (int c = 0; c < nc; c += 4) {
        float v0[4][CPL], v1[4][CPL];
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const float *po = base + (int64_t)(c0 + min(c + u, nc - 1)) * stride + lane * CPL;
          ld_cols<CPL>(po + (int64_t)j0 * D, v0[u]);
          ld_cols<CPL>(po + (int64_t)j1 * D, v1[u]);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          // a chunk with weight zero (none of its keys visible to the row) adds nothing
          const float x0 = __shfl_sync(0xffffffffu, w0, (c + u) & 31);
          const float x1 = __shfl_sync(0xffffffffu, w1, (c + u) & 31);
          const bool in = c + u < nc;
#pragma unroll
          for (int q = 0; q < CPL; ++q) {
            if (in && x0 != 0.0f) a0[q] = fmaf(v0[u][q], x0, a0[q]);
            if (in && x1 != 0.0f) a1[q] = fmaf(v1[u][q], x1, a1[q]);
          }
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      den0 += __shfl_xor_sync(0xffffffffu, den0, o);
      den1 += __shfl_xor_sync(0xffffffffu, den1, o);
    }
    const float i0 = 1.0f / den0, i1 = 1.0f / den1;
    const int rj0 = w.row0 + j0, rj1 = w.row0 + j1;
    st_cols<CPL>(og + ((int64_t)(w.q0 + rj0 / g) * p.Hq + w.h * g + rj0 % g) * D + lane * CPL, a0, i0);
    st_cols<CPL>(og + ((int64_t)(w.q0 + rj1 / g) * p.Hq + w.h * g + rj1 % g) * D + lane * CPL, a1, i1);
  }
}

}  // namespace wisp
