// attn_f32.cu -- paged GQA attention of the verification forward for fp32 KV, on the CUDA cores.
//
// Same contract as attn_tc.cu (Sec. 4.4-4.5: request r's k+1 new queries over its L_total = L_cached +
// L_new paged keys, query j seeing keys 0..c_r + j); products and sums in fp32 (tensor cores would
// round the operands).
//
// Persistent CTAs (one per SM) of eight warps take work items (request, KV head, key chunk, row group of
// at most 32 rows) from the plan's counter, longest first.  The warps share an item's queries (in shared
// memory) and split its keys by pages: warp w takes pages w, w + 8, ... of 16 tokens, and nothing but
// its own barriers orders its loop:
//   * K and V pages come by bulk copies, one per token row, into rows of D + 4 floats (the padding keeps
//     the eight rows that a warp reads together in different banks); K is double-buffered, V arrives
//     while the scores are computed, and P overwrites the K page just used;
//   * scores: lane (a, b) = (lane / 8, lane % 8) holds rows a + 4 j and keys b, b + 8: per four head-dim
//     elements RL + 2 16-byte loads feed 4 RL packed multiply-adds (two elements each);
//   * running maximum per row and exp2 weights; the O rows are rescaled only when a maximum moved;
//   * O: lane (a, b) holds rows a + 4 j and head-dim columns 4 b + 32 i: per key D / 32 loads of V for
//     RL D / 16 packed multiply-adds.
// RL (rows per lane) follows the item's row count, so a decode request with few rows does not pay for 32.
// At the item's end the warps' (O, m, l) are merged in shared memory; the last chunk of a split merges
// the chunks' partials.
//
// What bounds it: at full items the reads that feed the score loop (RL + 2 16-byte loads for 4 RL packed
// multiply-adds, at RL = 8 about 40 cycles of the shared-memory return path against 16 of arithmetic)
// and the two warps a scheduler has to hide its latencies with; at few rows the K / V stream.  38
// requests of 8192 tokens, 8 KV heads, D = 128: 38.7 TFLOP/s at 32 rows (about half of the fp32
// rate), 29.0 at 16, 4.4 TB/s at 8, 4.8 TB/s at 4.  32 requests of 512-4096 tokens with 8 to 36 rows:
// 285 us, 26.6 TFLOP/s; shared memory is busy 51% of the time there, issue 38%, DRAM 29%.  At RL = 8 and
// D = 128 the 255 registers do not hold everything: 116 bytes of spills a thread (none at D = 64), 0.2%
// of its instructions.
#include "attn_merge.cuh"

#include <cstring>

namespace wisp {

namespace {

constexpr int kWarps = 8;
constexpr int kThreads = kWarps * 32;
constexpr int kPage = 16;
constexpr int kRows = kF32RowsPerItem;
constexpr long long kWaitCycles = 4000000000LL;  // about two seconds: a wait that long is a failure

template <int D>
struct Cfg {
  static constexpr int LD = D + 4;                    // floats per row in shared memory
  static constexpr int PAGE_F = kPage * LD;           // floats of a K (or V) page
  static constexpr int WARP_F = 3 * PAGE_F;           // two K pages and a V page per warp
  static constexpr int OFF_Q = kWarps * WARP_F;       // [32][LD]
  static constexpr int OFF_ML = OFF_Q + kRows * LD;   // m [8][32], l [8][32]
  static constexpr int FLOATS = OFF_ML + 2 * kWarps * kRows;
  static constexpr int SMEM = FLOATS * 4;
  static constexpr int PLD = 20;                      // floats per row of P (16 keys)
  static_assert(SMEM <= 227 * 1024 - 512, "shared memory of one CTA on sm_103a");
  static_assert(kRows * PLD <= PAGE_F, "P fits a K page");
  static_assert(kRows * D <= 2 * PAGE_F, "a warp's O fits its two K pages");
};

struct Shared {
  uint64_t kbar[kWarps][2], vbar[kWarps];
  int item, last, abort_;
};

__device__ __forceinline__ bool wait_page(uint64_t *b, uint32_t parity, volatile int *abort) {
  if (ptx::mbar_try_wait(b, parity)) return true;
  const long long t0 = clock64();
  while (!ptx::mbar_try_wait(b, parity)) {
    if (clock64() - t0 > kWaitCycles) {
      *abort = 1;
      return false;
    }
  }
  return true;
}

// One item by the whole CTA with RL rows per lane (rows <= 4 RL); Q is in shared memory.  `phk`, `phv`:
// this warp's page copies so far (barrier parities).  Leaves the warps' O, m, l in shared memory.
template <int D, int RL>
__device__ __forceinline__ void item_rows(const AttnParams &p, const WorkItem &w, int g, float *smem, Shared &sh, int warp,
                                          uint32_t &nk, uint32_t &nv) {
  using C = Cfg<D>;
  constexpr int CI = D / 32;  // float4 columns per lane
  const int lane = threadIdx.x & 31, la = lane >> 3, lb = lane & 7;
  float *kb = smem + warp * C::WARP_F, *vb = kb + 2 * C::PAGE_F;
  const float *qs = smem + C::OFF_Q;
  volatile int *abort = &sh.abort_;
  const float scale_log2 = 1.4426950408889634f / sqrtf((float)D);
  const int32_t *bt = p.block_tables + (int64_t)w.r * p.max_blocks_per_seq + w.t0 / kPage;
  const int npages = (w.t1 - w.t0 + kPage - 1) / kPage;
  const float *kc = static_cast<const float *>(p.k_cache), *vc = static_cast<const float *>(p.v_cache);

  // page pg of the item: first float of its (block, head), or -1 for a block outside the pool
  auto page_at = [&](int pg) -> int64_t {
    const int32_t b = __ldg(bt + pg);
    return b < 0 || b >= p.num_blocks ? -1 : ((int64_t)b * p.Hkv + w.h) * kPage * D;
  };
  // rows 0 .. n-1 of a page into `dst`, one bulk copy per lane
  auto load = [&](const float *src, float *dst, int n, uint64_t *bar) {
    ptx::fence_proxy_async_smem();  // earlier generic accesses to dst come first
    __syncwarp();
    if (lane == 0) ptx::mbar_arrive_expect_tx(bar, (uint32_t)n * D * 4u);
    __syncwarp();
    if (lane < n) ptx::bulk_load(ptx::smem_u32(dst + lane * C::LD), src + (int64_t)lane * D, D * 4u, bar);
  };
  auto rows_of = [&](int pg) { return min(kPage, w.t1 - w.t0 - pg * kPage); };

  float2 o[RL][2 * CI];
  float m[RL], l[RL];
#pragma unroll
  for (int j = 0; j < RL; ++j) {
    m[j] = -INFINITY;
    l[j] = 0.0f;
#pragma unroll
    for (int i = 0; i < 2 * CI; ++i) o[j][i] = make_float2(0.0f, 0.0f);
  }
  bool ok = true;
  int64_t at = warp < npages ? page_at(warp) : -1;
  if (at >= 0) load(kc + at, kb + (nk & 1) * C::PAGE_F, rows_of(warp), &sh.kbar[warp][nk & 1]);
  for (int pg = warp; pg < npages && ok; pg += kWarps) {
    const int64_t cur = at;
    at = pg + kWarps < npages ? page_at(pg + kWarps) : -1;
    if (cur < 0) {  // outside the pool: the request is flagged, its outputs are unspecified
      if (lane == 0) report(p.status, WISP_DEV_BAD_BLOCK, p.request_ids, w.r);
      if (at >= 0) load(kc + at, kb + (nk & 1) * C::PAGE_F, rows_of(pg + kWarps), &sh.kbar[warp][nk & 1]);
      continue;
    }
    const int n = rows_of(pg);
    const uint32_t ks = nk & 1, kpar = (nk >> 1) & 1;
    ++nk;
    load(vc + cur, vb, n, &sh.vbar[warp]);
    if (at >= 0) load(kc + at, kb + (nk & 1) * C::PAGE_F, rows_of(pg + kWarps), &sh.kbar[warp][nk & 1]);
    const uint32_t vpar = nv & 1;
    ++nv;
    // ---- scores
    if (!wait_page(&sh.kbar[warp][ks], kpar, abort)) { ok = false; }
    float *kp = kb + ks * C::PAGE_F;
    float2 s2[RL][2];
#pragma unroll
    for (int j = 0; j < RL; ++j) s2[j][0] = s2[j][1] = make_float2(0.0f, 0.0f);
#pragma unroll 4
    for (int d = 0; d < D; d += 4) {
      const float4 k0 = *reinterpret_cast<const float4 *>(kp + lb * C::LD + d);
      const float4 k1 = *reinterpret_cast<const float4 *>(kp + (lb + 8) * C::LD + d);
#pragma unroll
      for (int j = 0; j < RL; ++j) {
        const float4 q = *reinterpret_cast<const float4 *>(qs + (la + 4 * j) * C::LD + d);
        s2[j][0] = __ffma2_rn(make_float2(q.x, q.y), make_float2(k0.x, k0.y), s2[j][0]);
        s2[j][1] = __ffma2_rn(make_float2(q.x, q.y), make_float2(k1.x, k1.y), s2[j][1]);
        s2[j][0] = __ffma2_rn(make_float2(q.z, q.w), make_float2(k0.z, k0.w), s2[j][0]);
        s2[j][1] = __ffma2_rn(make_float2(q.z, q.w), make_float2(k1.z, k1.w), s2[j][1]);
      }
    }
    // ---- weights against the running maxima; row rho sees key t iff t <= ctx + (row0 + rho) / g
    // (every row if t <= ctx: no product of g and a whole context, which 32 bits may not hold)
    const int tok = w.t0 + pg * kPage + lb;
    const int vis0 = tok < w.t1 ? g * max(tok - w.ctx, 0) - w.row0 : 0x7fffffff;  // rows >= vis see the key
    const int vis1 = tok + 8 < w.t1 ? g * max(tok + 8 - w.ctx, 0) - w.row0 : 0x7fffffff;
    float pw[RL][2], alpha[RL];
    bool moved = false;
#pragma unroll
    for (int j = 0; j < RL; ++j) {
      const int rho = la + 4 * j;
      const float a = rho >= vis0 ? (s2[j][0].x + s2[j][0].y) * scale_log2 : -INFINITY;
      const float b = rho >= vis1 ? (s2[j][1].x + s2[j][1].y) * scale_log2 : -INFINITY;
      float mx = fmaxf(a, b);
#pragma unroll
      for (int x = 1; x < 8; x <<= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, x));
      const float mn = fmaxf(m[j], mx);
      alpha[j] = mn == m[j] ? 1.0f : exp2f(m[j] - mn);
      moved |= mn != m[j];
      m[j] = mn;
      // a key not seen, or with a score of -inf, has weight zero (also while mn is -inf)
      pw[j][0] = a == -INFINITY ? 0.0f : exp2f(a - mn);
      pw[j][1] = b == -INFINITY ? 0.0f : exp2f(b - mn);
      l[j] = fmaf(l[j], alpha[j], pw[j][0] + pw[j][1]);
    }
    if (__any_sync(0xffffffffu, moved)) {
#pragma unroll
      for (int j = 0; j < RL; ++j) {
        const float2 al = make_float2(alpha[j], alpha[j]);
#pragma unroll
        for (int i = 0; i < 2 * CI; ++i) o[j][i] = __fmul2_rn(o[j][i], al);
      }
    }
    // ---- P over the K page just read
    __syncwarp();
#pragma unroll
    for (int j = 0; j < RL; ++j) {
      kp[(la + 4 * j) * C::PLD + lb] = pw[j][0];
      kp[(la + 4 * j) * C::PLD + lb + 8] = pw[j][1];
    }
    __syncwarp();
    // ---- O += P V
    if (!wait_page(&sh.vbar[warp], vpar, abort)) { ok = false; }
    if (n < kPage) {  // rows past the item carry weight zero: nothing stale may reach the products
      for (int t = n; t < kPage; ++t)
        for (int d = lane; d < D; d += 32) vb[t * C::LD + d] = 0.0f;
      __syncwarp();
    }
#pragma unroll 1
    for (int t = 0; t < kPage; t += 2) {
      float2 pr[RL];
#pragma unroll
      for (int j = 0; j < RL; ++j) pr[j] = *reinterpret_cast<const float2 *>(kp + (la + 4 * j) * C::PLD + t);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        float4 v[CI];
#pragma unroll
        for (int i = 0; i < CI; ++i) v[i] = *reinterpret_cast<const float4 *>(vb + (t + q) * C::LD + 4 * lb + 32 * i);
#pragma unroll
        for (int j = 0; j < RL; ++j) {
          const float2 x2 = q == 0 ? make_float2(pr[j].x, pr[j].x) : make_float2(pr[j].y, pr[j].y);
#pragma unroll
          for (int i = 0; i < CI; ++i) {
            o[j][2 * i] = __ffma2_rn(x2, make_float2(v[i].x, v[i].y), o[j][2 * i]);
            o[j][2 * i + 1] = __ffma2_rn(x2, make_float2(v[i].z, v[i].w), o[j][2 * i + 1]);
          }
        }
      }
    }
    __syncwarp();
  }
  if (!ok && at >= 0) wait_page(&sh.kbar[warp][nk & 1], (nk >> 1) & 1, abort);  // given up: let the page in flight land
  // ---- this warp's share of the item: row sums over its lanes, then O, m, l to shared memory (the
  // warp's copies have all landed and been read)
  float *po = kb;  // [32][D]
  float *sm = smem + C::OFF_ML + warp * kRows, *sl = sm + kWarps * kRows;
#pragma unroll
  for (int j = 0; j < RL; ++j) {
#pragma unroll
    for (int x = 1; x < 8; x <<= 1) l[j] += __shfl_xor_sync(0xffffffffu, l[j], x);
    const int rho = la + 4 * j;
#pragma unroll
    for (int i = 0; i < CI; ++i)
      *reinterpret_cast<float4 *>(po + rho * D + 4 * lb + 32 * i) =
          make_float4(o[j][2 * i].x, o[j][2 * i].y, o[j][2 * i + 1].x, o[j][2 * i + 1].y);
    if (lb == 0) {
      sm[rho] = m[j];
      sl[rho] = l[j];
    }
  }
}

}  // namespace

template <int D>
__global__ void __launch_bounds__(kThreads, 1) attn_f32_kernel(const __grid_constant__ AttnParams p) {
  using C = Cfg<D>;
  extern __shared__ __align__(128) float smem[];
  __shared__ Shared sh;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  if (tid == 0) {
    for (int i = 0; i < kWarps; ++i) {
      ptx::mbar_init(&sh.kbar[i][0], 1);
      ptx::mbar_init(&sh.kbar[i][1], 1);
      ptx::mbar_init(&sh.vbar[i], 1);
    }
    sh.abort_ = 0;
    ptx::fence_mbar_init();
  }
  // everything above may overlap the planner (programmatic dependent launch); the plan is read
  // only once the planner's grid has completed and its writes are visible
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int n_items = p.header->n_items;
  if ((int)blockIdx.x >= p.header->attn_ctas) return;  // the SM is left to the acceptance pass of the same step
  const int g = p.Hq / p.Hkv;
  uint32_t nk = 0, nv = 0;  // this warp's K and V page copies so far
  for (;;) {
    if (tid == 0) {
      int it;
      do {
        it = atomicAdd(&p.header_mut->next_item, 1);
        if (it >= n_items) it = -1;
      } while (it >= 0 && p.items[it].t1 <= p.items[it].t0);  // (a refused request's items are empty)
      sh.item = it;
    }
    __syncthreads();  // (also: the previous item's shared memory is no longer read)
    const int it = sh.item;
    if (it < 0 || *(volatile int *)&sh.abort_) break;
    const WorkItem w = p.items[it];
    // the item's query rows (rows past `rows` up to the lanes' share read as zero)
    const int rl = (w.rows + 3) / 4;
    const float *qg = static_cast<const float *>(p.q);
    for (int c = tid; c < 4 * rl * (D / 4); c += kThreads) {
      const int row = c / (D / 4), cc = c % (D / 4), rj = w.row0 + row;
      float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (row < w.rows)
        v = __ldg(reinterpret_cast<const float4 *>(qg + ((int64_t)(w.q0 + rj / g) * p.Hq + w.h * g + rj % g) * D) + cc);
      *reinterpret_cast<float4 *>(smem + C::OFF_Q + row * C::LD + 4 * cc) = v;
    }
    __syncthreads();
    switch (rl) {
      case 1: item_rows<D, 1>(p, w, g, smem, sh, warp, nk, nv); break;
      case 2: item_rows<D, 2>(p, w, g, smem, sh, warp, nk, nv); break;
      case 3: item_rows<D, 3>(p, w, g, smem, sh, warp, nk, nv); break;
      case 4: item_rows<D, 4>(p, w, g, smem, sh, warp, nk, nv); break;
      case 5: item_rows<D, 5>(p, w, g, smem, sh, warp, nk, nv); break;
      case 6: item_rows<D, 6>(p, w, g, smem, sh, warp, nk, nv); break;
      case 7: item_rows<D, 7>(p, w, g, smem, sh, warp, nk, nv); break;
      default: item_rows<D, 8>(p, w, g, smem, sh, warp, nk, nv); break;
    }
    __syncthreads();
    // ---- the warps' shares merged: row rho by warp rho mod 8, a lane D / 32 columns
    constexpr int CPL = D / 32;
    const float *sm = smem + C::OFF_ML, *sl = sm + kWarps * kRows;
    for (int rho = warp; rho < w.rows; rho += kWarps) {
      float mx = -INFINITY;
#pragma unroll
      for (int i = 0; i < kWarps; ++i) mx = fmaxf(mx, sm[i * kRows + rho]);
      float den = 0.0f, acc[CPL];
#pragma unroll
      for (int q = 0; q < CPL; ++q) acc[q] = 0.0f;
#pragma unroll
      for (int i = 0; i < kWarps; ++i) {
        const float mi = sm[i * kRows + rho];
        const float x = mi == -INFINITY ? 0.0f : exp2f(mi - mx);
        den = fmaf(sl[i * kRows + rho], x, den);
#pragma unroll
        for (int q = 0; q < CPL; ++q) acc[q] = fmaf(smem[i * C::WARP_F + rho * D + lane * CPL + q], x, acc[q]);
      }
      if (w.poff < 0) {
        const int rj = w.row0 + rho;
        st_cols<CPL>(static_cast<float *>(p.out) + ((int64_t)(w.q0 + rj / g) * p.Hq + w.h * g + rj % g) * D + lane * CPL, acc,
                     1.0f / den);
      } else {
        float *part = p.partials + w.poff;
#pragma unroll
        for (int q = 0; q < CPL; ++q) __stcg(part + (int64_t)rho * D + lane * CPL + q, acc[q]);
        if (lane == 0) {
          __stcg(part + w.rows * D + rho, mx);
          __stcg(part + w.rows * D + w.rows + rho, den);
        }
      }
    }
    if (w.poff >= 0) {
      // split: the last chunk of this (request, head, row group) to finish merges all
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        const int chunks = p.req_chunks[w.r];
        const int done = atomicAdd(p.pair_done + ((int64_t)w.r * p.Hkv + w.h) * p.row_groups + w.rg, 1);
        sh.last = done == chunks - 1 ? chunks : 0;
        __threadfence();
      }
      __syncthreads();
      if (sh.last > 0) merge_chunks<D, float>(p, w, g, sh.last, warp, kWarps);
    }
  }
  if (tid == 0 && *(volatile int *)&sh.abort_) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, -1);
}

cudaError_t attn_f32_setup() {
  cudaError_t e = cudaFuncSetAttribute(attn_f32_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<128>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_f32_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<64>::SMEM);
  return e;
}

cudaError_t attn_f32_launch(const AttnParams &p, int grid, cudaStream_t s) {
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof cfg);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kThreads);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.dynamicSmemBytes = p.D == 128 ? Cfg<128>::SMEM : Cfg<64>::SMEM;
  return p.D == 128 ? cudaLaunchKernelEx(&cfg, attn_f32_kernel<128>, p) : cudaLaunchKernelEx(&cfg, attn_f32_kernel<64>, p);
}

}  // namespace wisp
