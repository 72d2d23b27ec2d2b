// kv.cu -- paged KV-cache maintenance around the verification step (include/wisp_kv.h).
//
// Sec. 4.5: per-session KV lives in fixed-size pages (PageAttention) and a prefix cache that is
// updated in place, so a verification forwards only the new block.  Three kernels:
//   kv_reserve_kernel (one cluster of 8 CTAs): validates the lengths, counts each request's missing
//     pages among those covering tokens 0 .. c + k, serves requests in order from the top of the
//     device-side free stack (block-wide scans, so the assignment is deterministic), and maps every
//     new K/V row to its (request, position);
//   kv_append_kernel: one warp per (new row, KV head) copies the row into its page slot;
//   kv_commit_kernel (one CTA): c <- c + 1 + L (Eq. 2's L), and the pages past the new length
//     among those the step could use go back on the free stack in table order.
#include "common.cuh"

#include <cstring>

#include "wisp_kv.h"

namespace wisp {

namespace {

constexpr int kThreads = 1024;
constexpr int kPage = 16;
constexpr int kReserveCtas = 8;  // one cluster (the portable maximum): its barrier orders counting before serving

struct KvParams {
  int B, Hkv, D, max_blocks, num_blocks, total_rows, esize;
  const int64_t *request_ids;
  const int32_t *draft_lens;
  int32_t *context_lens, *block_tables, *free_blocks, *free_count;
  char *k_cache, *v_cache;
  const char *k_new, *v_new;
  const int32_t *accepted_len;
  DeviceStatus *status;
  int32_t *row_req, *row_pos;  // [total_rows]: request of a new row (-1: skipped) and its position
  int32_t *need, *first;       // [B]: a request's missing pages (-code: refused), its first missing table entry
};

__device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }

// Exclusive block-wide prefix sum; *total receives the block's sum.
__device__ int64_t scan_excl(int64_t v, int64_t *s_warp, int64_t *total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  int64_t x = v;
  for (int d = 1; d < 32; d <<= 1) {
    const int64_t o = __shfl_up_sync(0xffffffffu, x, d);
    if (lane >= d) x += o;
  }
  if (lane == 31) s_warp[w] = x;
  __syncthreads();
  if (w == 0) {
    int64_t t = s_warp[lane];
    for (int d = 1; d < 32; d <<= 1) {
      const int64_t o = __shfl_up_sync(0xffffffffu, t, d);
      if (lane >= d) t += o;
    }
    s_warp[lane] = t;
  }
  __syncthreads();
  const int64_t incl = x + (w > 0 ? s_warp[w - 1] : 0);
  *total = s_warp[31];
  __syncthreads();
  return incl - v;
}

// Block-wide maximum.
__device__ int64_t block_max(int64_t v, int64_t *s_warp) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  for (int d = 16; d > 0; d >>= 1) v = max(v, __shfl_xor_sync(0xffffffffu, v, d));
  if (lane == 0) s_warp[w] = v;
  __syncthreads();
  int64_t m = s_warp[0];
  for (int i = 1; i < 32; ++i) m = max(m, s_warp[i]);
  __syncthreads();
  return m;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

// Bound by the latency of reading the block tables (4 bytes a page, 0.1-1 MB a batch) and of its barriers.  A
// warp reads one request's row, lanes side by side and four loads ahead.  64 requests of up to 2048
// pages: 16 us with cold caches.
__global__ void __launch_bounds__(kThreads) __cluster_dims__(kReserveCtas, 1, 1) kv_reserve_kernel(const KvParams p) {
  // the append kernel may be placed now; it waits for this grid before it reads anything
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ int64_t s_warp[32];
  __shared__ int32_t s_before[kThreads], s_q0[kThreads];
  const int lane = threadIdx.x & 31;
  const int gw = blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);  // warp of the cluster
  constexpr int NWARPS = kReserveCtas * kThreads / 32;
  int64_t F = *p.free_count;  // read before the barrier, written after it
  const bool pool_bad = F < 0 || F > p.num_blocks;  // inconsistent pool: serve nobody
  if (pool_bad) F = 0;
  if (blockIdx.x == 0 && threadIdx.x == 0) {  // the launch's status word starts clear: reports come after the barrier
    p.status->code = 0;
    p.status->pad = 0;
    p.status->request_id = 0;
  }
  const int64_t cap = (int64_t)p.max_blocks * kPage;

  // count: request r by warp r mod NWARPS
  for (int r = gw; r < p.B; r += NWARPS) {
    const int64_t k = p.draft_lens[r], c = p.context_lens[r];
    int bad = k < 0 || c < 0 || c + k + 1 > cap ? WISP_DEV_BAD_LENGTH : 0;
    int n = 0, first = INT32_MAX;
    if (!bad) {
      const int32_t *row = p.block_tables + (int64_t)r * p.max_blocks;
      const int nb = (int)((c + k + 1 + kPage - 1) / kPage);
      bool over = false;
      for (int b0 = 0; b0 < nb; b0 += 128) {
        int32_t id[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) id[u] = b0 + 32 * u + lane < nb ? row[b0 + 32 * u + lane] : 0;
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const bool miss = id[u] < 0;
          over |= id[u] >= p.num_blocks;
          if (miss && first == INT32_MAX) first = b0 + 32 * u + lane;
          n += miss ? 1 : 0;
        }
      }
      n = __reduce_add_sync(0xffffffffu, n);
      first = __reduce_min_sync(0xffffffffu, first);
      if (__any_sync(0xffffffffu, over)) bad = WISP_DEV_BAD_BLOCK;
    }
    if (lane == 0) {
      __stcg(p.need + r, bad ? -bad : n);
      __stcg(p.first + r, first);
    }
  }
  __threadfence();
  cluster_sync();

  if (pool_bad && blockIdx.x == 0 && threadIdx.x == 0) report(p.status, WISP_DEV_BAD_BLOCK, p.request_ids, -1);
  // serve: every CTA scans the needs of 1024 requests at a time, then its warps take their requests
  int64_t carry_need = 0, carry_rows = 0, taken = 0;
  for (int base = 0; base < p.B; base += kThreads) {
    {
      const int r = base + threadIdx.x;
      const int64_t nd = r < p.B ? __ldcg(p.need + r) : 0, need = nd > 0 ? nd : 0;
      const int64_t k = r < p.B ? max(0, p.draft_lens[r]) : -1;
      int64_t tot_need, tot_rows;
      const int64_t before = carry_need + scan_excl(need, s_warp, &tot_need);
      const int64_t q0 = carry_rows + scan_excl(k + 1, s_warp, &tot_rows);
      // served requests form a prefix of the valid ones: `before + need` only grows with r
      const bool served = r < p.B && nd >= 0 && before + need <= F;
      s_before[threadIdx.x] = served ? (int32_t)before : -1;
      s_q0[threadIdx.x] = (int32_t)min64(q0, INT32_MAX);
      taken = max(taken, block_max(served ? before + need : 0, s_warp));  // (its barriers publish s_before, s_q0)
      carry_need += tot_need;
      carry_rows += tot_rows;
    }
    for (int r = base + gw; r < min(p.B, base + kThreads); r += NWARPS) {
      const int before = s_before[r - base];
      const bool served = before >= 0;
      const int k = max(0, p.draft_lens[r]), c = p.context_lens[r];
      const int need = __ldcg(p.need + r);
      if (!served && lane == 0) report(p.status, need < 0 ? -need : (int)WISP_DEV_NO_BLOCKS, p.request_ids, r);
      if (served && need > 0) {
        // pop from the top of the stack: this request's missing pages, in table order, take
        // entries F-1-before, F-2-before, ...
        int32_t *row = p.block_tables + (int64_t)r * p.max_blocks;
        const int nb = (int)(((int64_t)c + k + 1 + kPage - 1) / kPage);
        int t = 0;
        for (int b0 = __ldcg(p.first + r); t < need && b0 < nb; b0 += 32) {
          const bool miss = b0 + lane < nb && row[b0 + lane] < 0;
          const unsigned m = __ballot_sync(0xffffffffu, miss);
          if (miss) row[b0 + lane] = p.free_blocks[F - 1 - before - t - __popc(m & ((1u << lane) - 1))];
          t += __popc(m);
        }
      }
      const int64_t q0 = s_q0[r - base];
      for (int64_t j = lane; j <= k && q0 + j < p.total_rows; j += 32) {
        p.row_req[q0 + j] = served ? r : -1;
        p.row_pos[q0 + j] = (int32_t)(c + j);
      }
    }
    __syncthreads();  // s_before and s_q0 are rewritten by the next 1024 requests
  }
  // rows past the requests' (total_rows larger than the sum of the lengths): nobody's
  for (int64_t x = carry_rows + blockIdx.x * kThreads + threadIdx.x; x < p.total_rows; x += kReserveCtas * kThreads)
    p.row_req[x] = -1;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    *p.free_count = (int32_t)(F - taken);
    if (carry_rows != p.total_rows) atomicCAS(&p.status->code, 0, (int32_t)WISP_DEV_BAD_LENGTH);
  }
}

// One warp per (new row, KV head): the row's D values into their page slot (16-byte vectors).
__global__ void __launch_bounds__(256) kv_append_kernel(const KvParams p) {
  asm volatile("griddepcontrol.wait;" ::: "memory");  // launched as a programmatic dependent of the reservation
  const int lane = threadIdx.x & 31;
  const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const int nvec = p.D * p.esize / 16;
  for (int64_t wi = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); wi < (int64_t)p.total_rows * p.Hkv;
       wi += nwarps) {
    const int64_t row = wi / p.Hkv;
    const int h = (int)(wi % p.Hkv);
    const int r = p.row_req[row];
    if (r < 0) continue;
    const int pos = p.row_pos[row];
    const int32_t page = p.block_tables[(int64_t)r * p.max_blocks + pos / kPage];
    if (page < 0 || page >= p.num_blocks) {  // a page id from the free stack outside the pool
      if (lane == 0) report(p.status, WISP_DEV_BAD_BLOCK, p.request_ids, r);
      continue;
    }
    const int64_t dst = ((((int64_t)page * p.Hkv + h) * kPage) + pos % kPage) * p.D * p.esize;
    const int64_t src = (row * p.Hkv + h) * (int64_t)p.D * p.esize;
    for (int v = lane; v < nvec; v += 32) {
      reinterpret_cast<uint4 *>(p.k_cache + dst)[v] = __ldg(reinterpret_cast<const uint4 *>(p.k_new + src) + v);
      reinterpret_cast<uint4 *>(p.v_cache + dst)[v] = __ldg(reinterpret_cast<const uint4 *>(p.v_new + src) + v);
    }
  }
}

__global__ void __launch_bounds__(kThreads) kv_commit_kernel(const KvParams p) {
  __shared__ int64_t s_warp[32];
  const int64_t F = *p.free_count;
  if (threadIdx.x == 0) {  // the launch's status word starts clear
    p.status->code = 0;
    p.status->pad = 0;
    p.status->request_id = 0;
  }
  __syncthreads();
  if (F < 0 || F > p.num_blocks) {  // inconsistent pool: release nothing
    if (threadIdx.x == 0) report(p.status, WISP_DEV_BAD_BLOCK, p.request_ids, -1);
    return;
  }
  int64_t carry = 0;
  for (int base = 0; base < p.B; base += kThreads) {
    const int r = base + threadIdx.x;
    int64_t rel = 0, keep = 0, used = 0, cnew = 0;
    int bad = 0;
    if (r < p.B) {
      const int64_t k = p.draft_lens[r], c = p.context_lens[r], L = p.accepted_len[r];
      if (k < 0 || c < 0 || L < 0 || L > k || c + k + 1 > (int64_t)p.max_blocks * kPage) bad = WISP_DEV_BAD_LENGTH;
      if (!bad) {
        cnew = c + 1 + L;
        keep = (cnew + kPage - 1) / kPage;
        used = (c + k + 1 + kPage - 1) / kPage;
        const int32_t *row = p.block_tables + (int64_t)r * p.max_blocks;
        for (int64_t b = keep; b < used; ++b) rel += row[b] >= 0 ? 1 : 0;
      } else {
        report(p.status, bad, p.request_ids, r);
      }
    }
    int64_t tot;
    const int64_t at = F + carry + scan_excl(rel, s_warp, &tot);
    if (r < p.B && !bad) {
      int32_t *row = p.block_tables + (int64_t)r * p.max_blocks;
      int64_t t = 0;
      for (int64_t b = keep; b < used; ++b) {
        if (row[b] >= 0) {
          if (at + t >= p.num_blocks) {  // more pages than the pool holds: the caller's state is broken
            report(p.status, WISP_DEV_BAD_BLOCK, p.request_ids, r);
            break;
          }
          p.free_blocks[at + t++] = row[b];
          row[b] = -1;
        }
      }
      p.context_lens[r] = (int32_t)cnew;
    }
    carry += tot;
  }
  if (threadIdx.x == 0) *p.free_count = (int32_t)min64(F + carry, p.num_blocks);
}

struct KvLayout {
  size_t status = 0, row_req = 0, row_pos = 0, need = 0, first = 0, total = 0;
};

KvLayout kv_layout(const wisp_kv_args *a) {
  KvLayout L;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t at = off;
    off = (off + bytes + 255) & ~(size_t)255;
    return at;
  };
  L.status = take(sizeof(DeviceStatus));
  L.row_req = take(sizeof(int32_t) * (size_t)a->total_q_rows);
  L.row_pos = take(sizeof(int32_t) * (size_t)a->total_q_rows);
  L.need = take(sizeof(int32_t) * (size_t)a->B);
  L.first = take(sizeof(int32_t) * (size_t)a->B);
  L.total = off;
  return L;
}

bool al16(const void *p) { return ((uintptr_t)p & 15) == 0; }

wisp_status kv_check(const wisp_kv_args *a, bool need_new, bool need_accepted) {
  if (!a) return WISP_ERR_INVALID_ARG;
  if (a->B < 0 || a->Hkv <= 0 || a->total_q_rows < a->B || a->num_blocks <= 0 || a->max_blocks_per_seq <= 0)
    return WISP_ERR_INVALID_ARG;
  if (a->D != 64 && a->D != 128) return WISP_ERR_UNSUPPORTED;
  if (a->block_size != kPage) return WISP_ERR_UNSUPPORTED;
  if (a->kv_dtype != WISP_F32 && a->kv_dtype != WISP_BF16) return WISP_ERR_INVALID_ARG;
  if (a->B == 0) return WISP_OK;
  if (!a->draft_lens || !a->context_lens || !a->block_tables || !a->free_blocks || !a->free_count)
    return WISP_ERR_INVALID_ARG;
  if (need_new && (!a->k_cache || !a->v_cache || !a->k_new || !a->v_new)) return WISP_ERR_INVALID_ARG;
  if (need_new && (!al16(a->k_cache) || !al16(a->v_cache) || !al16(a->k_new) || !al16(a->v_new)))
    return WISP_ERR_INVALID_ARG;
  if (need_accepted && !a->accepted_len) return WISP_ERR_INVALID_ARG;
  if ((int64_t)a->max_blocks_per_seq * kPage > INT32_MAX / 2) return WISP_ERR_UNSUPPORTED;
  return WISP_OK;
}

KvParams kv_params(const wisp_kv_args *a, void *ws, const KvLayout &L) {
  KvParams p;
  std::memset(&p, 0, sizeof p);
  p.B = a->B;
  p.Hkv = a->Hkv;
  p.D = a->D;
  p.max_blocks = a->max_blocks_per_seq;
  p.num_blocks = a->num_blocks;
  p.total_rows = a->total_q_rows;
  p.esize = a->kv_dtype == WISP_BF16 ? 2 : 4;
  p.request_ids = a->request_ids;
  p.draft_lens = a->draft_lens;
  p.context_lens = a->context_lens;
  p.block_tables = a->block_tables;
  p.free_blocks = a->free_blocks;
  p.free_count = a->free_count;
  p.k_cache = static_cast<char *>(a->k_cache);
  p.v_cache = static_cast<char *>(a->v_cache);
  p.k_new = static_cast<const char *>(a->k_new);
  p.v_new = static_cast<const char *>(a->v_new);
  p.accepted_len = a->accepted_len;
  p.status = reinterpret_cast<DeviceStatus *>(static_cast<char *>(ws) + L.status);
  p.row_req = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + L.row_req);
  p.row_pos = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + L.row_pos);
  p.need = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + L.need);
  p.first = reinterpret_cast<int32_t *>(static_cast<char *>(ws) + L.first);
  return p;
}

wisp_status kv_ws_ok(void *ws, size_t bytes, const KvLayout &L) {
  return !ws || ((uintptr_t)ws & 255) != 0 || bytes < L.total ? WISP_ERR_WORKSPACE : WISP_OK;
}

}  // namespace

}  // namespace wisp

using namespace wisp;

extern "C" {

size_t wisp_kv_workspace_size(const wisp_kv_args *kv) {
  if (kv_check(kv, false, false) != WISP_OK) return 0;
  return kv_layout(kv).total;
}

wisp_status wisp_kv_reserve_append(const wisp_kv_args *kv, void *ws, size_t ws_bytes, void *stream) {
  wisp_status st = kv_check(kv, true, false);
  if (st != WISP_OK) return st;
  const KvLayout L = kv_layout(kv);
  if ((st = kv_ws_ok(ws, ws_bytes, L)) != WISP_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const KvParams p = kv_params(kv, ws, L);
  if (kv->B == 0)
    return cudaMemsetAsync(p.status, 0, sizeof(DeviceStatus), s) == cudaSuccess ? WISP_OK : WISP_ERR_CUDA;
  kv_reserve_kernel<<<kReserveCtas, kThreads, 0, s>>>(p);
  if (cudaGetLastError() != cudaSuccess) return WISP_ERR_CUDA;
  const int64_t warps = (int64_t)kv->total_q_rows * kv->Hkv;
  const int64_t blocks = (warps + 7) / 8;
  cudaLaunchConfig_t cfg;
  std::memset(&cfg, 0, sizeof cfg);
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)(blocks < 4096 ? blocks : 4096));
  cfg.blockDim = dim3(256);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kv_append_kernel, p) == cudaSuccess ? WISP_OK : WISP_ERR_CUDA;
}

wisp_status wisp_kv_commit(const wisp_kv_args *kv, void *ws, size_t ws_bytes, void *stream) {
  wisp_status st = kv_check(kv, false, true);
  if (st != WISP_OK) return st;
  const KvLayout L = kv_layout(kv);
  if ((st = kv_ws_ok(ws, ws_bytes, L)) != WISP_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const KvParams p = kv_params(kv, ws, L);
  if (kv->B == 0)
    return cudaMemsetAsync(p.status, 0, sizeof(DeviceStatus), s) == cudaSuccess ? WISP_OK : WISP_ERR_CUDA;
  kv_commit_kernel<<<1, kThreads, 0, s>>>(p);
  return cudaGetLastError() == cudaSuccess ? WISP_OK : WISP_ERR_CUDA;
}

}  // extern "C"
