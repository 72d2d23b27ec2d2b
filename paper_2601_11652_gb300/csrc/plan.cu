// plan.cu -- one-CTA planner: request offsets, length validation and the split-KV work list.
//
// The verification batch (Sec. 4.5) is ragged: request r contributes k_r + 1 query
// rows and c_r + k_r + 1 keys (L_total = L_cached + L_new, Sec. 4.4).  Lengths
// live on the device, so the planner runs there: it prefix-sums the row offsets,
// flags invalid requests, and cuts every (request, KV head) sequence into chunks
// of at most `chunk_len` keys so that the attention grid has about one item per
// SM (kItemsPerSM when there are fewer (request, head) pairs than SMs) whatever
// the length mix.
#include "plan.cuh"

namespace wisp {

namespace {

constexpr int kThreads = 1024;
constexpr int kOrderBuckets = 1024;  // tile-count buckets of the dispatch order
constexpr int kOrderTile = 64;       // tokens per KV tile of the attention kernels

__device__ __forceinline__ int64_t min64(int64_t a, int64_t b) { return a < b ? a : b; }
__device__ __forceinline__ int64_t max64(int64_t a, int64_t b) { return a > b ? a : b; }

// Inclusive block scan of one int per thread; returns the inclusive value, *total the block sum.  One
// barrier: every warp scans the warps' sums itself.  s_w (32 values) may be written again only after
// another barrier.
__device__ int block_scan(int v, int *s_w, int *total) {
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, v, d);
    if (lane >= d) v += o;
  }
  if (lane == 31) s_w[w] = v;
  __syncthreads();
  int t = s_w[lane];
#pragma unroll
  for (int d = 1; d < 32; d <<= 1) {
    const int o = __shfl_up_sync(0xffffffffu, t, d);
    if (lane >= d) t += o;
  }
  const int before = __shfl_sync(0xffffffffu, t, (w + 31) & 31);
  *total = __shfl_sync(0xffffffffu, t, 31);
  return v + (w > 0 ? before : 0);
}

// a / b rounded up, b > 0 (the 64-bit division only where 32 bits do not hold a)
__device__ __forceinline__ int64_t ceil_div(int64_t a, int64_t b) {
  const int64_t x = a + b - 1;
  return x <= 0xffffffffll && b <= 0xffffffffll ? (int64_t)((uint32_t)x / (uint32_t)b) : x / b;
}

// The acceptance pass's dispatch order and state.  Rows are listed level-major: row index 0 of
// every valid request, then row index 1, ... (the requests of a level in decreasing draft length, so
// that request r holds the same position pos(r) in every level it reaches).  The decision of row i
// of a request is then usually known before its row i + 1 comes up, and the acceptance kernel skips
// rows past a rejection.  Also clears the per-row and per-request state of the launch and gives the
// requests this planner refused -1 outputs.
// The caller has cleared sh.n and sh.nvalid before a barrier; one: at most kThreads requests, thread r holds
// request r's k and whether it is valid.
struct AcceptPlan {
  static constexpr int KB = kMaxDraft + 1;  // draft lengths 0..kMaxDraft
  int32_t n[2 * kThreads];                  // histogram of k, then the buckets' cursors
  int32_t ls[2 * kThreads];                 // level starts
  int w[2][32];
  int32_t nvalid;
};
static_assert(AcceptPlan::KB + 1 <= 2 * kThreads, "two buckets per thread");

__device__ __forceinline__ void plan_accept_clear(AcceptPlan &sh) {
  sh.n[threadIdx.x] = sh.n[threadIdx.x + kThreads] = 0;
  if (threadIdx.x == 0) sh.nvalid = 0;
}

__device__ void plan_accept(const PlanParams &p, AcceptPlan &sh, bool one, int my_k, bool my_ok) {
  const int tid = threadIdx.x;
  int nv = 0;
  for (int r = tid; r < p.B; r += kThreads) {
    p.req_rej[r] = INT32_MAX;
    p.req_claim[r] = 0;
    p.req_dcnt[r] = 0;
    p.queue[r] = -1;
    if (one ? my_ok : p.req_flag[r] == REQ_OK) {
      atomicAdd(&sh.n[one ? my_k : p.draft_lens[r]], 1);  // histogram of k
      ++nv;
    } else {
      p.accepted_len[r] = -1;
      p.next_token[r] = -1;
    }
  }
  // valid requests: a warp sum per warp, added into a shared counter
  nv = __reduce_add_sync(0xffffffffu, nv);
  if ((tid & 31) == 0 && nv) atomicAdd(&sh.nvalid, nv);
  for (int64_t j = tid; j < p.total_q_rows; j += kThreads) {
    p.row_cnt[j] = 0;
    p.row_code[j] = 0;
  }
  for (int j = tid; j < kTabCacheSlots; j += kThreads) {
    p.acc_ctr->tab_state[j] = 0;
    p.acc_ctr->tab_m[j] = 0;
  }
  __syncthreads();
  // per bucket b (two per thread): level size n_b = #{k >= b}, its start (the sum of the levels before), and
  // the bucket's cursor n_{b+1} (in every level the requests with a larger k come first)
  const int nvalid = sh.nvalid, h0 = sh.n[2 * tid], h1 = sh.n[2 * tid + 1];
  int tot, rows_valid;
  const int n0 = nvalid - (block_scan(h0 + h1, sh.w[0], &tot) - h0 - h1), n1 = n0 - h0;
  const int l0 = block_scan(n0 + n1, sh.w[1], &rows_valid) - n0 - n1;
  sh.ls[2 * tid] = l0;
  sh.ls[2 * tid + 1] = l0 + n0;
  sh.n[2 * tid] = n0 - h0;
  sh.n[2 * tid + 1] = n1 - h1;
  __syncthreads();
  for (int r = tid; r < p.B; r += kThreads) {
    if (!(one ? my_ok : p.req_flag[r] == REQ_OK)) continue;
    const int k = one ? my_k : p.draft_lens[r];
    const int pos = atomicAdd(&sh.n[k], 1);
    for (int i = 0; i <= k; ++i) p.row_order[sh.ls[i] + pos] = make_int2(r, i);
  }
  if (tid == 0) {
    p.acc_ctr->n_items = rows_valid * p.sslices;
    p.acc_ctr->n_valid = nvalid;
    p.acc_ctr->q_reserve = 0;
    p.acc_ctr->q_head = 0;
    p.acc_ctr->n_claimed = 0;
    p.acc_ctr->stats_next = 0;
  }
}

}  // namespace

// One CTA, bound by latency: global loads of the lengths, then barriers.  So: 32-bit scans with one barrier
// each, each item's request kept from pass to pass, and no 64-bit division where 32 bits hold the
// operands.  One request takes 8.6 us here and 256 requests 15 us (cold caches, launch included).
__global__ void __launch_bounds__(kThreads, 1) plan_kernel(const PlanParams p) {
  // a kernel launched after this one with programmatic stream serialization (the attention) may
  // start its own set-up now; it reads the plan only after waiting for this grid to complete
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int kKeep = 4;  // items per thread whose request is kept in registers
  __shared__ int s_w[6][32];
  __shared__ unsigned long long s_sum[2];  // keys of the valid requests; passes over their KV tiles per KV head
  __shared__ int32_t s_valid;
  __shared__ int32_t s_hist[kOrderBuckets];
  // the attention's per-request arrays (pass 3) come after the acceptance part is done with its own
  union Shared {
    AcceptPlan acc;
    struct {
      int32_t first[kThreads + 1], rows[kThreads], ch[kThreads], pf[kThreads], ctx[kThreads], q0[kThreads], nn[kThreads];
    } att;
  };
  __shared__ Shared sh;
  const int tid = threadIdx.x, lane = tid & 31;
  if (p.with_accept && !p.accept_apart) plan_accept_clear(sh.acc);
  // the launch's status word starts clear (every kernel of the call reports into it)
  if (tid == 0) {
    p.status->code = 0;
    p.status->pad = 0;
    p.status->request_id = 0;
    s_sum[0] = s_sum[1] = 0;
    s_valid = 0;
  }
  s_hist[tid] = 0;
  static_assert(kOrderBuckets == kThreads, "one bucket per thread");
  const int g = p.Hq > 0 && p.Hkv > 0 ? p.Hq / p.Hkv : 1;
  const int64_t cap_tokens = (int64_t)p.max_blocks_per_seq * p.block_size;
  // with at most kThreads requests, pass 3 reuses what this thread read and decided here
  const bool one = p.B <= kThreads;
  int32_t my_k = 0, my_ctx = 0, my_q0 = 0;
  bool my_ok = false;

  // pass 1: offsets (negative lengths count as 0) and validation.  A request's first query row is its
  // first draft row plus its index, so one scan gives both.
  int64_t carry_d = 0;
  for (int base = 0; base < p.B; base += kThreads) {
    const int r = base + tid;
    int64_t k = 0, n = 0;
    int bad = 0;
    if (r < p.B) {
      k = p.draft_lens[r];
      my_k = (int32_t)k;
      const int64_t c = p.with_attention ? p.context_lens[r] : 0;
      my_ctx = (int32_t)c;
      if (k < 0) { bad = WISP_DEV_BAD_LENGTH; k = 0; }
      if (!bad && k > kMaxDraft) bad = WISP_DEV_UNSUPPORTED;
      if (p.with_attention) {
        if (!bad && (c < 0 || c + k + 1 > cap_tokens)) bad = WISP_DEV_BAD_LENGTH;
        if (!bad && (int64_t)g * (k + 1) > kMaxRowsPerHead) bad = WISP_DEV_UNSUPPORTED;
        n = bad ? 0 : c + k + 1;
      }
    }
    // the scan in 32 bits (no sum of 1024 lengths up to 2^20 overflows), or in two parts of 16 bits when a
    // length, refused itself but counted in the offsets, is longer.  (The first barrier is also what makes
    // the cleared shared and status words visible.)
    int64_t incl, td;
    if (!__syncthreads_or(k > (1 << 20))) {
      int t;
      incl = block_scan((int)k, s_w[base / kThreads % 2], &t);
      td = t;
    } else {
      int tl, th;
      const int lo = block_scan((int)k & 0xffff, s_w[2], &tl);
      const int hi = block_scan((int)(k >> 16), s_w[base / kThreads % 2], &th);
      incl = lo + ((int64_t)hi << 16);
      td = tl + ((int64_t)th << 16);
    }
    const unsigned vm = __ballot_sync(0xffffffffu, n > 0);
    const unsigned n_lo = __reduce_add_sync(0xffffffffu, (unsigned)n & 0xffffu), n_hi = __reduce_add_sync(0xffffffffu, (unsigned)n >> 16);
    if (lane == 0 && vm) {
      atomicAdd(&s_sum[0], (unsigned long long)n_lo + ((unsigned long long)n_hi << 16));
      atomicAdd(&s_valid, __popc(vm));
    }
    if (p.split_sms) {  // (at most 2^25 tiles and 4 row groups each: a warp's sum fits 32 bits)
      const int nrg = n > 0 ? (g * ((int)k + 1) + p.max_rows_item - 1) / p.max_rows_item : 0;
      const unsigned t = __reduce_add_sync(0xffffffffu, (unsigned)((n + kOrderTile - 1) / kOrderTile) * nrg);
      if (lane == 0 && t) atomicAdd(&s_sum[1], (unsigned long long)t);
    }
    if (r < p.B) {
      const int64_t d0 = carry_d + incl - k, q0 = d0 + r;
      // a request whose rows fall outside the caller's buffers is never touched
      if (!bad && (q0 + k + 1 > p.total_q_rows || (p.total_draft >= 0 && d0 + k > p.total_draft)))
        bad = WISP_DEV_BAD_LENGTH;
      p.q_row_start[r] = (int32_t)min64(q0, INT32_MAX);
      p.draft_start[r] = (int32_t)min64(d0, INT32_MAX);
      p.req_flag[r] = bad ? REQ_BAD : REQ_OK;
      my_q0 = (int32_t)min64(q0, INT32_MAX);
      my_ok = !bad;
      if (bad) report(p.status, bad, p.request_ids, r);
    }
    carry_d += td;
  }
  if (p.B == 0) __syncthreads();
  if (tid == 0) {
    p.q_row_start[p.B] = (int32_t)min64(carry_d + p.B, INT32_MAX);
    p.draft_start[p.B] = (int32_t)min64(carry_d, INT32_MAX);
    if (carry_d + p.B != p.total_q_rows || (p.total_draft >= 0 && carry_d != p.total_draft)) {
      // the caller sized its buffers with other totals: flag it (requests that still fit run)
      atomicCAS(&p.status->code, 0, (int32_t)WISP_DEV_BAD_LENGTH);
    }
  }
  if (p.with_accept && !p.accept_apart) plan_accept(p, sh.acc, one, my_k, my_ok);
  if (!p.with_attention) return;
  __syncthreads();

  // SMs for the attention in a step whose acceptance pass runs beside it.  Both kernels are
  // persistent and each fills an SM's shared memory, so the acceptance CTAs start on the SMs the
  // attention leaves, and the step ends with the later of the two: the split that lets both end
  // together is the attention's share of the work.  Times on all SMs, in ns: 3.2 (D = 128; 2.7 at
  // 64) per pass over a KV tile of 64 tokens, 47 with an fp32 cache; 35.2 us, 12.3 per logit row and
  // 0.29 per 1000 logits.  The constants are a fit to the split measured best (32 to 152 of 152 SMs) for
  // 24 batches of 1 to 512 requests, contexts of 64 to 128K tokens and vocabularies of 4K to 152K.  With
  // fewer (request, head) pairs than SMs the tensor-core kernel's tiles count 3/2 times and 10 us more: its
  // sequences are cut into a fixed number of items (pass 2), which cost a merge each and fill a small
  // share in more rounds (fitted to the best share of 14 such batches).
  // Steps on GB300 with all SMs for the attention first and with this split: 256 requests 653, 588 us; 512
  // requests 1266, 1183; 32 requests 116, 92; 16 requests 94, 82; 8 requests with an fp32 cache 123, 109;
  // 512 short requests with 4K tokens of vocabulary 437, 360; 300 requests with 8K 823, 758; one
  // request of 100K tokens 123, 103.  At least a quarter of the SMs: a small batch's step is bound by
  // the acceptance's chain, which more SMs do not shorten.  The fp32 kernel's time is in proportion to
  // 1 / SMs, so beside less than 1/16 of its work the acceptance waits (4 requests of 30-60K: 503 us; 524
  // with 144 SMs).
  const int sms = max(1, p.target_items / kItemsPerSM);
  const bool many_pairs = (int64_t)s_valid * p.Hkv >= sms;
  int na = sms;
  if (p.split_sms && s_sum[1] > 0) {
    float att = (p.kv_f32 ? 47.0f : 2.24f + 0.0075f * (float)p.D) * (float)s_sum[1] * (float)p.Hkv;
    if (!p.kv_f32 && !many_pairs) att = 1.5f * att + 10000.0f;
    const float acc = 35200.0f + (12.3f + 0.29e-3f * (float)p.V) * (float)p.total_q_rows;
    if (!p.kv_f32 || att < 16.0f * acc) na = max((sms + 3) / 4, min(sms, (int)((float)sms * (att / (att + acc)) + 0.5f)));
  }
  // pass 2: chunk length.  With at least as many (request, head) pairs as SMs, a longest-first
  // order balances whole sequences: only a sequence longer than 5/4 of the average work per SM
  // is cut (a split costs a merge of its chunks).  With fewer pairs than SMs, sequences are cut
  // into about kItemsPerSM items per SM.  The fp32 kernel's time also grows with the item's rows, which
  // the order does not see, so it gets items of at most 2/3 of the average (32 requests of 512-4096
  // tokens: 307 us at 5/4, 290 at 2/3, 302 at 1/2; the tensor-core kernel there: 68, 80, 83 us).  All SMs
  // count, also in a step that gives the attention a share of them: where a sequence is cut decides the
  // last bits of its outputs, and those do not depend on the acceptance's sizes.
  const int64_t work = (int64_t)s_sum[0] * p.Hkv;
  const int64_t goal = many_pairs ? sms : p.target_items;
  int64_t chunk = ceil_div(work, goal);
  if (many_pairs) chunk = p.kv_f32 ? chunk - chunk / 3 : chunk + chunk / 4;
  chunk = max64(chunk, kMinChunk);
  chunk = min64((chunk + kChunkAlign - 1) / kChunkAlign * kChunkAlign, (int64_t)1 << 30);  // (a sequence is shorter)

  // pass 3: the requests' items and partial slots (request-major, then KV head, then row group, then chunk)
  // and the histogram of the items' lengths; pass 4: the items, each written at its place in the dispatch
  // order, longest first (counting sort on the tile count), so that the persistent kernel ends with its
  // shortest items and its CTAs finish close together.  Per chunk of kThreads requests: one thread per
  // request sizes its items (block scans into shared arrays), then consecutive threads take consecutive
  // items (the request found by binary search over the chunk's first items).  With one chunk of requests
  // pass 4 finds the shared arrays as pass 3 left them and its items' requests in registers.
  int32_t *s_first = sh.att.first;  // the chunk's requests' first items, relative
  // per request of the chunk: query rows, chunks (0: no items), first partial, context, first
  // query row, keys
  int32_t *s_rows = sh.att.rows, *s_ch = sh.att.ch, *s_pf = sh.att.pf, *s_ctx = sh.att.ctx, *s_q0 = sh.att.q0, *s_nn = sh.att.nn;
  auto bucket_of = [&](int tokens) -> int {  // bucket 0: the longest
    return kOrderBuckets - 1 - min((tokens + kOrderTile - 1) / kOrderTile, kOrderBuckets - 1);
  };
  int64_t item_carry = 0, poff_carry = 0;
  int ti = 0;  // items of the chunk of requests
  auto size_requests = [&](int base, bool refuse) {
    const int r = base + tid;
    int n = 0, chunks = 0, rows = 0, nrg = 1, rows0 = 0, ctx_r = 0;
    if (r < p.B && (one ? my_ok : p.req_flag[r] == REQ_OK)) {
      const int32_t k_r = one ? my_k : p.draft_lens[r];
      ctx_r = one ? my_ctx : p.context_lens[r];
      n = ctx_r + k_r + 1;
      chunks = (int)(((unsigned)n + (unsigned)chunk - 1) / (unsigned)chunk);
      rows = g * (k_r + 1);
      nrg = (rows + p.max_rows_item - 1) / p.max_rows_item;
      rows0 = (rows + nrg - 1) / nrg;  // every group but the last; rows <= row_groups * max_rows_item
    }
    const int nitems = chunks * p.Hkv * nrg;
    // each split item's partials start on a 16-byte boundary (vector stores)
    const int slot = (rows0 * (p.D + 2) + 3) / 4 * 4;
    const int pfl = chunks > 1 ? nitems * slot : 0;
    int tp;  // (a batch's items and partials are bounded by max_items and partial_cap: 32 bits hold them)
    const int ii = block_scan(nitems, s_w[3], &ti), ip = block_scan(pfl, s_w[4], &tp);
    bool fits = false;
    if (r < p.B) {
      fits = item_carry + ii <= p.max_items && poff_carry + ip <= p.partial_cap;
      if (!fits && nitems > 0 && refuse) {
        // cannot happen with the host's bounds; refuse the request rather than overflow
        p.req_flag[r] = REQ_BAD;
        report(p.status, WISP_DEV_UNSUPPORTED, p.request_ids, r);
      }
      if (refuse) p.req_chunks[r] = fits ? chunks : 0;
    }
    s_first[tid] = ii - nitems;
    if (tid == kThreads - 1) s_first[kThreads] = ti;
    s_rows[tid] = rows;
    s_ch[tid] = fits ? chunks : 0;
    s_pf[tid] = (int32_t)min64(poff_carry + ip - pfl, INT32_MAX);
    s_ctx[tid] = ctx_r;
    s_q0[tid] = r < p.B ? (one ? my_q0 : p.q_row_start[r]) : 0;
    s_nn[tid] = n;
    poff_carry += tp;
    __syncthreads();
  };
  auto request_of = [&](int i) -> int {  // the last one whose first item is <= i
    int lo = 0, hi = kThreads - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (s_first[mid] <= i) lo = mid;
      else hi = mid - 1;
    }
    return lo;
  };
  // item i's chunk of keys and its bucket (a refused request's items are empty and come last)
  auto keys_of = [&](int i, int lo, int &t0, int &t1) -> int {
    const int ch = s_ch[lo];
    t0 = t1 = 0;
    if (ch > 0) {
      const int64_t c = (unsigned)(i - s_first[lo]) % (unsigned)ch;
      t0 = (int)(c * chunk);
      t1 = (int)min64(s_nn[lo], (c + 1) * chunk);
    }
    return bucket_of(t1 - t0);
  };
  int keep[kKeep];  // the requests of this thread's first items
#pragma unroll
  for (int x = 0; x < kKeep; ++x) keep[x] = 0;
  for (int base = 0; base < p.B; base += kThreads) {
    size_requests(base, one);
    // per (request, head, row group) finished-chunk counters of the chunk's requests: zeroed, coalesced
    const int64_t pd0 = (int64_t)base * p.Hkv * p.row_groups;
    const int64_t pd1 = (int64_t)min(p.B, base + kThreads) * p.Hkv * p.row_groups;
    for (int64_t x = pd0 + tid; x < pd1; x += kThreads) p.pair_done[x] = 0;
    int x = 0;
    for (int i = tid; i < ti; i += kThreads, ++x) {
      if (item_carry + i >= p.max_items) break;  // (a request refused for want of room)
      int t0, t1;
      const int lo = request_of(i);
      atomicAdd(&s_hist[keys_of(i, lo, t0, t1)], 1);
#pragma unroll
      for (int y = 0; y < kKeep; ++y)
        if (y == x) keep[y] = lo;
    }
    item_carry += ti;
    __syncthreads();  // the shared arrays are rewritten by the next chunk; the histogram is complete after the last
  }
  const int n_items = (int)min64(item_carry, p.max_items);
  {
    const int h = s_hist[tid];
    int tot;
    s_hist[tid] = block_scan(h, s_w[5], &tot) - h;
  }
  __syncthreads();
  item_carry = 0;
  if (!one) poff_carry = 0;
  for (int base = 0; base < p.B; base += kThreads) {
    if (!one) size_requests(base, true);
    int x = 0;
    for (int i = tid; i < ti; i += kThreads, ++x) {
      if (item_carry + i >= p.max_items) break;
      int lo = -1;
      if (one) {
#pragma unroll
        for (int y = 0; y < kKeep; ++y)
          if (y == x) lo = keep[y];
      }
      if (lo < 0) lo = request_of(i);
      WorkItem it;
      const int bucket = keys_of(i, lo, it.t0, it.t1);
      const int ch = max(1, s_ch[lo]);
      const int rws = s_rows[lo];
      const int ng = max(1, (rws + p.max_rows_item - 1) / p.max_rows_item);
      const int r0 = (rws + ng - 1) / ng;
      const int j = i - s_first[lo];  // (head, row group, chunk) in that order
      const int hg = j / ch, c = j - hg * ch;
      const int h = hg / ng, rg = hg - h * ng;
      const int slot = (r0 * (p.D + 2) + 3) / 4 * 4;
      it.r = base + lo;
      it.h = h;
      it.row0 = rg * r0;
      it.rows = min(r0, rws - rg * r0);
      it.rg = rg;
      it.nrg = ng;
      it.poff = ch > 1 ? (int32_t)(s_pf[lo] + (int64_t)j * slot) : -1;
      it.pbase = it.poff - c * slot;
      it.q0 = s_q0[lo];
      it.ctx = s_ctx[lo];
      p.items[atomicAdd(&s_hist[bucket], 1)] = it;
    }
    item_carry += ti;
    if (!one) __syncthreads();  // the shared arrays are rewritten by the next chunk
  }

  if (tid == 0) {
    PlanHeader hd;
    hd.n_items = n_items;
    hd.chunk_len = (int32_t)chunk;
    hd.partial_floats = (int32_t)min64(poff_carry, p.partial_cap);
    hd.next_item = 0;
    hd.attn_ctas = na;
    for (int i = 0; i < 3; ++i) hd.pad[i] = 0;
    *p.header = hd;
  }
}

// The acceptance part of the plan on its own (a step: it runs on the acceptance pass's stream, so
// that the attention, which waits for the whole planner grid, does not wait for it).  Reads what
// plan_kernel's first pass wrote (flags and offsets).
__global__ void __launch_bounds__(kThreads, 1) plan_accept_kernel(const PlanParams p) {
  // the acceptance kernel may be placed and set itself up now (it waits for this grid)
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  __shared__ AcceptPlan sh;
  plan_accept_clear(sh);
  const int r = threadIdx.x;
  const bool one = p.B <= kThreads, mine = one && r < p.B;
  const int k = mine ? p.draft_lens[r] : 0;
  const bool ok = mine && p.req_flag[r] == REQ_OK;
  __syncthreads();
  plan_accept(p, sh, one, k, ok);
}

}  // namespace wisp
