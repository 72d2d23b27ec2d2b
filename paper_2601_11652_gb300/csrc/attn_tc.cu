// attn_tc.cu -- tensor-core paged GQA attention for the verification forward (bf16 KV).
//
// Same contract as attn_f32.cu (Sec. 4.4-4.5: request r's k+1 new queries over its
// L_total = L_cached + L_new paged keys, query j seeing keys 0..c_r + j), built for sm_103a.
//
// A verification item has few query rows (g * (k+1), at most 64 per item) and many keys, so the
// products run transposed: the keys are the MMA's M dimension and the query rows its N.
//   S^T = K Q^T       (M = 128 keys of a tile, N = the item's rows rounded up to 16, K = D)
//   O^T += V^T P^T    (M = D, N = rows, K = 128 keys)
// Nothing is replicated to fill the 128-row MMA, and the tensor core reads each K and V tile from
// shared memory once.
//
// Persistent CTAs (one per SM) take work items (request, KV head, key chunk, row group) from a
// global counter, in the planner's longest-first order.  Warp roles in a CTA:
//   * warp 2 takes the next item just in time (when the K producer is three tiles from the end of what
//     is published) and publishes it to the other warps through a 4-slot shared ring;
//   * warp 17 copies an item's query rows into one of two shared Q buffers (128-byte-swizzled, K-major:
//     the B operand of S^T);
//   * warps 0 and 3 (K and V producers) stream the item's K and V tiles of 128 tokens with TMA
//     tiled loads into two rings: one 16 KB box per 64-wide half of the head dim when the tile's
//     eight 16-token blocks are consecutive in the pool, else one 2 KB box per block; blocks past
//     the item read as zeros (out-of-range box).  A K stage is free again once S^T of its tile is
//     done, a V stage once its PV product is;
//   * warps 1 and 16 (one thread of each) issue tcgen05.mma: warp 1 S^T into one of two TMEM tiles
//     (key t in TMEM lane t, query row j in column j), warp 16 O^T into the item's TMEM accumulator
//     (head-dim index d in lane d, row j in column j; two accumulators alternating between items);
//   * warps 4-7 and 12-15 (softmax): the first group takes the first half of an item's rows, the
//     second the rest; within a group one warp per TMEM lane quadrant, i.e. 32 keys of each tile per
//     warp: a thread holds one key's scores for the group's rows.  The rows' reference maxima are
//     those of the item's first tile and stay fixed.  Each thread writes its key's part of the P row
//     (bf16, MN-major, swizzled: the B operand of the PV product) and keeps its share of every row sum.
//     An item with a P past kMaxP is taken again, its true maxima first: see kMaxP;
//   * warps 8-11 (epilogue) add the row-sum shares, read O^T from TMEM and write the normalised
//     output or, for a split item, the (O, m, l) partials; the last chunk of a split
//     (request, head, row group) to finish merges all its chunks.  This runs while the softmax
//     warps are already on the next item.
// What bounds it: the K and V stream (HBM).  An SM's own limit is the softmax warps' chain per tile
// (read S^T, P, publish): 0.77 us a 128-key tile up to 32 query rows and 0.90 us at 64 with K and V in L2,
// against the 1.47 us that a tile's 64 KB take at an SM's share of the copy rate (D = 128; at 64 the
// tile's 32 KB take 0.74).  An item of one tile takes 4 us (its claim, Q copy, first-tile references and
// epilogue overlap its neighbours').
//
// Every mbarrier wait is bounded in time; an expired wait records WISP_DEV_TIMEOUT and the CTA
// drains.  No named barrier is used: a warp that gives up cannot leave the others blocked, and the
// TMEM is freed once every warp has arrived on a final mbarrier.
#include "attn_merge.cuh"
#include "sm100_ptx.cuh"

#include <cudaTypedefs.h>
#include <cstring>
#include <mutex>
#include <type_traits>

namespace wisp {

namespace {

constexpr int kBT = 128;            // KV tokens per tile (the M of S^T)
constexpr int kNR = kTcRowsPerItem; // query rows per item at most (64: the planner cuts larger sets)
constexpr int kThreads = 640;       // warps 0-3 K producer, S^T issuer, item loader and V producer; 4-7 softmax
                                    // (first half of the rows); 8-11 epilogue; 12-15 softmax (second half);
                                    // 16 PV issuer; 17 Q loader (18, 19: registers are allotted per four warps)
constexpr int kSoftmaxWarps = 8;
constexpr uint32_t kTmemCols = 256; // S^T[2] at columns 0 / 64, O^T[2] at 128 / 192
constexpr long long kWaitCycles = 4000000000LL;  // about two seconds: a wait that long is a failure
// Largest P = 2^(s - m) an item may hold: m is the maximum of a row's first tile, so later scores may
// exceed it.  P (bf16), its row sums and O (fp32) keep their relative precision at any exponent; up to
// 2^64 nothing comes near the fp32 range (2^64 x 2^30 keys x |V| < 2^33).  An item that goes past it, or
// that has a row whose first tile scores -inf throughout, writes nothing: the epilogue hands it back to
// the item loader, which publishes it again for two passes over its keys, S^T alone for the rows' true
// maxima and then the ordinary one against those: 24 requests of 8192 tokens at 64 query rows, every item taken
// again, 389 us against 164 (D = 64: 290 against 117).  Whether an item is taken again follows from its
// own scores alone, so outputs repeat to the bit.
constexpr float kMaxP = 0x1p64f;
constexpr int kRedo = 8;            // items waiting to be taken again, at most: those published and undecided, RING + 1
constexpr uint32_t kAhead = 3;      // the item loader takes the next item when the K producer is this many tiles from
                                    // the end of what is published
static_assert(kNR == 64, "TMEM and shared-memory layout assume 64 rows per item");

template <int D>
struct Cfg {
  static constexpr int HALVES = D / 64;
  static constexpr int HALF = kBT * 128;        // one 64-wide half of a K / V tile: [128 tokens][128 B]
  static constexpr int KV_TILE = HALVES * HALF; // K (or V) of one tile
  static constexpr int QHALF = kNR * 128;       // one half of a Q buffer: [64 rows][128 B]
  static constexpr int Q_BYTES = HALVES * QHALF;
  static constexpr int P_BYTES = kBT * kNR * 2; // P^T: [128 tokens][64 rows] bf16
  static constexpr int NSK = D == 128 ? 2 : 4;  // K ring stages
  static constexpr int NSV = D == 128 ? 2 : 4;  // V ring stages
  static constexpr int NQ = 2;                  // Q buffers: item li's rows in buffer li % NQ
  static constexpr int NP = 2;                  // P buffers: P(n) in buffer n % NP
  static constexpr int RING = 4;                // slots of the item ring
  static constexpr int OFF_Q = 0;
  static constexpr int OFF_K = OFF_Q + NQ * Q_BYTES;
  static constexpr int OFF_V = OFF_K + NSK * KV_TILE;
  static constexpr int OFF_P = OFF_V + NSV * KV_TILE;
  static constexpr int OFF_BAR = OFF_P + NP * P_BYTES;
  static constexpr int N_BAR = 2 * NSK + 2 * NSV + 8 + 2 * NP + 6 + 1 + 2 * RING + 4;
  static constexpr int OFF_MW = (OFF_BAR + N_BAR * 8 + 15) / 16 * 16;  // float [8][32] per warp: minus the rows' references
  static constexpr int OFF_RED = OFF_MW + kSoftmaxWarps * 32 * 4;      // float [2][4][64] first-tile maxima per quadrant
  static constexpr int OFF_HL = OFF_RED + 2 * 4 * kNR * 4;             // float [2][4][64] row-sum shares per quadrant
  static constexpr int OFF_HM = OFF_HL + 2 * 4 * kNR * 4;              // float [2][64] row reference maxima
  static constexpr int OFF_MISC = OFF_HM + 2 * kNR * 4;                // tmem base, flags, counters
  static constexpr int OFF_RING = OFF_MISC + 80;                       // RING x (index, passes, WorkItem)
  static constexpr int SMEM = OFF_RING + RING * 64 + 1024;             // + slack to align the base to 1024
  static_assert(SMEM <= 227 * 1024, "shared memory of one CTA on sm_103a");
  static_assert(RING + 1 <= kRedo && OFF_RING % 16 == 0, "item ring");
  static_assert(OFF_K % 1024 == 0 && OFF_V % 1024 == 0 && OFF_P % 1024 == 0, "swizzled buffers need 1 KB alignment");
};

// The CTA's mbarriers: shared-memory addresses at constant offsets from one base.
template <int D>
struct Bars {
  using C = Cfg<D>;
  uint32_t base;
  __device__ __forceinline__ uint32_t at(int i) const { return base + 8 * i; }
  static constexpr int K_FULL = 0, K_EMPTY = C::NSK, V_FULL = 2 * C::NSK, V_EMPTY = V_FULL + C::NSV;
  static constexpr int Q_FULL = V_EMPTY + C::NSV, Q_EMPTY = Q_FULL + 2, S_FULL = Q_EMPTY + 2, S_EMPTY = S_FULL + 2;
  static constexpr int P_FULL = S_EMPTY + 2;      // [NP] per P buffer
  static constexpr int O_FULL = P_FULL + C::NP;   // [NP] per P buffer: PV of tiles n with n % NP == b
  static constexpr int O_EMPTY = O_FULL + C::NP;  // [2] per O buffer: its epilogue is done
  static constexpr int O_DONE = O_EMPTY + 2;      // [2] per O buffer: the item's last PV is done
  static constexpr int EP_FULL = O_DONE + 2;      // [2] per O buffer: the softmax warps handed the item over
  static constexpr int MMA_DONE = EP_FULL + 2;    // the two MMA issuers, at the end
  static constexpr int IT_FULL = MMA_DONE + 1, IT_EMPTY = IT_FULL + C::RING;
  static constexpr int EGRP = IT_EMPTY + C::RING; // the epilogue warps
  static constexpr int RED = EGRP + 1;            // [2] per softmax group: its four warps, once per item (first-tile maxima)
  static constexpr int FIN = RED + 2;             // every warp, once: its last access to TMEM is done
  static_assert(FIN + 1 <= C::N_BAR, "barrier count");
  __device__ __forceinline__ uint32_t k_full(int i) const { return at(K_FULL + i); }
  __device__ __forceinline__ uint32_t k_empty(int i) const { return at(K_EMPTY + i); }
  __device__ __forceinline__ uint32_t v_full(int i) const { return at(V_FULL + i); }
  __device__ __forceinline__ uint32_t v_empty(int i) const { return at(V_EMPTY + i); }
  __device__ __forceinline__ uint32_t q_full(int i) const { return at(Q_FULL + i); }
  __device__ __forceinline__ uint32_t q_empty(int i) const { return at(Q_EMPTY + i); }
  __device__ __forceinline__ uint32_t s_full(int i) const { return at(S_FULL + i); }
  __device__ __forceinline__ uint32_t s_empty(int i) const { return at(S_EMPTY + i); }
  __device__ __forceinline__ uint32_t p_full(int i) const { return at(P_FULL + i); }
  __device__ __forceinline__ uint32_t o_full(int i) const { return at(O_FULL + i); }
  __device__ __forceinline__ uint32_t o_empty(int i) const { return at(O_EMPTY + i); }
  __device__ __forceinline__ uint32_t o_done(int i) const { return at(O_DONE + i); }
  __device__ __forceinline__ uint32_t ep_full(int i) const { return at(EP_FULL + i); }
  __device__ __forceinline__ uint32_t it_full(int i) const { return at(IT_FULL + i); }
  __device__ __forceinline__ uint32_t it_empty(int i) const { return at(IT_EMPTY + i); }
  __device__ __forceinline__ uint32_t red(int i) const { return at(RED + i); }
  __device__ __forceinline__ uint32_t mma_done() const { return at(MMA_DONE); }
  __device__ __forceinline__ uint32_t egrp() const { return at(EGRP); }
  __device__ __forceinline__ uint32_t fin() const { return at(FIN); }
};

__device__ __forceinline__ bool wait_bar(uint32_t b, uint32_t parity, volatile int *abort) {
  if (ptx::mbar_try_wait(b, parity)) return true;
  const long long t0 = clock64();
  while (true) {
    if (ptx::mbar_try_wait(b, parity)) return true;
    if (*abort) return false;
    if (clock64() - t0 > kWaitCycles) {
      *abort = 1;
      return false;
    }
  }
}

__device__ __forceinline__ bool item_ok(const AttnParams &p, const WorkItem &w) {
  // (a refused request's items are empty)
  return w.r >= 0 && w.r < p.B && w.t1 > w.t0 && w.rows > 0 && w.rows <= kNR &&
         w.row0 >= 0 && w.nrg >= 1 && w.nrg <= p.row_groups && w.rg >= 0 && w.rg < w.nrg;
}

// Transposing sum over the 32 lanes of a warp (v is consumed): on return lane i holds the sum over all
// lanes of v[i].  31 shuffles for 32 values.
__device__ __forceinline__ float warp_transpose_sum(float (&v)[32], int lane) {
#pragma unroll
  for (int w = 16; w >= 1; w >>= 1) {
    const bool up = (lane & w) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float keep = up ? v[i + w] : v[i];
      const float send = up ? v[i] : v[i + w];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, w);
    }
  }
  return v[0];
}

__device__ __forceinline__ uint32_t bmax2(uint32_t a, uint32_t b) {  // NaN never wins
  uint32_t r;
  asm("max.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

}  // namespace

template <int D>
__global__ void __launch_bounds__(kThreads, 1)
    attn_tc_kernel(const __grid_constant__ AttnParams p, const __grid_constant__ CUtensorMap tmk,
                   const __grid_constant__ CUtensorMap tmv, const __grid_constant__ CUtensorMap tmk8,
                   const __grid_constant__ CUtensorMap tmv8) {
  using C = Cfg<D>;
  extern __shared__ uint8_t smem_raw[];
  // aligned by an offset, not through an integer: the compiler then still knows the address space
  uint8_t *smem = smem_raw + ((1024u - (ptx::smem_u32(smem_raw) & 1023u)) & 1023u);
  const uint32_t sbase = ptx::smem_u32(smem);
  const Bars<D> B{sbase + C::OFF_BAR};
  float *s_mw = reinterpret_cast<float *>(smem + C::OFF_MW);
  float *s_red = reinterpret_cast<float *>(smem + C::OFF_RED);
  float *s_hl = reinterpret_cast<float *>(smem + C::OFF_HL);
  float *s_hm = reinterpret_cast<float *>(smem + C::OFF_HM);
  uint32_t *s_tmem = reinterpret_cast<uint32_t *>(smem + C::OFF_MISC);
  volatile int *s_abort = reinterpret_cast<volatile int *>(smem + C::OFF_MISC + 4);
  volatile int *s_last = reinterpret_cast<volatile int *>(smem + C::OFF_MISC + 8);
  volatile uint32_t *s_issued = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_MISC + 12);  // K tiles issued
  // items decided by the epilogue (to be taken again, or not), and those to be taken again: their number and a ring
  // of their indexes.  Written by one lane of warp 8, read by one lane of warp 2.
  volatile uint32_t *s_decided = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_MISC + 16);
  volatile uint32_t *s_nredo = reinterpret_cast<volatile uint32_t *>(smem + C::OFF_MISC + 20);
  volatile int *s_redo = reinterpret_cast<volatile int *>(smem + C::OFF_MISC + 24);
  volatile uint8_t *s_ovf = smem + C::OFF_MISC + 64;  // [2][8] per O buffer and softmax warp: the item must be taken again
  struct RingSlot {
    int it;
    int passes;  // over the keys: 1, or 2 for an item that is taken again
    int pad[2];
    WorkItem w;
  };
  static_assert(sizeof(RingSlot) <= 64, "item ring slot");
  RingSlot *s_ring = reinterpret_cast<RingSlot *>(smem + C::OFF_RING);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::NSK; ++s) {
      ptx::mbar_init(B.k_full(s), 1);
      ptx::mbar_init(B.k_empty(s), 1);
    }
    for (int s = 0; s < C::NSV; ++s) {
      ptx::mbar_init(B.v_full(s), 1);
      ptx::mbar_init(B.v_empty(s), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(B.q_full(b), 1);
      ptx::mbar_init(B.q_empty(b), 1);
      ptx::mbar_init(B.s_full(b), 1);
      ptx::mbar_init(B.s_empty(b), kSoftmaxWarps);
    }
    for (int b = 0; b < C::NP; ++b) {
      ptx::mbar_init(B.p_full(b), kSoftmaxWarps);
      ptx::mbar_init(B.o_full(b), 1);
    }
    for (int b = 0; b < 2; ++b) {
      ptx::mbar_init(B.o_empty(b), 4);  // the four epilogue warps
      ptx::mbar_init(B.o_done(b), 1);
      ptx::mbar_init(B.ep_full(b), kSoftmaxWarps);
    }
    ptx::mbar_init(B.mma_done(), 2);  // the two MMA issuers
    for (int i = 0; i < C::RING; ++i) {
      ptx::mbar_init(B.it_full(i), 1);
      ptx::mbar_init(B.it_empty(i), 5 + kSoftmaxWarps + 4);  // KV producers, MMA issuers, Q loader, softmax and epilogue warps
    }
    ptx::mbar_init(B.egrp(), 4);      // the four epilogue warps
    ptx::mbar_init(B.red(0), 4);
    ptx::mbar_init(B.red(1), 4);
    ptx::mbar_init(B.fin(), kThreads / 32);
    *s_issued = 0;
    *s_abort = 0;
    *s_decided = 0;
    *s_nredo = 0;
    ptx::fence_mbar_init();
  }
  if (warp == 0 && lane == 0) {
    ptx::prefetch_tmap(&tmk);
    ptx::prefetch_tmap(&tmv);
    ptx::prefetch_tmap(&tmk8);
    ptx::prefetch_tmap(&tmv8);
  }
  __syncwarp();
  if (warp == 1) {
    ptx::tmem_alloc(s_tmem, kTmemCols);
    ptx::tmem_relinquish();
  }
  ptx::tc_fence_before();
  __syncthreads();
  ptx::tc_fence_after();
  const uint32_t tmem = *s_tmem;

  // everything above may overlap the planner (programmatic dependent launch); the plan is read
  // only once the planner's grid has completed and its writes are visible
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const int n_items = p.header->n_items;
  if ((int)blockIdx.x >= p.header->attn_ctas) {
    // the planner leaves this SM to the acceptance pass of the same step: nothing was issued yet
    if (warp == 1) ptx::tmem_dealloc(tmem, kTmemCols);
    return;
  }
  const int g = p.Hq / p.Hkv;
  // a query row's position and head: row / g for rows below 128 as a product (exact: 127 (g - 1) < 2^16)
  const unsigned gm = (65536u + g - 1) / g;
  auto div_g = [&](int row) -> int { return (int)(((unsigned)row * gm) >> 16); };

  if (warp == 0 || warp == 3) {
    // ------------------------------------------------------------------ K / V producers
    // K and V have rings of their own: a K stage is free again once S^T of its tile is done, a V
    // stage once PV is, so each tensor is fetched about as many tiles ahead of its use as its ring
    // has stages.
    const bool is_k = warp == 0;
    const uint32_t ns = is_k ? C::NSK : C::NSV;
    const CUtensorMap *tm1 = is_k ? &tmk : &tmv;
    const CUtensorMap *tm8 = is_k ? &tmk8 : &tmv8;
    const uint32_t off_t = sbase + (is_k ? C::OFF_K : C::OFF_V);
    const uint32_t full = is_k ? B.k_full(0) : B.v_full(0), empty = is_k ? B.k_empty(0) : B.v_empty(0);
    uint32_t tile_n = 0;
    bool ok = true;
    for (uint32_t j = 0; ok; ++j) {
      const int slot = j % C::RING;
      if (!wait_bar(B.it_full(slot), (j / C::RING) & 1, s_abort)) { ok = false; break; }
      const int it = s_ring[slot].it;
      const WorkItem w = s_ring[slot].w;
      const int passes = is_k ? s_ring[slot].passes : 1;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.it_empty(slot));
      if (it < 0) break;
      const int32_t *bt = p.block_tables + (int64_t)w.r * p.max_blocks_per_seq + w.t0 / 16;
      const int nblk = (w.t1 - w.t0 + 15) / 16;
      auto fetch = [&](int base) -> int {
        const int i = base + lane;
        return i < nblk ? __ldg(bt + i) : -1;
      };
      int cur = fetch(0), nxt = fetch(32);  // block ids of tiles t..t+3 and t+4..t+7
      const int ntiles = (w.t1 - w.t0 + kBT - 1) / kBT;
      for (int t = 0, left = passes * ntiles; left > 0; ++t, --left, ++tile_n) {
        if (is_k && lane == 0) *s_issued = tile_n;
        if (t == ntiles) {  // the keys once more
          t = 0;
          cur = fetch(0);
          nxt = fetch(32);
        } else if (t > 0 && (t & 3) == 0) {
          cur = nxt;
          nxt = fetch(32 * ((t >> 2) + 1));
        }
        const int s = (int)(tile_n % ns);
        const uint32_t round = tile_n / ns;
        if (!wait_bar(empty + 8 * s, (round & 1) ^ 1, s_abort)) { ok = false; break; }
        if (lane == 0) ptx::mbar_arrive_expect_tx(full + 8 * s, C::KV_TILE);
        __syncwarp();
        const int bi = lane & 7;  // block of the tile this lane looks after
        int bid = __shfl_sync(0xffffffffu, cur, (8 * t + bi) & 31);
        const int rel = 8 * t + bi;
        bool valid = rel < nblk && bid >= 0 && bid < p.num_blocks;
        if (is_k && lane < 8 && rel < nblk && !valid) report(p.status, WISP_DEV_BAD_BLOCK, p.request_ids, w.r);
        const int b0 = __shfl_sync(0xffffffffu, bid, 0);
        // eight consecutive valid blocks: one 16 KB box per (tensor, half) with the 8-block maps
        const unsigned contig = __ballot_sync(0xffffffffu, lane < 8 && valid && bid == b0 + lane);
        if (contig == 0xFFu) {
          if (lane == 0) {
#pragma unroll
            for (int hf = 0; hf < C::HALVES; ++hf) {
              ptx::tma_load_4d(off_t + s * C::KV_TILE + hf * C::HALF, tm8, full + 8 * s, hf * 64, 0, w.h, b0);
            }
          }
        } else if (lane < 8) {
          if (!valid) bid = p.num_blocks;  // past the item (or invalid): out-of-range box, reads zeros
#pragma unroll
          for (int hf = 0; hf < C::HALVES; ++hf) {
            const uint32_t off = s * C::KV_TILE + hf * C::HALF + lane * (16 * 128);
            ptx::tma_load_4d(off_t + off, tm1, full + 8 * s, hf * 64, 0, w.h, bid);
          }
        }
      }
    }
    if (!ok && lane == 0) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, 0);
    // drain: every stage issued must land before the CTA's shared memory goes away
    if (lane == 0) {
      for (uint32_t k = 0; k < ns && k < tile_n; ++k) {
        const uint32_t n = tile_n - 1 - k;
        const long long t0 = clock64();
        while (!ptx::mbar_try_wait(full + 8 * (n % ns), (n / ns) & 1) && clock64() - t0 < kWaitCycles) {
        }
      }
    }
  } else if (warp == 2) {
    // ------------------------------------------------------------------ item loader
    uint32_t published = 0;           // K tiles of the items published so far
    uint32_t items = 0, redone = 0;   // (lane 0) items published, and those of them taken again
    bool left = true;                 // (lane 0) the plan may have items left
    bool ok = true;
    for (uint32_t j = 0; ok; ++j) {
      // next valid work item: publish it to the other warps.  Items are taken just in time, so the work
      // counter balances the CTAs to the end, but early enough to hide the way from the claim to the first
      // load: when the K producer is kAhead tiles from the end of what is published, which for items of
      // a tile or two means several items ahead.  Items to be taken again go first.  The end is published
      // once every item is decided, before the last one's epilogue.
      const int slot = j % C::RING;
      for (const long long g0 = clock64(); published > *s_issued + kAhead;) {
        if (*s_abort || clock64() - g0 > kWaitCycles) {
          *s_abort = 1;
          ok = false;
          break;
        }
        __nanosleep(100);
      }
      if (!ok) break;
      if (!wait_bar(B.it_empty(slot), ((j / C::RING) & 1) ^ 1, s_abort)) { ok = false; break; }
      int tiles = 0;
      if (lane == 0) {
        int it = -1, passes = 1;
        WorkItem w;
        if (left && redone == *s_nredo) {
          do {
            it = atomicAdd(&p.header_mut->next_item, 1);
            if (it >= n_items) { it = -1; break; }
            w = p.items[it];
          } while (!item_ok(p, w));
          left = it >= 0;
        }
        if (it < 0) {  // an item to be taken again, or the end
          uint32_t seen = 0;
          for (long long g0 = clock64();;) {
            const uint32_t decided = *s_decided;
            __threadfence_block();  // and with them what they ask for
            if (redone != *s_nredo) {
              __threadfence_block();
              it = s_redo[redone++ % kRedo];
              w = p.items[it];
              passes = 2;
              break;
            }
            if (decided == items) break;
            if (decided != seen) g0 = clock64();
            seen = decided;
            if (*s_abort || clock64() - g0 > kWaitCycles) {
              *s_abort = 1;
              break;
            }
            __nanosleep(32);
          }
        }
        s_ring[slot].it = it;
        if (it >= 0) {
          s_ring[slot].w = w;
          s_ring[slot].passes = passes;
          tiles = passes * ((w.t1 - w.t0 + kBT - 1) / kBT);
          ++items;
        }
        ptx::mbar_arrive(B.it_full(slot));
      }
      tiles = __shfl_sync(0xffffffffu, tiles, 0);
      if (tiles == 0) {
        // no item left for this CTA: a kernel launched after this one as a programmatic
        // dependent may be scheduled; it still waits for this grid to finish
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
        ok = !*s_abort;
        break;
      }
      published += tiles;
    }
    if (!ok && lane == 0) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, 0);
  } else if (warp == 17) {
    // ------------------------------------------------------------------ Q loader
    // (a warp of its own: in the item loader, the copy would delay the next claim, which bounds short items)
    int li = 0;
    bool ok = true;
    for (uint32_t j = 0; ok; ++j) {
      const int slot = j % C::RING;
      if (!wait_bar(B.it_full(slot), (j / C::RING) & 1, s_abort)) { ok = false; break; }
      const int it = s_ring[slot].it;
      const WorkItem w = s_ring[slot].w;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.it_empty(slot));
      if (it < 0) break;
      const int qb = li % C::NQ;
      if (!wait_bar(B.q_empty(qb), ((li / C::NQ) & 1) ^ 1, s_abort)) { ok = false; break; }
      ++li;
      // the item's query rows -> Q[qb], row rho (query row row0 + rho = j*g + hh) at MMA row rho.
      // Loads are issued QBATCH at a time per lane before any store.  Rows past `rows` up to the
      // MMA's N only feed S^T columns that the softmax masks.
      const uint16_t *qg = static_cast<const uint16_t *>(p.q);
      uint8_t *qs = smem + C::OFF_Q + qb * C::Q_BYTES;
      constexpr int CPR = D / 8;       // 16-byte chunks per row: a lane keeps its chunk of every row it copies
      constexpr int RPI = 32 / CPR;    // rows per warp load
      constexpr int QBATCH = 8;
      const int cc = lane % CPR;
      const uint16_t *qi = qg + ((int64_t)w.q0 * p.Hq + w.h * g) * D + cc * 8;
      for (int base = lane / CPR; base < w.rows; base += RPI * QBATCH) {
        uint4 v[QBATCH];
#pragma unroll
        for (int u = 0; u < QBATCH; ++u) {
          const int row = base + u * RPI;
          if (row < w.rows) {
            const int rj = w.row0 + row, jj = div_g(rj), hh = rj - jj * g;
            v[u] = __ldg(reinterpret_cast<const uint4 *>(qi + (int64_t)(jj * p.Hq + hh) * D));
          }
        }
#pragma unroll
        for (int u = 0; u < QBATCH; ++u) {
          const int row = base + u * RPI;
          if (row < w.rows)
            *reinterpret_cast<uint4 *>(qs + (cc >> 3) * C::QHALF + row * 128 + (((cc & 7) ^ (row & 7)) << 4)) = v[u];
        }
      }
      ptx::fence_proxy_async_smem();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.q_full(qb));
    }
    if (!ok && lane == 0) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, 0);
  } else if (warp == 1 || warp == 16) {
    // ------------------------------------------------------------------ MMA issuers
    // One warp issues S^T, another PV, so that neither waits behind the other's barriers: an MMA takes
    // its issuer 45-90 cycles and a commit 100, and one thread for both would bound every item.
    const bool is_s = warp == 1;
    uint32_t n = 0;
    int li = 0;
    bool ok = true;
    for (uint32_t j = 0; ok; ++j, ++li) {
      const int slot = j % C::RING;
      if (!wait_bar(B.it_full(slot), (j / C::RING) & 1, s_abort)) { ok = false; break; }
      const int it = s_ring[slot].it;
      const int rows = s_ring[slot].w.rows, ntok = s_ring[slot].w.t1 - s_ring[slot].w.t0;
      const int passes = is_s ? s_ring[slot].passes : 1;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.it_empty(slot));
      if (it < 0) break;
      const int nt = passes * ((ntok + kBT - 1) / kBT);
      const int nrow = (rows + 15) / 16 * 16;  // the MMA's N: rows rounded up to 16
      if (is_s) {
        // S^T(n): K(n) has landed, the item's Q is loaded, the TMEM tile has been read
        const uint32_t idesc = ptx::idesc_bf16_f32(kBT, nrow, false, false);
        const int qb = li % C::NQ;
        if (!wait_bar(B.q_full(qb), (li / C::NQ) & 1, s_abort)) { ok = false; break; }
        const uint64_t qd = ptx::sdesc_sw128(sbase + C::OFF_Q + qb * C::Q_BYTES, 16, 1024);
        for (int t = 0; t < nt; ++t, ++n) {
          const int st = (int)(n % C::NSK), sb = n & 1;
          if (!wait_bar(B.k_full(st), (n / C::NSK) & 1, s_abort) ||
              !wait_bar(B.s_empty(sb), ((n >> 1) & 1) ^ 1, s_abort)) {
            ok = false;
            break;
          }
          if (lane == 0) {
            ptx::tc_fence_after();
            const uint64_t kd = ptx::sdesc_sw128(sbase + C::OFF_K + st * C::KV_TILE, 16, 1024);
#pragma unroll
            for (int ks = 0; ks < D / 16; ++ks)  // descriptor addresses are in units of 16 bytes
              ptx::umma_f16(tmem + sb * kNR, kd + (((ks >> 2) * C::HALF + (ks & 3) * 32) >> 4),
                            qd + (((ks >> 2) * C::QHALF + (ks & 3) * 32) >> 4), idesc, ks > 0);
            ptx::umma_commit(B.s_full(sb));
            ptx::umma_commit(B.k_empty(st));
            if (t == nt - 1) ptx::umma_commit(B.q_empty(qb));
          }
          __syncwarp();
        }
      } else {
        // PV(n): P(n) is published, V(n) has landed and, for an item's first tile, the O buffer has
        // been read.  A = V^T, MN-major: the head dim's 64-wide halves are HALF apart (for D = 64 both
        // MMA halves read the same half, so O^T lanes 64..127 repeat lanes 0..63 and are not used)
        const uint32_t idesc = ptx::idesc_bf16_f32(128, nrow, true, true);
        const int ob = li & 1;  // the item's O buffer
        constexpr uint32_t lbo_v = D == 128 ? C::HALF : 0;
        for (int t = 0; t < nt; ++t, ++n) {
          const int st = (int)(n % C::NSV), pb = (int)(n % C::NP);
          if ((t == 0 && !wait_bar(B.o_empty(ob), ((li >> 1) & 1) ^ 1, s_abort)) ||
              !wait_bar(B.v_full(st), (n / C::NSV) & 1, s_abort) ||
              !wait_bar(B.p_full(pb), (n / C::NP) & 1, s_abort)) {
            ok = false;
            break;
          }
          if (lane == 0) {
            ptx::tc_fence_after();
            const uint64_t vd = ptx::sdesc_sw128(sbase + C::OFF_V + st * C::KV_TILE, lbo_v, 1024);
            const uint64_t pd = ptx::sdesc_sw128(sbase + C::OFF_P + pb * C::P_BYTES, C::P_BYTES, 1024);
#pragma unroll
            for (int ks = 0; ks < kBT / 16; ++ks)
              ptx::umma_f16(tmem + 128 + ob * kNR, vd + ((ks * 16 * 128) >> 4), pd + ((ks * 16 * 128) >> 4), idesc,
                            (t > 0 || ks > 0) ? 1u : 0u);
            ptx::umma_commit(B.o_full(pb));
            ptx::umma_commit(B.v_empty(st));
            if (t == nt - 1) ptx::umma_commit(B.o_done(ob));
          }
          __syncwarp();
        }
      }
    }
    if (lane == 0) {
      if (!ok) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, 0);
      // every MMA the issuers issued must finish before the TMEM is released
      ptx::umma_commit(B.mma_done());
      const long long t0 = clock64();
      while (!ptx::mbar_try_wait(B.mma_done(), 0) && clock64() - t0 < kWaitCycles) {
      }
    }
  } else if (warp >= 8 && warp < 12) {
    // ------------------------------------------------------------------ epilogue warps
    // One warp per TMEM lane quadrant: thread d (lane d of O^T) owns head-dim index d of every row.
    // Item li's O^T (buffer li & 1) is read once the softmax warps have handed the item over and
    // its last PV is done; the output (or, for a split item, the partial O, m, l) is written, the
    // buffer released, and the last chunk of a split (request, head, row group) to finish merges
    // all of its chunks.
    const int qd = warp & 3;
    const int d = qd * 32 + lane;
    const bool dval = d < D;  // for D = 64 the upper two quadrants hold copies
    const uint32_t lane_addr = (uint32_t)(qd * 32) << 16;
    uint32_t gph = 0;
    int li = 0;
    bool ok = true;
    // barrier of the four epilogue warps (an mbarrier, so that the wait is bounded)
    auto group_sync = [&]() -> bool {
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.egrp());
      return wait_bar(B.egrp(), (gph++) & 1, s_abort);
    };
    for (uint32_t j = 0; ok; ++j) {
      const int slot = j % C::RING;
      if (!wait_bar(B.it_full(slot), (j / C::RING) & 1, s_abort)) { ok = false; break; }
      const int it = s_ring[slot].it;
      const WorkItem w = s_ring[slot].w;
      const int passes = s_ring[slot].passes;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.it_empty(slot));
      if (it < 0) break;
      const int ob = li & 1;
      const uint32_t o_col = 128 + ob * kNR;
      // the softmax warps' hand-over and the item's last PV
      if (!wait_bar(B.ep_full(ob), (li >> 1) & 1, s_abort)) { ok = false; break; }
      const bool again = passes == 1 && *reinterpret_cast<volatile unsigned long long *>(s_ovf + 8 * ob) != 0;
      if (warp == 8 && lane == 0) {
        const uint32_t nr = *s_nredo;
        if (again) {
          s_redo[nr % kRedo] = it;
          __threadfence_block();
          *s_nredo = nr + 1;
          __threadfence_block();
        }
        *s_decided = *s_decided + 1;
      }
      if (!wait_bar(B.o_done(ob), (li >> 1) & 1, s_abort)) { ok = false; break; }
      ++li;
      ptx::tc_fence_after();
      const int nc = (w.rows + 31) / 32;
      for (int c = 0; c < nc && !again; ++c) {
        uint32_t x[32];  // O^T[d][rows 32c..]
        ptx::tmem_ld32(tmem + lane_addr + o_col + 32 * c, x);
        ptx::tmem_wait_ld();
        // lane i: row 32c + i's sum (the four softmax warps' shares)
        const int jl = 32 * c + lane;
        const float *hl = s_hl + ob * 4 * kNR;
        const float lsum = hl[jl] + hl[kNR + jl] + hl[2 * kNR + jl] + hl[3 * kNR + jl];
        if (w.poff < 0) {
          const float linv = 1.0f / lsum;
          // (row pointers stepped from row to row: a division per row would bound items of a few tiles)
          int hh = w.row0 + 32 * c - div_g(w.row0 + 32 * c) * g;
          uint16_t *og = static_cast<uint16_t *>(p.out) +
                         ((int64_t)(w.q0 + div_g(w.row0 + 32 * c)) * p.Hq + w.h * g + hh) * D + d;
          const int wrap = (p.Hq - g + 1) * D;  // from a position's last head to the next one's first
#pragma unroll
          for (int i0 = 0; i0 < 32; i0 += 8) {
            if (32 * c + i0 >= w.rows) break;
#pragma unroll
            for (int i = i0; i < i0 + 8; ++i) {
              const float inv = __shfl_sync(0xffffffffu, linv, i);
              if (32 * c + i < w.rows && dval) *og = __bfloat16_as_ushort(__float2bfloat16_rn(__uint_as_float(x[i]) * inv));
              const bool last_head = hh == g - 1;
              og += last_head ? wrap : D;
              hh = last_head ? 0 : hh + 1;
            }
          }
        } else {
          float *part = p.partials + w.poff;
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const int jr = 32 * c + i;
            if (jr < w.rows && dval) __stcg(part + (int64_t)jr * D + d, __uint_as_float(x[i]));
          }
          if (qd == 0 && jl < w.rows) {
            __stcg(part + w.rows * D + jl, s_hm[ob * kNR + jl]);
            __stcg(part + w.rows * D + w.rows + jl, lsum);
          }
        }
      }
      ptx::tc_fence_before();
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.o_empty(ob));

      // ---- split item: the last chunk of this (request, head, row group) to finish merges all ----
      if (w.poff >= 0 && !again) {
        __threadfence();
        if (!group_sync()) { ok = false; break; }
        if (warp == 8 && lane == 0) {
          const int chunks = p.req_chunks[w.r];
          const int done = atomicAdd(p.pair_done + ((int64_t)w.r * p.Hkv + w.h) * p.row_groups + w.rg, 1);
          *s_last = done == chunks - 1 ? chunks : 0;
          __threadfence();
        }
        if (!group_sync()) { ok = false; break; }
        const int chunks = *s_last;
        if (chunks > 0) {
          merge_chunks<D, uint16_t>(p, w, g, chunks, qd, 4);
        }
      }
    }
    if (!ok && lane == 0) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, 0);
  } else if (warp < 16) {
    // ------------------------------------------------------------------ softmax warps
    // Two groups of four: warps 4-7 take the first half of an item's rows, warps 12-15 the second (the
    // MMA's N is a multiple of 16, so both halves are whole 8-row units and both groups always have
    // work).  Within a group, one warp per TMEM lane quadrant, i.e. 32 keys of each tile: a thread holds
    // one key's scores for the group's rows.  The rows' reference maxima are those of the item's first
    // tile (its four warps exchange them once per item): a key of the item that a row can see at all is
    // preceded by one in the first tile, and later tiles then need no agreement between warps.
    const int qd = warp & 3;                  // TMEM lane quadrant: keys 32*qd .. 32*qd + 31 of a tile
    const int grp = warp >= 12 ? 1 : 0;
    const uint32_t lane_addr = (uint32_t)(qd * 32) << 16;
    const float scale_log2 = 1.4426950408889634f / sqrtf((float)D);
    const float2 scale2 = make_float2(scale_log2, scale_log2);
    float *mw = s_mw + (grp * 4 + qd) * 32;   // minus the rows' references, this warp's copy
    uint32_t n = 0;                           // P tiles so far
    uint32_t ns = 0;                          // S^T tiles so far: an item that is taken again has two per P tile
    int li = 0;                               // items so far: item li accumulates into O buffer li & 1
    bool ok = true;
    for (uint32_t j = 0; ok; ++j) {
      const int slot = j % C::RING;
      if (!wait_bar(B.it_full(slot), (j / C::RING) & 1, s_abort)) { ok = false; break; }
      const int it = s_ring[slot].it;
      const int t0 = s_ring[slot].w.t0, t1 = s_ring[slot].w.t1, rows = s_ring[slot].w.rows;
      const int ctx = s_ring[slot].w.ctx, row0 = s_ring[slot].w.row0, passes = s_ring[slot].passes;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.it_empty(slot));
      if (it < 0) break;
      const int ob = li & 1;
      const int ntiles = (t1 - t0 + kBT - 1) / kBT;
      const int nfull = (max(t0, min(t1, ctx + 1)) - t0) / kBT;  // tiles whose keys every row sees
      const int half = (rows + 15) / 16 * 8;  // rows per group
      const int nu = half / 8;                // its 8-row units, 1 to 4
      const int r0 = grp * half;              // the group's first row
      float2 lp[16];  // this thread's (key's) share of every row sum of the group
#pragma unroll
      for (int i = 0; i < 16; ++i) lp[i] = make_float2(0.0f, 0.0f);
      uint32_t pmax = 0;        // largest P so far (two bf16 lanes); +inf too for a row that sees keys of -inf only so far
      float mref = -INFINITY;   // lane i: row r0 + i's maximum so far, then its reference (-inf: no key visible)
      // tiles whose maxima are still to be taken: 1, the first, or for an item that is taken again all of them,
      // counted up to 0, in a pass of their own
      int pre = passes == 2 ? -ntiles : 1;
      for (int t = 0; t < ntiles; ++ns) {
        const int sb = ns & 1;
        if (!wait_bar(B.s_full(sb), (ns >> 1) & 1, s_abort)) { ok = false; break; }
        ptx::tc_fence_after();
        uint32_t x[2][16];
        ptx::tmem_ld16(tmem + lane_addr + sb * kNR + r0, x[0]);
        if (nu > 2) ptx::tmem_ld16(tmem + lane_addr + sb * kNR + r0 + 16, x[1]);
        ptx::tmem_wait_ld();
        // the tile is in registers: it may be overwritten by the S^T after next
        ptx::tc_fence_before();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(B.s_empty(sb));
        // causal mask: key tok is visible to row jr iff tok <= ctx + (row0 + jr) / g, i.e.
        // row0 + jr >= g * (tok - ctx); keys past the item are masked too.  Only an item's last tiles
        // (from nfull on) have such keys.
        if (t >= nfull) {
          const int tok = t0 + t * kBT + qd * 32 + lane;
          const int jmin = tok >= t1 ? 32 : max(0, min(32, g * (tok - ctx) - row0 - r0));
          const uint32_t seen = (uint32_t)(0xffffffffull << jmin);
#pragma unroll
          for (int i = 0; i < 32; ++i)
            if (!(seen & (1u << i))) x[i >> 4][i & 15] = 0xff800000u;
        }
        if (pre != 0) {
          const bool apart = pre < 0;
          // exact row maxima over this warp's 32 keys, and after the last such tile over the group's four
          // quadrants: the references.  Padding rows get +inf (P = 0), rows without a visible key 0 (P = 0:
          // all their scores are -inf).  s_red alternates between items: a warp that writes it for item
          // li + 2 has passed the barrier of item li + 1, where every reader of item li has arrived.
          float wm = -INFINITY;
#pragma unroll
          for (int u = 0; u < 4; ++u) {
            if (u < nu) {
#pragma unroll
              for (int i = 8 * u; i < 8 * u + 8; ++i) {
                const float rm = ptx::warp_max(__uint_as_float(x[i >> 4][i & 15]));
                if (lane == i) wm = rm;
              }
            }
          }
          mref = fmaxf(mref, wm);
          pre += apart ? 1 : -1;
          if (pre == 0) {
            float *red = s_red + (li & 1) * 4 * kNR + r0 + lane;
            if (lane < half) red[qd * kNR] = mref;
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(B.red(grp));
            if (!wait_bar(B.red(grp), li & 1, s_abort)) { ok = false; break; }
            if (lane < half)
              mref = fmaxf(fmaxf(red[0], red[kNR]), fmaxf(red[2 * kNR], red[3 * kNR])) * scale_log2;
            const bool pad = r0 + lane >= rows || lane >= half;
            mw[lane] = pad ? -INFINITY : mref == -INFINITY ? 0.0f : -mref;
            if (!pad && mref == -INFINITY && g * max(t0 - ctx, 0) <= row0 + r0 + lane) pmax = 0x7F80u;
            __syncwarp();
          }
          if (apart) {
            t = pre == 0 ? 0 : t + 1;
            continue;
          }
        }
        // P buffer n % NP is free again once PV(n - NP) is done; PV(n) needs the P(n) about to be
        // published, so the parity is exact
        const int pbuf = (int)(n % C::NP);
        if (n >= (uint32_t)C::NP && !wait_bar(B.o_full(pbuf), ((n - C::NP) / C::NP) & 1, s_abort)) {
          ok = false;
          break;
        }
        uint8_t *prow = smem + C::OFF_P + pbuf * C::P_BYTES + (qd * 32 + lane) * 128;
        const int sw = lane & 7;
        // P = 2^(s - m) (masked: 0), two rows at a time in packed fp32x2 arithmetic, written straight to
        // the P buffer and added to the row-sum shares
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          if (u < nu) {
            uint32_t pk[4];
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const float4 m4 = reinterpret_cast<const float4 *>(mw + 8 * u + 4 * h)[0];
#pragma unroll
              for (int q = 0; q < 2; ++q) {
                const int i = 8 * u + 4 * h + 2 * q;
                const float2 s2 = make_float2(__uint_as_float(x[i >> 4][i & 15]), __uint_as_float(x[i >> 4][(i & 15) + 1]));
                const float2 a = __ffma2_rn(s2, scale2, q == 0 ? make_float2(m4.x, m4.y) : make_float2(m4.z, m4.w));
                const float2 e = make_float2(ptx::ex2(a.x), ptx::ex2(a.y));
                lp[i >> 1] = __fadd2_rn(lp[i >> 1], e);
                const uint32_t pe = pack_bf16(e.x, e.y);
                pmax = bmax2(pmax, pe);
                pk[2 * h + q] = pe;
              }
            }
            *reinterpret_cast<uint4 *>(prow + (((r0 / 8 + u) ^ sw) << 4)) = make_uint4(pk[0], pk[1], pk[2], pk[3]);
          }
        }
        // P(n) is published
        ptx::fence_proxy_async_smem();
        __syncwarp();
        if (lane == 0) ptx::mbar_arrive(B.p_full(pbuf));
        ++t;
        ++n;
      }
      if (!ok) break;
      // ---- hand the item over to the epilogue warps: this quadrant's share of each row sum of
      // the group, and the references.  The epilogue of item li - 2 (same buffers) must be
      // done with them.
      float ls[32];
#pragma unroll
      for (int i = 0; i < 16; ++i) {
        ls[2 * i] = lp[i].x;
        ls[2 * i + 1] = lp[i].y;
      }
      const float lsh = warp_transpose_sum(ls, lane);
      const bool ovf =
          __any_sync(0xffffffffu, fmaxf(__uint_as_float(pmax << 16), __uint_as_float(pmax & 0xffff0000u)) > kMaxP);
      if (!wait_bar(B.o_empty(ob), ((li >> 1) & 1) ^ 1, s_abort)) { ok = false; break; }
      if (lane < half) {
        s_hl[(ob * 4 + qd) * kNR + r0 + lane] = lsh;
        if (qd == 0) s_hm[ob * kNR + r0 + lane] = mref;
      }
      if (lane == 0) s_ovf[8 * ob + 4 * grp + qd] = ovf ? 1 : 0;
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(B.ep_full(ob));
      ++li;
    }
    if (!ok && lane == 0) report(p.status, WISP_DEV_TIMEOUT, p.request_ids, 0);
  }

  // Teardown: every warp reports on an mbarrier that it is done with TMEM, and warp 1 frees the
  // TMEM once all have (a bounded wait; the warps' shared memory stays until the last one exits).
  __syncwarp();
  ptx::tc_fence_before();
  if (lane == 0) ptx::mbar_arrive(B.fin());
  if (warp == 1) {
    const long long t0 = clock64();
    while (!ptx::mbar_try_wait(B.fin(), 0) && clock64() - t0 < kWaitCycles) {
    }
    __syncwarp();
    ptx::tc_fence_after();
    ptx::tmem_dealloc(tmem, kTmemCols);
  }
}

// ---------------------------------------------------------------------------- host side
namespace {

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;

cudaError_t get_encode() {
  if (g_encode) return cudaSuccess;
  void *fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  cudaError_t e = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q);
  if (e != cudaSuccess || q != cudaDriverEntryPointSuccess || !fn) return cudaErrorNotSupported;
  g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  return cudaSuccess;
}

// The paged pool [num_blocks, Hkv, 16, D] bf16 as a 4-D tensor (d, slot, head, block);
// one box = 64 head-dim elements (128 bytes, swizzled) x 16 slots of one head in `box_blocks`
// consecutive blocks (1, or 8 for a whole 128-token tile of consecutive blocks).
cudaError_t encode_pool(CUtensorMap *map, const void *base, int D, int Hkv, int num_blocks, int box_blocks) {
  const cuuint64_t dims[4] = {(cuuint64_t)D, 16, (cuuint64_t)Hkv, (cuuint64_t)num_blocks};
  const cuuint64_t strides[3] = {(cuuint64_t)D * 2, (cuuint64_t)16 * D * 2, (cuuint64_t)Hkv * 16 * D * 2};
  const cuuint32_t box[4] = {64, 16, 1, (cuuint32_t)box_blocks};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  const CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(base), dims, strides, box,
                              estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                              CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

}  // namespace

cudaError_t attn_tc_setup() {
  cudaError_t e = get_encode();
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_tc_kernel<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<128>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, Cfg<64>::SMEM);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_tc_kernel<128>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(attn_tc_kernel<64>, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared);
  return e;
}

namespace {

// The four tensor maps of a (K pool, V pool, D, Hkv, num_blocks) are the same from step to step:
// the last few sets are kept, so that a launch does not encode them again.
struct PoolMaps {
  const void *k = nullptr, *v = nullptr;
  int D = 0, Hkv = 0, num_blocks = 0;
  alignas(64) CUtensorMap tk, tv, tk8, tv8;
};
constexpr int kMapCache = 8;
PoolMaps g_maps[kMapCache];
int g_maps_next = 0;
std::mutex g_maps_mu;

cudaError_t pool_maps(const AttnParams &p, PoolMaps *out) {
  std::lock_guard<std::mutex> lk(g_maps_mu);
  for (const PoolMaps &m : g_maps) {
    if (m.k == p.k_cache && m.v == p.v_cache && m.D == p.D && m.Hkv == p.Hkv && m.num_blocks == p.num_blocks) {
      *out = m;
      return cudaSuccess;
    }
  }
  PoolMaps m;
  m.k = p.k_cache;
  m.v = p.v_cache;
  m.D = p.D;
  m.Hkv = p.Hkv;
  m.num_blocks = p.num_blocks;
  cudaError_t e = encode_pool(&m.tk, p.k_cache, p.D, p.Hkv, p.num_blocks, 1);
  if (e == cudaSuccess) e = encode_pool(&m.tv, p.v_cache, p.D, p.Hkv, p.num_blocks, 1);
  if (e == cudaSuccess) e = encode_pool(&m.tk8, p.k_cache, p.D, p.Hkv, p.num_blocks, 8);
  if (e == cudaSuccess) e = encode_pool(&m.tv8, p.v_cache, p.D, p.Hkv, p.num_blocks, 8);
  if (e != cudaSuccess) return e;
  g_maps[g_maps_next] = m;
  g_maps_next = (g_maps_next + 1) % kMapCache;
  *out = m;
  return cudaSuccess;
}

}  // namespace

cudaError_t attn_tc_launch(const AttnParams &p, int grid, cudaStream_t s) {
  PoolMaps m;
  const cudaError_t e = pool_maps(p, &m);
  if (e != cudaSuccess) return e;
  const CUtensorMap &tk = m.tk, &tv = m.tv, &tk8 = m.tk8, &tv8 = m.tv8;
  // programmatic dependent launch: the CTAs' set-up overlaps the kernel before this one (the
  // planner), which the kernel waits for before it reads the plan
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
  if (p.D == 128) {
    cfg.dynamicSmemBytes = Cfg<128>::SMEM;
    return cudaLaunchKernelEx(&cfg, attn_tc_kernel<128>, p, tk, tv, tk8, tv8);
  }
  cfg.dynamicSmemBytes = Cfg<64>::SMEM;
  return cudaLaunchKernelEx(&cfg, attn_tc_kernel<64>, p, tk, tv, tk8, tv8);
}

}  // namespace wisp
