// The visual side of the query-aware score (Eq. 10) with per-head linear embeddings, bf16 operands.
//
// A cluster of two CTAs owns a pair of neighbouring 128-token tiles and multiplies with
// tcgen05.mma.cta_group::2 (M = 256 across the pair).  Per work item (one pair of tiles, one group of one or two
// heads) it computes
//   Kp = X_tile * Wk[heads]^T           256 x 256 over the pair, 256 accumulator columns in each SM's TMEM
//   per token and head: ||Kp||^2        epilogue warps read TMEM, keep the norm in float32 and restage the
//                                       head as bf16 hi + lo K-major tiles in shared memory
//   logits = Kp * Qn[head]^T            second product against the unit-length query elements, up to 128 of them
//                                       at a time, as hi*hi + lo*hi + hi*lo so that bf16 staging costs ~2^-16
//   S^query = max_j,h logits / ||Kp||   row max in registers, atomic max into the score array
// so the projected embeddings never leave the SM.
//
// Why two SMs: a CTA fetches its own tokens and only its half of the weights, 32 KB per 64 features and 512 tensor
// cycles.  Measured per chunk, whatever the depth of the ring: 786 cycles for the 128 x 256 products of one SM, which write and
// read 96 KB of shared memory (768 cycles at 128 bytes a cycle); 725-750 here with about 80 KB (640), of which some
// 100 are not explained (the tensor pipe is busy 76 % of the time; 16,384 tokens, d = 3584, 28 heads: 308 us).  Under the power
// limit of long runs the kernel went from 1.35 to 1.42 PFLOP/s, the three hi and lo products of the logits counted.  The
// query elements are shared the same way.
//
// The second product and the epilogue of one item run beside the main loop of the next: TMEM holds two
// accumulators of 256 columns, and the logits of a head take the place of that head's own columns, which have
// been read by then.  The main loop, the logits and their operands have issuing threads of their own, so
// nothing interleaves them but the tensor pipe; a head is restaged while the logits of the one before are read.
// Below d = 2048 that chain is the longer one (per head 1.3 k cycles of restaging, 24 products of about 128 cycles each
// whatever their width up to 128, the reading): 148 tiles, 16 heads, d = 256, 256 query elements 170 -> 104 us.
// The tiles of a pair may belong to two requests (tiles are paired across the whole batch).  Their query elements are
// neighbouring rows, so such a pair goes through them as through one request's, and each CTA looks at its own columns (512
// requests of 100 tokens, d = 512, 8 heads, 32 and 64 query elements each: 221 and 246 us with logits tiles of one
// request each, 164 and 191 now).  Both requests' products are computed for all 256 rows, which shows where nearly all pairs are
// such ones and the logits are most of the work: with 256 query elements each 615 us, 602 on one SM per tile.
//
// Warp roles per CTA (384 threads): 0-7 epilogue (a TMEM lane = a token; warps w and w + 4 share 32 tokens, each
// taking half of the columns), 8 TMA producer of the main ring, 9 TMEM owner and, in the leader CTA, MMA issuer of
// the main loop, 10 (leader) MMA issuer of the logits, 11 TMA producer of the query blocks.  Loads are plain
// per-CTA tile loads whose bytes are counted on the leader's barriers; tcgen05.commit signals the barriers of both
// CTAs; barriers that the issuers wait on live in the leader.  Every wait is bounded; on expiry the CTA raises
// a status bit and stops working, and both CTAs meet at a cluster barrier before they exit.
#pragma once
#include "relevance_tc.cuh"

namespace covspec {
namespace tc {

// Shared memory: the ring of the main loop (four stages of two heads, five of one), one restaged head (hi and lo, two
// halves of 64 features each), a ring of query
// blocks [kq query elements x 64 features] (hi and lo blocks alternate; kq is half of the widest logits tile of
// the call), barriers, the exchange between the two threads of a token.
// A cluster with a single item restages its heads when the main loop is over: its ring takes their place as well (six
// stages of two heads, eight of one).  With few items the main loop is bound by the time a stage takes to come round.
constexpr int kVisRing = 128 * 1024;
constexpr int kVisMaxStages = 8;
constexpr int kVisThreads = 384;
// Bounds for 64 registers a thread: 24,576 of the SM's 65,536, which is what a block of the activity stream leaves (score_kernels.cuh).
// The kernel takes 62 without spills; with 80 it is 0 to 3 % faster by itself, and no stream block of enough warps fits beside it.
constexpr int kVisMaxThreads = 512;
constexpr int kVisEpiWarps = 8;
constexpr int kVisHeadBytes = kHeadDim / 2 * kBK * 2;      // 8 KB: this CTA's half of a head's weight chunk
constexpr int kLogitN = 128;                              // query elements per logits tile (UMMA N of the 2nd product)
constexpr int kQueryRing = 28 * 1024;
constexpr int kMaxQuerySlots = 8;
constexpr int kVisSmem = kVisRing + 4 * kBytesKp + kQueryRing + 1024 /*barriers*/ + 1024 /*exchange*/;
static_assert(kVisSmem <= kQuerySmem, "see kQuerySmem");

// ---- two-CTA forms of the building blocks of tc_common.cuh ----
// TMA tile load into this CTA's shared memory whose bytes are counted on a barrier of the pair's
// leader CTA (bar_cluster_addr: see map_to_cta).  No multicast.
__device__ __forceinline__ void tma_load_2d_pair(uint32_t smem_dst, const CUtensorMap* map, int x, int y,
                                                 uint32_t bar_cluster_addr) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(smem_dst), "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster_addr)
      : "memory");
}
__device__ __forceinline__ void umma_bf16_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                               uint32_t accumulate) {
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "setp.ne.b32 p, %4, 0;\n"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives (once the MMAs issued so far have completed) on the barrier at this offset in both CTAs.
__device__ __forceinline__ void umma_commit_pair(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(
          smem_u32(bar)),
      "h"((unsigned short)3)
      : "memory");
}

// Largest of three, NaN if one of them is.
__device__ __forceinline__ float max3_nan(float a, float b, float c) {
  float r;
  asm("max.NaN.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}
// One poll that never suspends the thread (try_wait may, while the current chunk's products are still to be issued).
__device__ __forceinline__ bool mbar_test(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      ".reg .pred p;\n"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      "selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

struct VisParams {
  const int4* tiles;    // [n_tiles] 128-token tiles over all requests: first row of X, rows, first query row, query elements
  int n_tiles;
  int n_items;          // (pair of tiles, group of heads) pairs
  int n_groups;         // groups of heads
  int group_heads;      // heads per group, 2 or 1 (the weight map's boxes are 64 rows high per head)
  int stages;           // of the main ring, kBytesA + group_heads * kVisHeadBytes each
  int n_heads;
  int k_chunks;         // ceil(d / 64)
  int rows_total;       // rows of X
  int query_rows;       // kq: query elements of a block, per CTA (the boxes of the query maps)
  float* s_query;       // out (pre-filled with -inf)
  int* status;
};

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kVisMaxThreads, 2)
relevance_vis_kernel(const __grid_constant__ CUtensorMap map_x,   // X: [rows, d]
                     const __grid_constant__ CUtensorMap map_w,   // Wk: [P, d]
                     const __grid_constant__ CUtensorMap map_q,   // Qn hi: [sum T, P]
                     const __grid_constant__ CUtensorMap map_ql,  // Qn lo
                     const VisParams prm) {
  extern __shared__ __align__(1024) uint8_t rel_smem_raw[];
  uint8_t* smem = rel_smem_raw;
  uint8_t* kp_smem = smem + kVisRing;                      // hi half 0, hi half 1, lo half 0, lo half 1
  uint8_t* q_smem = kp_smem + 4 * kBytesKp;                // [slots][kq x 64]
  uint64_t* bars = reinterpret_cast<uint64_t*>(q_smem + kQueryRing);
  uint64_t* full = bars;                                 // [kVisMaxStages] leader: bytes of both CTAs' loads
  uint64_t* empty = full + kVisMaxStages;                // [kVisMaxStages] both
  uint64_t* q_full = empty + kVisMaxStages;                // [kMaxQuerySlots] leader: bytes of both CTAs' loads
  uint64_t* q_empty = q_full + kMaxQuerySlots;           // [kMaxQuerySlots] both
  uint64_t* acc_full = q_empty + kMaxQuerySlots;         // [2] both
  uint64_t* acc_empty = acc_full + 2;                    // [2] leader, one arrival per epilogue warp of both CTAs
  uint64_t* logit_full = acc_empty + 2;                  // [2] both
  uint64_t* logit_empty = logit_full + 2;                // [2] leader, epilogue warps
  uint64_t* kp_ready = logit_empty + 2;                  // leader, epilogue warps
  uint64_t* kp_free = kp_ready + 1;                      // both
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(kp_free + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* exchange = reinterpret_cast<float*>(q_smem + kQueryRing + 1024);      // [2][128] largest logit of the second thread
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const bool aligned = (smem_u32(smem) & 1023u) == 0;      // the swizzled tiles need a 1024-byte aligned base

  if (threadIdx.x == 0) {
    for (int s = 0; s < kVisMaxStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int s = 0; s < kMaxQuerySlots; ++s) { mbar_init(&q_full[s], 1); mbar_init(&q_empty[s], 1); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 2 * kVisEpiWarps);
      mbar_init(&logit_full[i], 1); mbar_init(&logit_empty[i], 2 * kVisEpiWarps);
    }
    mbar_init(kp_ready, 2 * kVisEpiWarps);
    mbar_init(kp_free, 1);
    *abort_flag = aligned ? 0 : 1;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                      // both CTAs' barriers exist before anything arrives on them
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int n_clusters = gridDim.x >> 1, cluster_id = blockIdx.x >> 1;

  // Item -> this CTA's tile rows, first head and heads of the group, the query rows of the pair (of one request, or of two
  // neighbouring ones) and this CTA's own among them; every role walks the same list.
  struct Item {
    int row0, nrows, head0, heads;
    int txt0, T, tiles;                    // first query row, query elements, logits tiles of the pair
    int own0, own1;                        // this CTA's query elements
  };
  auto decode = [&](int item) {
    Item it;
    const int pair = item / prm.n_groups, g = item - pair * prm.n_groups;
    it.head0 = g * prm.group_heads;
    it.heads = min(prm.group_heads, prm.n_heads - it.head0);
    const int4 a = prm.tiles[2 * pair], b = prm.tiles[min(2 * pair + 1, prm.n_tiles - 1)];
    const bool two = a.z != b.z;           // requests (each has query rows of its own)
    it.txt0 = a.z;
    it.T = a.w + (two ? b.w : 0);
    it.tiles = (it.T + kLogitN - 1) / kLogitN;
    it.own0 = two && rank != 0 ? a.w : 0;
    it.own1 = two && rank == 0 ? a.w : it.T;
    const bool exists = 2 * pair + (int)rank < prm.n_tiles;      // no tile: all rows read as zeros
    it.row0 = exists ? (rank != 0 ? b.x : a.x) : prm.rows_total;
    it.nrows = exists ? (rank != 0 ? b.y : a.y) : 0;
    return it;
  };
  // Width of logits tile i of an item (a multiple of 32)
  auto logits_width = [&](const Item& it, int i) { return min(kLogitN, (it.T - i * kLogitN + 31) & ~31); };
  const int stage_bytes = kBytesA + prm.group_heads * kVisHeadBytes;
  const int q_bytes = prm.query_rows * kHalf * 2, q_slots = min(kMaxQuerySlots, kQueryRing / q_bytes);

  if (warp == 8) {
    // ---------------------------------------------------------------- TMA producer, main ring (both CTAs)
    if (lane == 0 && aligned) {
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (int item = cluster_id; item < prm.n_items && ok; item += n_clusters) {
        const Item it = decode(item);
        // the CTA's half of the group's features (a lone last head: 64 of the 128 rows are used)
        const int wrow = it.head0 * kHeadDim + (int)rank * it.heads * (kHeadDim / 2);
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = mbar_wait(&empty[s], ph, abort_flag))) break;
          if (leader) mbar_expect_tx(&full[s], 2 * stage_bytes);
          const uint32_t dst = smem_u32(smem + s * stage_bytes), bar = map_to_cta(&full[s], 0);
          tma_load_2d_pair(dst, &map_x, kc * kBK, it.row0, bar);
          tma_load_2d_pair(dst + kBytesA, &map_w, kc * kBK, wrow, bar);
          if (++s == prm.stages) { s = 0; ph ^= 1u; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 9) {
    // ---------------------------------------------------------------- MMA issuer, main loop (leader)
    if (lane == 0 && leader && aligned) {
      int s = 0;
      uint32_t ph = 0, n = 0;
      bool ok = true, ready = false;
      for (int item = cluster_id; item < prm.n_items && ok; item += n_clusters, ++n) {
        const uint32_t buf = n & 1u;
        if (!(ok = mbar_wait(&acc_empty[buf], ((n >> 1) & 1u) ^ 1u, abort_flag))) break;
        tc_fence_after();
        const int head0 = item % prm.n_groups * prm.group_heads;
        const uint32_t idesc = umma_idesc(2 * kTileM, min(prm.group_heads, prm.n_heads - head0) * kHeadDim);
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!ready && !(ok = mbar_wait(&full[s], ph, abort_flag))) break;
          tc_fence_after();
          const uint32_t a_addr = smem_u32(smem + s * stage_bytes);
          const uint64_t adesc = umma_desc(a_addr), bdesc = umma_desc(a_addr + kBytesA);
          const int cur = s;
          if (++s == prm.stages) { s = 0; ph ^= 1u; }
          ready = mbar_test(&full[s], ph);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            umma_bf16_pair(tmem_base + buf * kTileN, adesc + 2 * k, bdesc + 2 * k, idesc, (kc | k) != 0);
          umma_commit_pair(&empty[cur]);
        }
        if (ok) umma_commit_pair(&acc_full[buf]);
      }
    }
    __syncwarp();
  } else if (warp == 10) {
    // ---------------------------------------------------------------- MMA issuer, logits (leader)
    if (lane == 0 && leader && aligned) {
      uint32_t n = 0, head_it = 0, lt = 0, q_ph = 0;
      int qs = 0;
      bool ok = true;
      for (int item = cluster_id; item < prm.n_items && ok; item += n_clusters, ++n) {
        const Item it = decode(item);
        const int ntt = it.tiles;
        for (int h = 0; h < it.heads && ok; ++h, ++head_it) {
          if (!(ok = mbar_wait_cluster(kp_ready, head_it & 1u, abort_flag))) break;      // both CTAs have restaged this head
          const uint32_t kp_addr = smem_u32(kp_smem);
          const uint32_t d_col = tmem_base + (n & 1u) * kTileN + h * kHeadDim;
          for (int i = 0; i < ntt && ok; ++i, ++lt) {
            // the tile before the last has been read (its barrier is used again), and within a head the last one
            // too: it lies in the same columns
            if (lt >= 2 && !(ok = mbar_wait(&logit_empty[lt & 1u], ((lt - 2) >> 1) & 1u, abort_flag))) break;
            if (i > 0 && !(ok = mbar_wait(&logit_empty[(lt - 1) & 1u], ((lt - 1) >> 1) & 1u, abort_flag))) break;
            const uint32_t idesc = umma_idesc(2 * kTileM, logits_width(it, i));
            // logits = sum over the two halves of Kp_hi Qn_hi^T + Kp_lo Qn_hi^T + Kp_hi Qn_lo^T
            for (int half = 0; half < 2 && ok; ++half) {
              const uint64_t hi = umma_desc(kp_addr + half * kBytesKp), lo = umma_desc(kp_addr + (2 + half) * kBytesKp);
#pragma unroll 1
              for (int part = 0; part < 2; ++part) {
                if (!(ok = mbar_wait(&q_full[qs], q_ph, abort_flag))) break;
                tc_fence_after();
                const uint64_t q = umma_desc(smem_u32(q_smem + qs * q_bytes));
#pragma unroll
                for (int ks = 0; ks < kHalf / 16; ++ks) umma_bf16_pair(d_col, hi + 2 * ks, q + 2 * ks, idesc, (half | part | ks) != 0);
                if (part == 0) {
#pragma unroll
                  for (int ks = 0; ks < kHalf / 16; ++ks) umma_bf16_pair(d_col, lo + 2 * ks, q + 2 * ks, idesc, 1u);
                }
                umma_commit_pair(&q_empty[qs]);
                if (++qs == q_slots) { qs = 0; q_ph ^= 1u; }
              }
            }
            if (ok) umma_commit_pair(&logit_full[lt & 1u]);
          }
          if (ok) umma_commit_pair(kp_free);
        }
      }
    }
    __syncwarp();
  } else if (warp == 11) {
    // ---------------------------------------------------------------- TMA producer, query blocks (both CTAs)
    if (lane == 0 && aligned) {
      int qs = 0;
      uint32_t ph = 1;
      bool ok = true;
      wait_for_previous_kernel();              // the unit query elements are complete
      for (int item = cluster_id; item < prm.n_items && ok; item += n_clusters) {
        const Item it = decode(item);
        const int ntt = it.tiles;
        for (int h = 0; h < it.heads && ok; ++h)
          for (int i = 0; i < ntt && ok; ++i) {
            const int y = it.txt0 + i * kLogitN + (int)rank * (logits_width(it, i) >> 1);
            for (int p = 0; p < 4; ++p) {      // half, hi / lo: the order in which the logits issuer uses them
              if (!(ok = mbar_wait(&q_empty[qs], ph, abort_flag))) break;
              if (leader) mbar_expect_tx(&q_full[qs], 2 * q_bytes);
              tma_load_2d_pair(smem_u32(q_smem + qs * q_bytes), (p & 1) ? &map_ql : &map_q,
                               (it.head0 + h) * kHeadDim + (p >> 1) * kHalf, y, map_to_cta(&q_full[qs], 0));
              if (++qs == q_slots) { qs = 0; ph ^= 1u; }
            }
          }
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- epilogue (warps 0-7, both CTAs)
    const int r = (warp & 3) * 32 + lane;                  // token row inside the tile = TMEM lane
    const int part = warp >> 2;                            // which half of the columns this thread takes
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    const uint32_t l_kp_ready = map_to_cta(kp_ready, 0), l_acc_empty = map_to_cta(acc_empty, 0),
                   l_logit_empty = map_to_cta(logit_empty, 0);       // [2] each: 8 bytes apart
    uint32_t n = 0, head_it = 0, lt = 0;
    bool ok = aligned;                                     // a thread that gave up stays for the barriers
    Item next = decode(cluster_id);
    for (int item = cluster_id; item < prm.n_items; item += n_clusters, ++n) {
      const Item it = next;
      next = decode(min(item + n_clusters, prm.n_items - 1));       // its loads are back by the time it is needed
      const uint32_t buf = n & 1u;
      const int ntt = it.tiles;
      float best = -INFINITY, top = -INFINITY, ss = 0.f;    // top: largest product of the head so far (NaN if one is)
      bool nonfinite = false;
      ok = ok && mbar_wait(&acc_full[buf], (n >> 1) & 1u, abort_flag);
      tc_fence_after();
      // logits tile i of head h: this thread's half of the CTA's own columns
      auto read_logits = [&](int h, int i) {
        ok = ok && mbar_wait(&logit_full[lt & 1u], (lt >> 1) & 1u, abort_flag);
        tc_fence_after();
        const int lo = max(it.own0 - i * kLogitN, 0), hi = min(it.own1 - i * kLogitN, kLogitN);
        if (lo < hi) {
          const uint32_t cols = t_lane + buf * kTileN + h * kHeadDim;
          // from the 16 columns that lo lies in; the tile's width is a multiple of 32, so what is read has been written
          const int first = lo & ~15, half = ((hi - first + 1) / 2 + 15) & ~15;
          const int c0 = first + part * half, c_end = part ? hi : min(hi, first + half);
#pragma unroll 1
          for (int c = c0; c < c_end; c += 32) {
            float v[32];
            if (c_end - c > 16) {
              tmem_ld32(cols + c, v);
            } else {
              float u[16];
              tmem_ld16(cols + c, u);
#pragma unroll
              for (int e = 0; e < 32; ++e) v[e] = e < 16 ? u[e] : -INFINITY;
            }
            if (c < lo || c + 32 > hi) {
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (c + e < lo || c + e >= hi) v[e] = -INFINITY;
            }
#pragma unroll
            for (int e = 0; e < 32; e += 2) top = max3_nan(top, v[e], v[e + 1]);
          }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_at(l_logit_empty + 8 * (lt & 1u));
        ++lt;
      };
      // last logits tile of a head, then the two threads of a token put their halves together: a cosine is the
      // largest product over the length (rounding keeps the order, so scaling after the maximum changes nothing)
      auto finish_head = [&](int h, float ss_h) {
        read_logits(h, ntt - 1);
        float* x = exchange + ((head_it + (uint32_t)h) & 1u) * 128 + r;
        if (part == 1) *x = top;
        named_barrier(1, kVisEpiWarps * 32);
        if (part == 0) {
          const float o = *x;
          nonfinite |= o != o || top != top || !(ss_h <= 3.402823466e38f);
          float inv = 0.f;
          if (ss_h > 1.17549435e-38f) { inv = rsqrtf(ss_h); inv = inv * (1.5f - 0.5f * ss_h * inv * inv); }
          best = fmaxf(best, fmaxf(top, o) * inv);
        }
        top = -INFINITY;
      };
      for (int h = 0; h < it.heads; ++h) {
        // restage this thread's 64 features of the head as bf16 hi + lo, once the previous head's products have read theirs
        const uint32_t cols = t_lane + buf * kTileN + h * kHeadDim + part * kHalf;
        const float ss_before = ss;
        ss = 0.f;
        ok = ok && mbar_wait(kp_free, ((head_it + (uint32_t)h) & 1u) ^ 1u, abort_flag);
#pragma unroll 1
        for (int c2 = 0; c2 < 2; ++c2) {
          float v[32];
          tmem_ld32(cols + c2 * 32, v);
          uint32_t pk[16], pl[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            float a = v[2 * e], b = v[2 * e + 1];
            ss += a * a + b * b;
            __nv_bfloat162 hi = __floats2bfloat162_rn(a, b);
            pk[e] = *reinterpret_cast<uint32_t*>(&hi);
            pl[e] = pack_bf16(a - __low2float(hi), b - __high2float(hi));
          }
          uint8_t* rowp = kp_smem + part * kBytesKp + r * 128;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int chunk = (c2 * 4 + q) ^ (r & 7);
            *reinterpret_cast<uint4*>(rowp + chunk * 16) =
                make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
            *reinterpret_cast<uint4*>(rowp + 2 * kBytesKp + chunk * 16) =
                make_uint4(pl[4 * q], pl[4 * q + 1], pl[4 * q + 2], pl[4 * q + 3]);
          }
        }
        if (part == 0) {
          // the other half of the squared length: one thread adds up all features in their order
#pragma unroll 1
          for (int c2 = 0; c2 < 2; ++c2) {
            float v[32];
            tmem_ld32(cols + kHalf + c2 * 32, v);
#pragma unroll
            for (int e = 0; e < 16; ++e) {
              float a = v[2 * e], b = v[2 * e + 1];
              ss += a * a + b * b;
            }
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_release_at(l_kp_ready);
        if (h > 0) finish_head(h - 1, ss_before);
        for (int i = 0; i + 1 < ntt; ++i) read_logits(h, i);
      }
      finish_head(it.heads - 1, ss);
      head_it += (uint32_t)it.heads;
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_at(l_acc_empty + 8 * buf);       // projections and logits of the item have been read
      if (item == cluster_id) wait_for_previous_kernel();         // the scores are filled with -inf
      if (part == 0 && r < it.nrows && ok) {
        if (nonfinite) atomicOr(prm.status, kStatusNonFinite);
        else atomic_max_float(prm.s_query + it.row0 + r, best);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                      // nothing of the peer may still point at this CTA
  if (warp == 9) {
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(kTmemCols)
                 : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag) atomicOr(prm.status, kStatusTimeout);
}

}  // namespace tc
}  // namespace covspec
