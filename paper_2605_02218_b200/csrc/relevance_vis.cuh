// The visual side of the query-aware score (Eq. 10) with per-head linear embeddings, bf16 operands.
//
// Per work item (one 128-token tile of one request, one pair of heads) the kernel computes
//   Kp = X_tile * Wk[heads]^T           tcgen05.mma kind::f16, 128 x 256 accumulator in TMEM, operands
//                                       streamed by TMA through a shared-memory ring
//   per token and head: ||Kp||^2        epilogue warps read TMEM, keep the norm in float32 and restage the
//                                       head as bf16 hi + lo K-major tiles in shared memory
//   logits = Kp * Qn[head]^T            second product against the unit-length query elements, 64 of them at a
//                                       time, as hi*hi + lo*hi + hi*lo so that bf16 staging costs ~2^-16
//   S^query = max_j,h logits / ||Kp||   row max in registers, atomic max into the score array
// so the projected embeddings never leave the SM.
//
// The second product and the epilogue of one item run beside the main loop of the next: TMEM holds two
// accumulators of 256 columns, and the logits of a head take the place of that head's own columns, which have
// been read by then.  The main loop, the logits and their operands have issuing threads of their own, so
// nothing interleaves them but the tensor pipe.  With one accumulator the pipe waited for the restaging,
// the query tiles and the small products of every item: 18 % of the launch at d = 3584 with 64 query
// elements, 24 % at d = 4096 with 128 and 57 % at d = 1536 with 16-256.
//
// Warp roles (256 threads): 0-3 epilogue (one TMEM lane = one token each), 4 TMA producer of the main ring,
// 5 MMA issuer of the main loop and TMEM owner, 6 MMA issuer of the logits, 7 TMA producer of the query
// tiles.  Every mbarrier wait is bounded; on expiry the CTA raises a status bit, leaves its loops, frees
// TMEM and exits.
#pragma once
#include "relevance_tc.cuh"

namespace covspec {
namespace tc {

// Shared memory: three ring stages (a fourth bought nothing), one restaged head (hi and lo, two halves of 64
// features each), a ring of two query blocks [64 elements x 64 features] (hi and lo blocks alternate).
constexpr int kVisStages = 3;
constexpr int kVisThreads = 256;
constexpr int kQueryBlock = kTT * kHalf * 2;              // 8 KB
constexpr int kVisSmem = kVisStages * kBytesStage + 4 * kBytesKp + 2 * kQueryBlock + 1024 /*barriers*/;
static_assert(kVisSmem == kQuerySmem, "see kQuerySmem");
constexpr int kLogitTiles = kHeadDim / kTT;               // logits tiles in the columns of one head

__global__ void __launch_bounds__(kVisThreads, 1)
relevance_vis_kernel(const __grid_constant__ CUtensorMap map_x,   // X: [rows, d]
                     const __grid_constant__ CUtensorMap map_w,   // Wk: [P, d]
                     const __grid_constant__ CUtensorMap map_q,   // Qn hi: [sum T, P]
                     const __grid_constant__ CUtensorMap map_ql,  // Qn lo
                     const Params prm) {
  extern __shared__ __align__(1024) uint8_t rel_smem_raw[];
  uint8_t* smem = rel_smem_raw;
  if (smem_u32(smem) & 1023u) {          // the swizzled tiles need a 1024-byte aligned base
    if (threadIdx.x == 0) atomicOr(prm.status, kStatusTimeout);
    return;
  }
  uint8_t* kp_smem = smem + kVisStages * kBytesStage;    // hi half 0, hi half 1, lo half 0, lo half 1
  uint8_t* q_smem = kp_smem + 4 * kBytesKp;              // [2][kQueryBlock]
  uint64_t* bars = reinterpret_cast<uint64_t*>(q_smem + 2 * kQueryBlock);
  uint64_t* full = bars;                                 // [kVisStages]
  uint64_t* empty = bars + kVisStages;                   // [kVisStages]
  uint64_t* acc_full = bars + 2 * kVisStages;            // [2]
  uint64_t* acc_empty = acc_full + 2;                    // [2]
  uint64_t* kp_ready = acc_full + 4;
  uint64_t* kp_free = acc_full + 5;
  uint64_t* logit_full = acc_full + 6;                   // [kLogitTiles]
  uint64_t* logit_empty = acc_full + 8;                  // [kLogitTiles]
  uint64_t* q_full = acc_full + 10;                      // [2]
  uint64_t* q_empty = acc_full + 12;                     // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 14);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kVisStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 128);
      mbar_init(&logit_full[i], 1); mbar_init(&logit_empty[i], 128);
      mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1);
    }
    mbar_init(kp_ready, 128);
    mbar_init(kp_free, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) tmem_alloc(tmem_slot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // Item -> tile rows, query rows, first head; every role walks the same list.
  auto decode = [&](int item, int& row0, int& nrows, int& txt0, int& T, int& hp, int& heads) {
    const int tile = item / prm.n_groups;
    hp = item % prm.n_groups;
    heads = min(2, prm.n_heads - 2 * hp);
    const int b = find_request(tile, prm.batch, [&](int q) { return prm.plan[q].tile_off; });
    const ReqPlan rp = prm.plan[b];
    const int t = tile - rp.tile_off;
    row0 = rp.vis_off + t * kTileM;
    nrows = min(kTileM, rp.n - t * kTileM);
    txt0 = rp.txt_off;
    T = rp.t;
  };

  if (warp == 4) {
    // ---------------------------------------------------------------- TMA producer, main ring
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x) {
        int row0, nrows, txt0, T, hp, heads;
        decode(item, row0, nrows, txt0, T, hp, heads);
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = mbar_wait(&empty[s], ph, abort_flag))) break;
          mbar_expect_tx(&full[s], kBytesStage);
          const uint32_t dst = smem_u32(smem + s * kBytesStage);
          tma_load_2d(dst, &map_x, kc * kBK, row0, &full[s]);
          tma_load_2d(dst + kBytesA, &map_w, kc * kBK, hp * kTileN, &full[s]);
          if (++s == kVisStages) { s = 0; ph ^= 1u; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 5) {
    // ---------------------------------------------------------------- MMA issuer, main loop
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0, n = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x, ++n) {
        const uint32_t buf = n & 1u;
        if (!(ok = mbar_wait(&acc_empty[buf], ((n >> 1) & 1u) ^ 1u, abort_flag))) break;
        tc_fence_after();
        // a lone last head takes half the columns and half the tensor time (576 tokens, one float32 head, d = 1024: a
        // call 171.0 -> 169.0 us; fetching half the weight tile as well gained nothing)
        const uint32_t idesc = umma_idesc(kTileM, item % prm.n_groups * 2 + 1 < prm.n_heads ? kTileN : kHeadDim);
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = mbar_wait(&full[s], ph, abort_flag))) break;
          tc_fence_after();
          const uint32_t a_addr = smem_u32(smem + s * kBytesStage);
          const uint64_t adesc = umma_desc(a_addr), bdesc = umma_desc(a_addr + kBytesA);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            umma_bf16(tmem_base + buf * kTileN, adesc + 2 * k, bdesc + 2 * k, idesc, (kc | k) != 0);
          umma_commit(&empty[s]);
          if (++s == kVisStages) { s = 0; ph ^= 1u; }
        }
        if (ok) umma_commit(&acc_full[buf]);
      }
    }
    __syncwarp();
  } else if (warp == 6) {
    // ---------------------------------------------------------------- MMA issuer, logits
    if (lane == 0) {
      const uint32_t idesc = umma_idesc(kTileM, kTT);
      uint32_t n = 0, head_it = 0, q_it = 0, uses[kLogitTiles] = {0u, 0u};
      bool ok = true;
      for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x, ++n) {
        int row0, nrows, txt0, T, hp, heads;
        decode(item, row0, nrows, txt0, T, hp, heads);
        const int ntt = (T + kTT - 1) / kTT;
        for (int h = 0; h < heads && ok; ++h, ++head_it) {
          if (!(ok = mbar_wait(kp_ready, head_it & 1u, abort_flag))) break;      // this head is restaged
          const uint32_t kp_addr = smem_u32(kp_smem);
          for (int t = 0; t < ntt && ok; ++t) {
            const int slot = t & 1;
            if (!(ok = mbar_wait(&logit_empty[slot], (uses[slot] & 1u) ^ 1u, abort_flag))) break;
            ++uses[slot];
            const uint32_t d_col = tmem_base + (n & 1u) * kTileN + h * kHeadDim + slot * kTT;
            // logits = sum over the two halves of Kp_hi Qn_hi^T + Kp_lo Qn_hi^T + Kp_hi Qn_lo^T
            for (int half = 0; half < 2 && ok; ++half) {
              const uint64_t hi = umma_desc(kp_addr + half * kBytesKp), lo = umma_desc(kp_addr + (2 + half) * kBytesKp);
#pragma unroll 1
              for (int part = 0; part < 2; ++part, ++q_it) {
                const uint32_t qs = q_it & 1u;
                if (!(ok = mbar_wait(&q_full[qs], (q_it >> 1) & 1u, abort_flag))) break;
                tc_fence_after();
                const uint64_t q = umma_desc(smem_u32(q_smem + qs * kQueryBlock));
#pragma unroll
                for (int ks = 0; ks < kHalf / 16; ++ks) umma_bf16(d_col, hi + 2 * ks, q + 2 * ks, idesc, (half | part | ks) != 0);
                if (part == 0) {
#pragma unroll
                  for (int ks = 0; ks < kHalf / 16; ++ks) umma_bf16(d_col, lo + 2 * ks, q + 2 * ks, idesc, 1u);
                }
                umma_commit(&q_empty[qs]);
              }
            }
            if (ok) umma_commit(&logit_full[slot]);
          }
          if (ok) umma_commit(kp_free);
        }
      }
    }
    __syncwarp();
  } else if (warp == 7) {
    // ---------------------------------------------------------------- TMA producer, query blocks
    if (lane == 0) {
      uint32_t q_it = 0;
      bool ok = true;
      wait_for_previous_kernel();              // the unit query elements are complete
      for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x) {
        int row0, nrows, txt0, T, hp, heads;
        decode(item, row0, nrows, txt0, T, hp, heads);
        const int blocks = heads * ((T + kTT - 1) / kTT) * 4;
        for (int i = 0; i < blocks; ++i, ++q_it) {
          // head, tile, half, hi / lo: the order in which the logits issuer uses them
          const int part = i & 1, half = (i >> 1) & 1, ht = i >> 2, ntt = (T + kTT - 1) / kTT;
          const int h = ht / ntt, t = ht - h * ntt;
          const uint32_t qs = q_it & 1u;
          if (!(ok = mbar_wait(&q_empty[qs], ((q_it >> 1) & 1u) ^ 1u, abort_flag))) break;
          mbar_expect_tx(&q_full[qs], kQueryBlock);
          tma_load_2d(smem_u32(q_smem + qs * kQueryBlock), part ? &map_ql : &map_q,
                      (2 * hp + h) * kHeadDim + half * kHalf, txt0 + t * kTT, &q_full[qs]);
        }
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- epilogue (warps 0-3)
    const int r = warp * 32 + lane;                        // token row inside the tile = TMEM lane
    const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
    uint32_t n = 0, head_it = 0, uses[kLogitTiles] = {0u, 0u};
    bool ok = true;
    for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x, ++n) {
      int row0, nrows, txt0, T, hp, heads;
      decode(item, row0, nrows, txt0, T, hp, heads);
      const uint32_t buf = n & 1u;
      const int ntt = (T + kTT - 1) / kTT;
      float best = -INFINITY;
      bool nonfinite = false;
      if (!(ok = mbar_wait(&acc_full[buf], (n >> 1) & 1u, abort_flag))) break;
      tc_fence_after();
      for (int h = 0; h < heads && ok; ++h, ++head_it) {
        const uint32_t cols = t_lane + buf * kTileN + h * kHeadDim;
        float ss = 0.f;
        // restage the head as bf16 hi + lo, 32 features at a time, once the previous head's products have read theirs
        if (!(ok = mbar_wait(kp_free, (head_it & 1u) ^ 1u, abort_flag))) break;
#pragma unroll 1
        for (int c4 = 0; c4 < 4; ++c4) {
          float v[32];
          tmem_ld32(cols + c4 * 32, v);
          uint32_t pk[16], pl[16];
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            float a = v[2 * e], b = v[2 * e + 1];
            ss += a * a + b * b;
            __nv_bfloat162 hi = __floats2bfloat162_rn(a, b);
            pk[e] = *reinterpret_cast<uint32_t*>(&hi);
            pl[e] = pack_bf16(a - __low2float(hi), b - __high2float(hi));
          }
          uint8_t* rowp = kp_smem + (c4 >> 1) * kBytesKp + r * 128;
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            int chunk = ((c4 & 1) * 4 + q) ^ (r & 7);
            *reinterpret_cast<uint4*>(rowp + chunk * 16) =
                make_uint4(pk[4 * q], pk[4 * q + 1], pk[4 * q + 2], pk[4 * q + 3]);
            *reinterpret_cast<uint4*>(rowp + 2 * kBytesKp + chunk * 16) =
                make_uint4(pl[4 * q], pl[4 * q + 1], pl[4 * q + 2], pl[4 * q + 3]);
          }
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        tc_fence_before();
        mbar_arrive(kp_ready);
        nonfinite |= !(ss <= 3.402823466e38f);
        float inv = 0.f;
        if (ss > 1.17549435e-38f) { inv = rsqrtf(ss); inv = inv * (1.5f - 0.5f * ss * inv * inv); }
        for (int t = 0; t < ntt; ++t) {
          const int slot = t & 1;
          if (!(ok = mbar_wait(&logit_full[slot], uses[slot] & 1u, abort_flag))) break;
          ++uses[slot];
          tc_fence_after();
#pragma unroll 1
          for (int c2 = 0; c2 < 2; ++c2) {
            const int jbase = t * kTT + c2 * 32;
            if (jbase >= T) break;
            float v[32];
            tmem_ld32(cols + slot * kTT + c2 * 32, v);
#pragma unroll
            for (int e = 0; e < 32; ++e)
              if (jbase + e < T) {
                nonfinite |= v[e] != v[e];
                best = fmaxf(best, v[e] * inv);
              }
          }
          tc_fence_before();
          mbar_arrive(&logit_empty[slot]);
        }
      }
      if (!ok) break;
      mbar_arrive(&acc_empty[buf]);            // projections and logits of the item have been read
      if (item == (int)blockIdx.x) wait_for_previous_kernel();      // the scores are filled with -inf
      if (r < nrows) {
        if (nonfinite) atomicOr(prm.status, kStatusNonFinite);
        else atomic_max_float(prm.s_query + row0 + r, best);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem_base, kTmemCols);
  if (threadIdx.x == 0 && *abort_flag) atomicOr(prm.status, kStatusTimeout);
}

}  // namespace tc
}  // namespace covspec
