// Shared pieces of the tensor-core kernels of the query-aware score (Eq. 10) with per-head linear embeddings, and
// the query side: Qp = Q * Wq^T, normalised per head and written as bf16 hi + lo for the visual side
// (relevance_vis.cuh).
//
// Work item of the query side: one 128-row tile of all query elements, one or two heads.  Warp roles
// (192 threads): warps 0-3 epilogue (one TMEM lane = one query element each), warp 4 TMA producer, warp 5 MMA
// issuer and TMEM owner; two accumulators, so that the epilogue of an item runs beside the next one's main
// loop.  Two 96 KB stages of two chunks instead of four of one were slower (15.0 -> 17.6 us at d = 2048).
// An item takes as long as its chain of chunks (about 500 cycles each with one head).  Sharing the inner dimension among
// four CTAs gained about 1 us of a call with one request and moved scores by 1e-6, enough to exchange near-tied tokens;
// loading only the rows that a lone tile has gained nothing.
// Every mbarrier wait is bounded; on expiry the CTA raises a status bit, leaves its loops, frees TMEM and exits.
#pragma once
#include "tc_common.cuh"

namespace covspec {

namespace tc {

constexpr int kTileM = 128;            // tokens per tile (UMMA M)
constexpr int kTileN = 256;            // projected features per pass: one pair of heads (UMMA N)
constexpr int kHeadDim = 128;
constexpr int kBK = 64;                // bf16 elements per k-chunk = one 128-byte swizzle row
constexpr int kHalf = 64;              // features of a restaged half head (one 128-byte swizzle row)
constexpr int kBytesA = kTileM * kBK * 2;          // 16 KB
constexpr int kBytesB = kTileN * kBK * 2;          // 32 KB
constexpr int kBytesStage = kBytesA + kBytesB;
constexpr int kBytesKp = kTileM * kHalf * 2;       // 16 KB: [128 x 64] of one half head; hi and lo
constexpr int kTmemCols = 512;
constexpr int kQueryStages = 4;        // of two heads (48 KB); six of one
constexpr int kQueryMaxStages = kQueryStages * kBytesStage / (kBytesA + kHeadDim * kBK * 2);
// 193 KB would do.  A little more than the visual side's 222 KB, so that what finds room beside one finds room beside the other:
// with smaller blocks of the activity stream than today's one per SM, more room made those gather on few SMs.
constexpr int kQuerySmem = 225 * 1024;
static_assert(kQueryStages * kBytesStage + 1024 <= kQuerySmem, "ring and barriers");

struct QueryParams {
  int n_items;          // (128-row tile, group of heads) pairs
  int n_groups;         // groups of heads
  int group_heads;      // heads per item, 2 or 1
  int n_heads;
  int k_chunks;         // ceil(d / 64)
  int P;                // n_heads * 128
  long long rows_total; // query rows
  __nv_bfloat16* qn_out;// out: hi [rows_total, P] followed by lo at qn_out + qn_lo_off
  long long qn_lo_off;
  float* fill;          // score array to fill with -inf for the visual side's launch that follows
  long long fill_n;     // (nullptr: nothing to fill)
  int* status;
};

__global__ void __launch_bounds__(192, 1)
query_embed_kernel(const __grid_constant__ CUtensorMap map_a,   // Q: [rows, d]
                   const __grid_constant__ CUtensorMap map_b,   // Wq: [P, d]
                   const QueryParams prm) {
  extern __shared__ __align__(1024) uint8_t rel_smem_raw[];
  uint8_t* smem = rel_smem_raw;
  if (smem_u32(smem) & 1023u) {          // the swizzled tiles need a 1024-byte aligned base
    if (threadIdx.x == 0) atomicOr(prm.status, kStatusTimeout);
    return;
  }
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + kQueryStages * kBytesStage);
  uint64_t* full = bars;                     // [kQueryMaxStages]
  uint64_t* empty = full + kQueryMaxStages;  // [kQueryMaxStages]
  uint64_t* acc_full = empty + kQueryMaxStages;   // [2]
  uint64_t* acc_empty = acc_full + 2;             // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kQueryMaxStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 128); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) tmem_alloc(tmem_slot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // The visual side starts while the query side still runs, on the SMs that it leaves: its main loops need
  // nothing of it; what it fills in is waited for before the first query tile and the first maximum.
  launch_dependents_now();
  if (prm.fill != nullptr) {
    // the visual side combines pairs of heads with an atomic max: its score array starts at -inf
    for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < prm.fill_n;
         i += (long long)gridDim.x * blockDim.x)
      prm.fill[i] = -INFINITY;
  }

  // Epilogue of one head: unit-length bf16 slices (hi and lo) of the tile's projected query elements, which lie from
  // column `cols` of TMEM on.
  const int r = (warp & 3) * 32 + lane;                    // row inside the tile = TMEM lane
  const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
  auto store_head = [&](int row0, int nrows, int head, uint32_t cols) {
    float ss = 0.f;
#pragma unroll 1
    for (int c4 = 0; c4 < 4; ++c4) {
      float v[32];
      tmem_ld32(cols + c4 * 32, v);
#pragma unroll
      for (int e = 0; e < 32; ++e) ss += v[e] * v[e];
    }
    float inv = 0.f;
    if (ss > 1.17549435e-38f) { inv = rsqrtf(ss); inv = inv * (1.5f - 0.5f * ss * inv * inv); }
    if (!(ss <= 3.402823466e38f)) inv = __int_as_float(0x7fc00000);
#pragma unroll 1
    for (int c4 = 0; c4 < 4; ++c4) {
      float v[32];
      tmem_ld32(cols + c4 * 32, v);
      if (r < nrows) {
        __nv_bfloat16* dst = prm.qn_out + (size_t)(row0 + r) * prm.P + (size_t)head * kHeadDim + c4 * 32;
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          uint32_t ph[4], pw[4];
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            float a = v[8 * q + 2 * e] * inv, b = v[8 * q + 2 * e + 1] * inv;
            __nv_bfloat162 hi = __floats2bfloat162_rn(a, b);
            ph[e] = *reinterpret_cast<uint32_t*>(&hi);
            pw[e] = pack_bf16(a - __low2float(hi), b - __high2float(hi));
          }
          *reinterpret_cast<uint4*>(dst + q * 8) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
          *reinterpret_cast<uint4*>(dst + prm.qn_lo_off + q * 8) = make_uint4(pw[0], pw[1], pw[2], pw[3]);
        }
      }
    }
  };

  const int stage_bytes = kBytesA + prm.group_heads * kHeadDim * kBK * 2, stages = kQueryStages * kBytesStage / stage_bytes;

  if (warp == 4) {
    // ---------------------------------------------------------------- TMA producer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x) {
        const int row0 = item / prm.n_groups * kTileM, head0 = item % prm.n_groups * prm.group_heads;
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = mbar_wait(&empty[s], ph, abort_flag))) break;
          mbar_expect_tx(&full[s], stage_bytes);
          const uint32_t dst = smem_u32(smem + s * stage_bytes);
          tma_load_2d(dst, &map_a, kc * kBK, row0, &full[s]);
          tma_load_2d(dst + kBytesA, &map_b, kc * kBK, head0 * kHeadDim, &full[s]);
          if (++s == stages) { s = 0; ph ^= 1u; }
        }
      }
    }
    __syncwarp();
  } else if (warp == 5) {
    // ---------------------------------------------------------------- MMA issuer
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 0, n = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x, ++n) {
        const uint32_t buf = n & 1u;
        if (!(ok = mbar_wait(&acc_empty[buf], ((n >> 1) & 1u) ^ 1u, abort_flag))) break;
        tc_fence_after();
        // a lone last head takes half the columns (see relevance_vis_kernel)
        const int head0 = item % prm.n_groups * prm.group_heads;
        const uint32_t idesc = umma_idesc(kTileM, min(prm.group_heads, prm.n_heads - head0) * kHeadDim);
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = mbar_wait(&full[s], ph, abort_flag))) break;
          tc_fence_after();
          const uint32_t addr = smem_u32(smem + s * stage_bytes);
          const uint64_t adesc = umma_desc(addr), bdesc = umma_desc(addr + kBytesA);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            umma_bf16(tmem_base + buf * kTileN, adesc + 2 * k, bdesc + 2 * k, idesc, (kc | k) != 0);
          umma_commit(&empty[s]);
          if (++s == stages) { s = 0; ph ^= 1u; }
        }
        if (ok) umma_commit(&acc_full[buf]);
      }
    }
    __syncwarp();
  } else {
    // ---------------------------------------------------------------- epilogue (warps 0-3)
    uint32_t n = 0;
    bool ok = true;
    for (int item = blockIdx.x; item < prm.n_items && ok; item += gridDim.x, ++n) {
      const int row0 = item / prm.n_groups * kTileM, head0 = item % prm.n_groups * prm.group_heads;
      const long long rem = prm.rows_total - row0;
      const uint32_t buf = n & 1u;
      if (!(ok = mbar_wait(&acc_full[buf], (n >> 1) & 1u, abort_flag))) break;
      tc_fence_after();
      const int heads = min(prm.group_heads, prm.n_heads - head0);
      for (int h = 0; h < heads; ++h)
        store_head(row0, rem < kTileM ? (int)rem : kTileM, head0 + h, t_lane + buf * kTileN + h * kHeadDim);
      tc_fence_before();
      mbar_arrive(&acc_empty[buf]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem_base, kTmemCols);
  if (threadIdx.x == 0 && *abort_flag) atomicOr(prm.status, kStatusTimeout);
}

}  // namespace tc
}  // namespace covspec
