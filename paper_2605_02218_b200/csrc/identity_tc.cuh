// Eq. 10 with the identity embedding (e(x) = x, no projection heads) on the tensor cores, bf16 inputs.
//
//   S^query_i = max_j (x_i . q_j) / (|x_i| |q_j|)
// bf16 inputs enter the products exactly: one tcgen05.mma per 16 features on the raw rows, float32
// accumulators in TMEM, and the two lengths in float32 from the same tiles while they lie in shared
// memory, so that X is read once and nothing is converted or staged in between.  The accumulation is cut
// into up to four column groups of TMEM, each over a contiguous range of features, that the epilogue adds
// up in registers: the tensor core's sums truncate, and short chains keep that near the rounding of
// ordinary float32 sums.
//
// One CTA per 128-token tile of a request (or per 64 tokens, while that leaves at most two CTAs per SM: a
// block is bound by the latency of its loads and by shared-memory bandwidth); the request's query elements pass in groups of up to 128.
// Warps 0-3: one token per thread (length of x, epilogue); 4-7: one query element per thread (length of
// q); warp 8: TMA producer; warp 9: MMA issuer and TMEM owner.  Bound by HBM (X once).  The CUDA-core
// kernel (cosmax_kernel, one warp per token) read every query element once per token through L1: 16
// requests of 400-729 tokens, d = 2048, 210 us for 37 MB.
#pragma once
#include "tc_common.cuh"

namespace covspec {
namespace ident {

using namespace tc;

constexpr int kTokens = 128;             // tokens per tile (UMMA M)
constexpr int kQueries = 128;            // query elements per pass (UMMA N at most)
constexpr int kChunk = 64;               // features per k-chunk (one 128-byte swizzle row)
constexpr int kMaxStages = 12;
constexpr int kColumns = 256;            // TMEM columns: two CTAs fit on an SM
constexpr int kIdThreads = 320;
constexpr int kGroupChunks = 8;          // k-chunks per accumulation group, if TMEM has the columns
constexpr int kTailBytes = 2048;         // barriers, reciprocal query lengths

// Requests handed over by value (the allocation-free entry point, which has no plan on the device).
constexpr int kInlineReqs = 64;
struct InlineReqs {
  int4 e[kInlineReqs];                   // vis_off, n, txt_off, t
  int tile_off[kInlineReqs];
};

struct IdParams {
  const ReqPlan* plan;                   // or nullptr: the inline requests
  int batch;
  int k_chunks;
  int n_cols;                            // query elements per pass, a multiple of 16
  int stages, stage_bytes;
  int tile_rows;                         // tokens per block: 128 or 64
  float* s_query;
  int* status;                           // may be nullptr
  uint32_t spin_limit;                   // polls after which a wait gives up
};

// Sums of squares of one 128-byte row of a swizzled tile, in four pairs of running sums (packed float32
// multiply-adds; short chains, the loads of a row in flight together).
__device__ __forceinline__ void add_row_squares(const uint8_t* tile, int r, unsigned long long (&acc)[4]) {
  const uint8_t* row = tile + r * 128;
  uint4 v[8];
#pragma unroll
  for (int c = 0; c < 8; ++c) v[c] = *reinterpret_cast<const uint4*>(row + ((c ^ (r & 7)) * 16));
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint32_t u[4] = {v[c].x, v[c].y, v[c].z, v[c].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      unsigned long long x;
      asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(u[e] << 16), "r"(u[e] & 0xffff0000u));
      asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc[e]) : "l"(x));
    }
  }
}
__device__ __forceinline__ float total_squares(const unsigned long long (&acc)[4]) {
  float s = 0.f;
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    float lo, hi;
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(acc[e]));
    s += lo + hi;
  }
  return s;
}
// 1 / sqrt(ss); 0 for a zero row, NaN for a row that is not finite.
__device__ __forceinline__ float inverse_length(float ss) {
  if (!(ss <= 3.402823466e38f)) return __int_as_float(0x7fc00000);
  if (!(ss > 1.17549435e-38f)) return 0.f;
  float inv = rsqrtf(ss);
  return inv * (1.5f - 0.5f * ss * inv * inv);
}

__global__ void __launch_bounds__(kIdThreads, 2)
identity_tc_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_q,
                   const __grid_constant__ InlineReqs reqs, const IdParams prm) {
  extern __shared__ uint8_t id_smem_raw[];
  uint8_t* smem = id_smem_raw + ((0u - smem_u32(id_smem_raw)) & 1023u);
  uint8_t* tail = smem + (size_t)prm.stages * prm.stage_bytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(tail);      // [kMaxStages]
  uint64_t* empty = full + kMaxStages;                     // [kMaxStages]
  uint64_t* acc_full = empty + kMaxStages;
  uint64_t* acc_empty = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_empty + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* inv_q = reinterpret_cast<float*>(tail + 512);     // [kQueries]
  const int warp = warp_index(), lane = threadIdx.x & 31;
  auto wait = [&](uint64_t* bar, uint32_t parity) { return mbar_wait_limited(bar, parity, abort_flag, prm.spin_limit); };

  if (threadIdx.x == 0) {
    for (int s = 0; s < prm.stages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 9); }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 4);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 9) tmem_alloc(tmem_slot, kColumns);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // tile_rows = 64: two blocks share a 128-token tile (the MMA still computes 128 rows: the upper 64 read whatever
  // follows in the ring and go nowhere)
  const int R = prm.tile_rows, item = (int)blockIdx.x / (kTokens / R), half = (int)blockIdx.x % (kTokens / R);
  int vis_off, n, txt_off, T, tile;
  if (prm.plan != nullptr) {
    const int b = find_request(item, prm.batch, [&](int q) { return prm.plan[q].tile_off; });
    vis_off = prm.plan[b].vis_off; n = prm.plan[b].n; txt_off = prm.plan[b].txt_off; T = prm.plan[b].t;
    tile = item - prm.plan[b].tile_off;
  } else {
    const int b = find_request(item, prm.batch, [&](int q) { return reqs.tile_off[q]; });
    vis_off = reqs.e[b].x; n = reqs.e[b].y; txt_off = reqs.e[b].z; T = reqs.e[b].w;
    tile = item - reqs.tile_off[b];
  }
  const int at = tile * kTokens + half * R, row0 = vis_off + at, nrows = min(R, n - at);
  const int passes = nrows > 0 ? (T + prm.n_cols - 1) / prm.n_cols : 0;
  // accumulation groups: contiguous ranges of k-chunks, one set of TMEM columns each
  const int group_cols = (prm.n_cols + 31) & ~31;
  const int n_groups = max(1, min(kColumns / group_cols, (prm.k_chunks + kGroupChunks - 1) / kGroupChunks));
  const int per_group = (prm.k_chunks + n_groups - 1) / n_groups;
  const int groups_used = (prm.k_chunks + per_group - 1) / per_group;

  if (warp == 8) {
    if (lane == 0) {
      int s = 0;
      uint32_t ph = 1;
      bool ok = true;
      for (int pass = 0; pass < passes && ok; ++pass)
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = wait(&empty[s], ph))) break;
          mbar_expect_tx(&full[s], prm.stage_bytes);
          const uint32_t dst = smem_u32(smem + (size_t)s * prm.stage_bytes);
          tma_load_2d(dst, &map_x, kc * kChunk, row0, &full[s]);
          tma_load_2d(dst + R * 128, &map_q, kc * kChunk, txt_off + pass * prm.n_cols, &full[s]);
          if (++s == prm.stages) { s = 0; ph ^= 1u; }
        }
    }
    __syncwarp();
  } else if (warp == 9) {
    if (lane == 0) {
      const uint32_t idesc = umma_idesc(kTokens, prm.n_cols);
      int s = 0;
      uint32_t ph = 0;
      bool ok = true;
      for (int pass = 0; pass < passes && ok; ++pass) {
        if (!(ok = wait(acc_empty, (pass & 1u) ^ 1u))) break;
        tc_fence_after();
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          if (!(ok = wait(&full[s], ph))) break;
          tc_fence_after();
          const uint32_t x_addr = smem_u32(smem + (size_t)s * prm.stage_bytes);
          const uint64_t adesc = umma_desc(x_addr), bdesc = umma_desc(x_addr + R * 128);
          const int g = kc / per_group;
#pragma unroll
          for (int k = 0; k < kChunk / 16; ++k)
            umma_bf16(tmem_base + g * group_cols, adesc + 2 * k, bdesc + 2 * k, idesc, (kc - g * per_group + k) != 0);
          umma_commit(&empty[s]);
          if (++s == prm.stages) { s = 0; ph ^= 1u; }
        }
        if (ok) umma_commit(acc_full);
      }
    }
    __syncwarp();
  } else {
    const int r = (warp & 3) * 32 + lane;              // token (warps 0-3) or query element (4-7) of the tile
    const bool tokens = warp < 4;
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    float best = -INFINITY, inv_x = 0.f;
    bool nonfinite = false, ok = true;
    int s = 0;
    uint32_t ph = 0;
    for (int pass = 0; pass < passes; ++pass) {
      unsigned long long sq[4] = {0ull, 0ull, 0ull, 0ull};
      const bool measure = tokens ? pass == 0 && (warp & 3) * 32 < nrows : r < prm.n_cols;
      for (int kc = 0; kc < prm.k_chunks; ++kc) {
        ok = ok && wait(&full[s], ph);
        if (measure) add_row_squares(smem + (size_t)s * prm.stage_bytes + (tokens ? 0 : R * 128), r, sq);
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[s]);
        if (++s == prm.stages) { s = 0; ph ^= 1u; }
      }
      if (tokens && pass == 0) { inv_x = inverse_length(total_squares(sq)); nonfinite = inv_x != inv_x; }
      named_barrier(1, 256);                           // the previous pass no longer reads inv_q
      if (!tokens && measure) inv_q[r] = inverse_length(total_squares(sq));
      named_barrier(1, 256);
      if (tokens) {
        ok = ok && wait(acc_full, pass & 1u);
        tc_fence_after();
        const int cols = min(prm.n_cols, T - pass * prm.n_cols);
#pragma unroll 1
        for (int c0 = 0; c0 < cols; c0 += 16) {
          float v[16];
          tmem_ld16(t_lane + c0, v);
          for (int g = 1; g < groups_used; ++g) {
            float u[16];
            tmem_ld16(t_lane + g * group_cols + c0, u);
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] += u[e];
          }
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (c0 + e < cols) {
              const float c = v[e] * inv_q[c0 + e];
              nonfinite |= c != c;
              best = fmaxf(best, c);
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
    }
    // a wait that gave up leaves NaN, for callers that have no status word to look at
    if (tokens && r < nrows) prm.s_query[row0 + r] = nonfinite || !ok ? __int_as_float(0x7fc00000) : best * inv_x;
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem_base, kColumns);
  if (threadIdx.x == 0 && *abort_flag && prm.status != nullptr) atomicOr(prm.status, kStatusTimeout);
}

}  // namespace ident
}  // namespace covspec
