// Eq. 10 with the identity embedding (e(x) = x, no projection heads) on the tensor cores, bf16 inputs.
//
//   S^query_i = max_j (x_i . q_j) / (|x_i| |q_j|)
// The tensor cores find the query elements that can attain the maximum, ordinary float32 arithmetic computes the score:
//   1. products of all tokens of a tile with the request's query elements by tcgen05.mma on the raw bf16 rows, float32
//      accumulators in TMEM, and the lengths in float32 from the same tiles while they lie in shared memory; X is read
//      from HBM once and nothing is converted or staged in between.
//   2. the accumulators truncate, by less than 2^-23 |x| |q| a step of 16 features (a fifth of that was measured).  A sum is
//      cut into as many groups of contiguous features as TMEM has columns for, up to eight, added up in float32: the
//      bound falls with their number.  Every query element within twice the bound of the largest value is a
//      candidate; nearly always there is one.
//   3. identity_exact_kernel computes the cosine of every candidate again, one warp per token, with the arithmetic of
//      cosmax_kernel in its order (score_kernels.cuh), and the largest is the score: the bits are those of that kernel,
//      whatever the batch a request comes in.  (Tensor-core sums as scores were off by 2.5e-7 to 2.1e-6 relative,
//      d = 1024-4096, against 6e-8 to 1e-7, and depended on the longest query of the call.)  A second launch because
//      a row is a handful of loads whose latency is all there is: it takes the whole chip's warps to wait for them.  With
//      step 3 in the first kernel, by eight warps a tile, 2 x 16384 tokens at d = 3584 took 121.7 us instead of 89.1 and 4 x 576 at
//      d = 1024 19.1 instead of 16.1 (the sums themselves as scores: 43.4 and 11.2; cosmax_kernel 1093 and 48.9).
//
// One CTA per 128-token tile of a request (or per 64 tokens, while that leaves at most two CTAs per SM: a
// block is bound by the latency of its loads and by shared-memory bandwidth); the request's query elements pass in groups of up to 128.
// Warps 0-3: one token per thread (length of x, candidates); 4-7: one query element per thread (length of
// q); warp 8: TMA producer; warp 9: MMA issuer and TMEM owner.  Bound by HBM (X once).  cosmax_kernel (one warp per token)
// reads every query element once per token through L1: 16 requests of 400-729 tokens, d = 2048, 210 us for 37 MB.
#pragma once
#include <float.h>

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
constexpr int kGroupChunks = 4;          // k-chunks per accumulation group, if TMEM has the columns
constexpr int kTailBytes = 2048;         // barriers, reciprocal query lengths

// Requests handed over by value (the allocation-free entry point, which has no plan on the device).
constexpr int kInlineReqs = 64;
struct InlineReqs {
  int4 e[kInlineReqs];                   // vis_off, n, txt_off, t
  int tile_off[kInlineReqs];
};

struct IdParams {
  float* inv_q;                          // reciprocal query lengths for identity_exact_kernel
  float margin;                          // candidates: within margin |x| |q| of the largest product
  int per_group, groups;                 // accumulation groups: k-chunks each, their number
  int pairs;                             // 1: codes of two candidates fit (see kPairRows)
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
// The same for the 32 sums in which qnorm_kernel's lanes take a row: feature k goes to sum k % 32, in ascending order.
__device__ __forceinline__ void add_row_squares_by_lane(const uint8_t* tile, int r, unsigned long long (&acc)[16]) {
  const uint8_t* row = tile + r * 128;
#pragma unroll
  for (int c = 0; c < 8; ++c) {
    const uint4 v = *reinterpret_cast<const uint4*>(row + ((c ^ (r & 7)) * 16));
    const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      unsigned long long x;
      asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "r"(u[e] << 16), "r"(u[e] & 0xffff0000u));
      asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc[(4 * c + e) & 15]) : "l"(x));
    }
  }
}
// Their total as warp_sum adds the lanes up.
__device__ __forceinline__ float total_by_lane(const unsigned long long (&acc)[16]) {
  float s[32];
#pragma unroll
  for (int e = 0; e < 16; ++e) asm("mov.b64 {%0, %1}, %2;" : "=f"(s[2 * e]), "=f"(s[2 * e + 1]) : "l"(acc[e]));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int l = 0; l < o; ++l) s[l] += s[l + o];
  return s[0];
}
// 1 / sqrt(ss); 0 for a zero row, NaN for a row that is not finite.
__device__ __forceinline__ float inverse_length(float ss) {
  if (!(ss <= 3.402823466e38f)) return __int_as_float(0x7fc00000);
  if (!(ss > 1.17549435e-38f)) return 0.f;
  float inv = rsqrtf(ss);
  return inv * (1.5f - 0.5f * ss * inv * inv);
}

// Cosine of a token with a query element, by one warp, as cosmax_kernel computes it; inv: the token's reciprocal length.
__device__ __forceinline__ float exact_cosine(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ q,
                                              float inv_q, int d, int lane, float& inv) {
  constexpr int kFlight = 8;                             // iterations of 128 features whose loads are in flight together
  float ss = 0.f, dot = 0.f;
  auto add = [&](const uint2& xr, const uint2& qr) {
    const float v[4] = {__uint_as_float(xr.x << 16), __uint_as_float(xr.x & 0xffff0000u), __uint_as_float(xr.y << 16), __uint_as_float(xr.y & 0xffff0000u)};
    const float u[4] = {__uint_as_float(qr.x << 16), __uint_as_float(qr.x & 0xffff0000u), __uint_as_float(qr.y << 16), __uint_as_float(qr.y & 0xffff0000u)};
    const float4 w = make_float4(u[0] * inv_q, u[1] * inv_q, u[2] * inv_q, u[3] * inv_q);
    ss += v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
    dot += v[0] * w.x + v[1] * w.y + v[2] * w.z + v[3] * w.w;
  };
  int k = lane * 4;
  for (int left = d >> 7; left > 0; left -= kFlight) {
    uint2 vx[kFlight], vq[kFlight];
#pragma unroll
    for (int i = 0; i < kFlight; ++i)
      if (i < left) {
        vx[i] = __ldg(reinterpret_cast<const uint2*>(x + k + 128 * i));
        vq[i] = __ldg(reinterpret_cast<const uint2*>(q + k + 128 * i));
      }
#pragma unroll
    for (int i = 0; i < kFlight; ++i)
      if (i < left) add(vx[i], vq[i]);
    k += 128 * min(left, kFlight);
  }
  if (k < d) add(__ldg(reinterpret_cast<const uint2*>(x + k)), __ldg(reinterpret_cast<const uint2*>(q + k)));
  ss = warp_sum(ss);
  inv = 0.f;
  if (ss > FLT_MIN) { inv = rsqrtf(ss); inv = inv * (1.5f - 0.5f * ss * inv * inv); }
  return warp_sum(dot) * inv;
}

// What the first kernel leaves in a token's place for identity_exact_kernel: a NaN that no score has (scores that are not
// finite are the positive one) with the row of its only candidate in the query array; in arrays of up to kPairRows
// rows, with the row of the first of two and the distance to the second; or kAll: every query element of the request (three
// candidates and more, lengths near the float32 range's lower end).
constexpr uint32_t kCode = 0xffc00000u, kAll = 0x3fffffu;
constexpr long long kCodeRows = (1ll << 22) - 1;
constexpr int kPairBits = 14, kPairReach = 254;
constexpr long long kPairRows = 1ll << kPairBits;

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
  // Without an activity stream beside it (no status word) the second kernel may come up already; its blocks would
  // take that stream's places otherwise.  Not before this CTA has its TMEM: the next call's first kernel allocates too.
  if (prm.status == nullptr) launch_dependents_now();
  wait_for_previous_kernel();

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
  const int group_cols = (prm.n_cols + 31) & ~31;
  // 16 columns of the products: the groups added up in their order
  auto products16 = [&](uint32_t t_col, float (&v)[16]) {
    tmem_ld16(t_col, v);
    for (int g = 1; g < prm.groups; ++g) {
      float u[16];
      tmem_ld16(t_col + g * group_cols, u);
#pragma unroll
      for (int e = 0; e < 16; ++e) v[e] += u[e];
    }
  };

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
          const int g = kc / prm.per_group;
#pragma unroll
          for (int k = 0; k < kChunk / 16; ++k)
            umma_bf16(tmem_base + g * group_cols, adesc + 2 * k, bdesc + 2 * k, idesc, (kc - g * prm.per_group + k) != 0);
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
    float best = -INFINITY, len_x = 0.f, inv_x = 0.f;    // best: largest product so far, divided by the query length
    bool nonfinite = false, ok = true;
    int s = 0;
    // up to two candidates so far (product and query row; a row of -1: none), and the largest product of those beyond
    float c1 = 0.f, c2 = 0.f, beyond = -INFINITY;
    int q1 = -1, q2 = -1;
    bool all = false;
    uint32_t ph = 0;
    for (int pass = 0; pass < passes; ++pass) {
      if (tokens) {
        unsigned long long sq[4] = {0ull, 0ull, 0ull, 0ull};
        const bool measure = pass == 0 && (warp & 3) * 32 < nrows;
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          ok = ok && wait(&full[s], ph);
          if (measure) add_row_squares(smem + (size_t)s * prm.stage_bytes, r, sq);
          __syncwarp();
          if (lane == 0) mbar_arrive(&empty[s]);
          if (++s == prm.stages) { s = 0; ph ^= 1u; }
        }
        if (pass == 0) {
          const float ss = total_squares(sq);
          inv_x = inverse_length(ss);
          len_x = ss * inv_x;
          nonfinite = inv_x != inv_x;
        }
        named_barrier(1, 256);                           // the previous pass no longer reads inv_q
      } else {
        unsigned long long sq[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) sq[e] = 0ull;
        const bool measure = r < prm.n_cols;
        for (int kc = 0; kc < prm.k_chunks; ++kc) {
          ok = ok && wait(&full[s], ph);
          if (measure) add_row_squares_by_lane(smem + (size_t)s * prm.stage_bytes + R * 128, r, sq);
          __syncwarp();
          if (lane == 0) mbar_arrive(&empty[s]);
          if (++s == prm.stages) { s = 0; ph ^= 1u; }
        }
        named_barrier(1, 256);
        if (measure) {
          const float inv = ok ? inverse_length(total_by_lane(sq)) : __int_as_float(0x7fc00000);
          inv_q[r] = inv;
          if (at == 0 && pass * prm.n_cols + r < T) prm.inv_q[txt_off + pass * prm.n_cols + r] = inv;
        }
      }
      named_barrier(1, 256);
      if (tokens) {
        ok = ok && wait(acc_full, pass & 1u);
        tc_fence_after();
        const int cols = min(prm.n_cols, T - pass * prm.n_cols);
        float top = -INFINITY, most = 0.f;
#pragma unroll 1
        for (int c0 = 0; c0 < cols; c0 += 16) {
          float v[16];
          products16(t_lane + c0, v);
#pragma unroll
          for (int e = 0; e < 16; ++e)
            if (c0 + e < cols) {
              const float c = v[e] * inv_q[c0 + e];
              nonfinite |= c != c;
              top = fmaxf(top, c);
              most = fmaxf(most, inv_q[c0 + e]);
            }
        }
        // |x| |q| so small that the products themselves may be lost below the float32 range: every element is a candidate
        all |= inv_x == 0.f || !(most * inv_x <= 1.2e24f);
        best = fmaxf(best, top);
        const float limit = best - prm.margin * len_x;
        if (q2 >= 0 && c2 < limit) q2 = -1;
        if (q1 >= 0 && c1 < limit) { c1 = c2; q1 = q2; q2 = -1; }
#pragma unroll 1
        for (int c0 = 0; c0 < cols; c0 += 16) {
          float v[16];
          products16(t_lane + c0, v);
#pragma unroll
          for (int e = 0; e < 16; ++e) {
            const float c = c0 + e < cols ? v[e] * inv_q[c0 + e] : -INFINITY;
            if (c >= limit) {
              const int row = txt_off + pass * prm.n_cols + c0 + e;
              if (q1 < 0) { c1 = c; q1 = row; }
              else if (q2 < 0) { c2 = c; q2 = row; }
              else beyond = fmaxf(beyond, c);
            }
          }
        }
        if (beyond < limit) beyond = -INFINITY;
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
    }
    // a wait that gave up leaves NaN, for callers that have no status word to look at
    if (tokens && r < nrows) {
      uint32_t code = (uint32_t)q1;
      if (q2 >= 0) code |= (uint32_t)(q2 - q1) << kPairBits;
      if (all || q1 < 0 || beyond > -INFINITY || (q2 >= 0 && (!prm.pairs || q2 - q1 > kPairReach))) code = kAll;
      reinterpret_cast<uint32_t*>(prm.s_query)[row0 + r] = nonfinite || !ok ? 0x7fc00000u : kCode | code;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem_base, kColumns);
  if (threadIdx.x == 0 && *abort_flag && prm.status != nullptr) atomicOr(prm.status, kStatusTimeout);
}

// The scores from the candidates that identity_tc_kernel found; one warp per token, bound by the latency and issue of a
// row's loads and sums (32,768 tokens, d = 3584: about 45 us, 36 of them HBM).
__global__ void __launch_bounds__(256, 4)
identity_exact_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ q,
                      const float* __restrict__ inv_q, const __grid_constant__ InlineReqs reqs, const IdParams prm, int d,
                      int first, int rows) {
  const int row = first + (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  wait_for_previous_kernel();
  launch_dependents_now();
  if (row >= first + rows) return;
  const uint32_t code = __float_as_uint(prm.s_query[row]);
  if ((code & kCode) != kCode) return;                   // not finite
  int low, high, step;                                   // candidates low, low + step, .. high
  if ((code & kAll) == kAll) {
    if (prm.plan != nullptr) {
      const int b = find_request(row, prm.batch, [&](int i) { return prm.plan[i].vis_off; });
      low = prm.plan[b].txt_off; high = low + prm.plan[b].t - 1;
    } else {
      const int b = find_request(row, prm.batch, [&](int i) { return reqs.e[i].x; });
      low = reqs.e[b].z; high = low + reqs.e[b].w - 1;
    }
    step = 1;
  } else {
    low = (int)(code & (prm.pairs ? (uint32_t)kPairRows - 1u : kAll));
    step = max(1, prm.pairs ? (int)((code & kAll) >> kPairBits) : 0);
    high = prm.pairs ? low + (int)((code & kAll) >> kPairBits) : low;
  }
  float best = -FLT_MAX;
  bool nonfinite = false;
  for (int j = low; j <= high; j += step) {
    const float iq = inv_q[j];
    float inv;
    best = fmaxf(best, exact_cosine(x + (size_t)row * d, q + (size_t)j * d, iq, d, lane, inv));
    nonfinite |= iq != iq;
    if (inv == 0.f) break;                               // a zero token: 0 with every element
  }
  if (lane == 0) prm.s_query[row] = nonfinite ? __int_as_float(0x7fc00000) : best;
}

}  // namespace ident
}  // namespace covspec
