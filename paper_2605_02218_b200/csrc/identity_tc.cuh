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
//   3. the cosine of every candidate is computed again by one warp per token, with the arithmetic of cosmax_kernel in its
//      order (score_kernels.cuh), and the largest is the score: the bits are those of that kernel, whatever the
//      batch a request comes in.  (Tensor-core sums as scores were off by 2.5e-7 to 2.1e-6 relative, d = 1024-4096,
//      against 6e-8 to 1e-7, and depended on the longest query of the call.)  One or two candidates
//      of a token go to identity_exact_kernel, which has the whole chip's warps to wait for the rows; more of them, and
//      requests of more than one pass, are seen to here.  (All of it here: 4 requests of 576 tokens, d = 1024, 32 query
//      elements 19.1 us, so 17.2; 16 of 400-729 at d = 2048 beside the activity stream 66.8 and 61.2; 2 of 16384 at
//      d = 3584 121.7 and 93.5: a single token with two candidates held a tile up for 3 to 18 us.)
//
// One CTA per 128-token tile of a request (or per 64 tokens, while that leaves at most two CTAs per SM: a
// block is bound by the latency of its loads and by shared-memory bandwidth); the request's query elements pass in groups of up to 128.
// Warps 0-3: one token per thread (length of x, candidates); 4-7: one query element per thread (length of
// q); 0-7: step 3; warp 8: TMA producer; warp 9: MMA issuer and TMEM owner.  Bound by HBM (X once).  cosmax_kernel (one warp
// per token) reads every query element once per token through L1: 16 requests of 400-729 tokens, d = 2048, 210 us
// for 37 MB.
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
// barriers (512), reciprocal query lengths [kQueries], best exact cosine [kTokens], candidate bits [kTokens][kQueries]
constexpr int kTailBytes = 512 + kQueries * 4 + kTokens * 4 + kTokens * kQueries / 8;

// Requests handed over by value (the allocation-free entry point, which has no plan on the device).
constexpr int kInlineReqs = 64;
struct InlineReqs {
  int4 e[kInlineReqs];                   // vis_off, n, txt_off, t
  int tile_off[kInlineReqs];
};

struct IdParams {
  const __nv_bfloat16* x;                // the arrays behind the tensor maps
  const __nv_bfloat16* q;
  int d;
  float* inv_q;                          // reciprocal query lengths for identity_exact_kernel
  float margin;                          // candidates: within margin |x| |q| of the largest product
  int per_group, groups;                 // accumulation groups: k-chunks each, their number
  int defer;                             // candidates that may be left to identity_exact_kernel: 0, 1 or 2
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

// Takes the lowest set bit out of a set of 128; -1: none left.
__device__ __forceinline__ int next_candidate(uint4& m) {
  if (m.x) { const int b = __ffs((int)m.x) - 1; m.x &= m.x - 1u; return b; }
  if (m.y) { const int b = __ffs((int)m.y) - 1; m.y &= m.y - 1u; return 32 + b; }
  if (m.z) { const int b = __ffs((int)m.z) - 1; m.z &= m.z - 1u; return 64 + b; }
  if (m.w) { const int b = __ffs((int)m.w) - 1; m.w &= m.w - 1u; return 96 + b; }
  return -1;
}

// Cosines of PT tokens with a query element each, by one warp, as cosmax_kernel computes them; *inv: the tokens'
// reciprocal lengths.  A row is a handful of loads per lane, whose latency is all there is: several at a time.
template <int PT, int UNROLL>
__device__ __forceinline__ void exact_cosines(const __nv_bfloat16* const (&x)[PT], const __nv_bfloat16* const (&q)[PT],
                                              const float (&inv_q)[PT], int d, int lane, float (&inv)[PT], float (&dot)[PT]) {
  float ss[PT];
#pragma unroll
  for (int p = 0; p < PT; ++p) ss[p] = dot[p] = 0.f;
  auto add = [&](int p, const uint2& xr, const uint2& qr) {
    const float v[4] = {__uint_as_float(xr.x << 16), __uint_as_float(xr.x & 0xffff0000u), __uint_as_float(xr.y << 16), __uint_as_float(xr.y & 0xffff0000u)};
    const float u[4] = {__uint_as_float(qr.x << 16), __uint_as_float(qr.x & 0xffff0000u), __uint_as_float(qr.y << 16), __uint_as_float(qr.y & 0xffff0000u)};
    const float4 w = make_float4(u[0] * inv_q[p], u[1] * inv_q[p], u[2] * inv_q[p], u[3] * inv_q[p]);
    ss[p] += v[0] * v[0] + v[1] * v[1] + v[2] * v[2] + v[3] * v[3];
    dot[p] += v[0] * w.x + v[1] * w.y + v[2] * w.z + v[3] * w.w;
  };
  int k = lane * 4;
  for (int left = d >> 7; left > 0; left -= UNROLL) {    // 128 features an iteration, UNROLL of them in flight
    uint2 vx[UNROLL][PT], vq[UNROLL][PT];
#pragma unroll
    for (int i = 0; i < UNROLL; ++i)
#pragma unroll
      for (int p = 0; p < PT; ++p)
        if (i < left) {
          vx[i][p] = __ldg(reinterpret_cast<const uint2*>(x[p] + k + 128 * i));
          vq[i][p] = __ldg(reinterpret_cast<const uint2*>(q[p] + k + 128 * i));
        }
#pragma unroll
    for (int i = 0; i < UNROLL; ++i)
#pragma unroll
      for (int p = 0; p < PT; ++p)
        if (i < left) add(p, vx[i][p], vq[i][p]);
    k += 128 * min(left, UNROLL);
  }
  if (k < d) {
#pragma unroll
    for (int p = 0; p < PT; ++p)
      add(p, __ldg(reinterpret_cast<const uint2*>(x[p] + k)), __ldg(reinterpret_cast<const uint2*>(q[p] + k)));
  }
#pragma unroll
  for (int p = 0; p < PT; ++p) {
    ss[p] = warp_sum(ss[p]);
    inv[p] = 0.f;
    if (ss[p] > FLT_MIN) { inv[p] = rsqrtf(ss[p]); inv[p] = inv[p] * (1.5f - 0.5f * ss[p] * inv[p] * inv[p]); }
    dot[p] = warp_sum(dot[p]) * inv[p];
  }
}

// A token left to identity_exact_kernel: a NaN that no score has (scores that are not finite are the positive one) with the
// row of its only candidate in the query array; or, in arrays of up to kPairRows rows, with the row of the first of two
// and the distance to the second.
constexpr uint32_t kDeferred = 0xffc00000u;
constexpr long long kDeferredRows = 1ll << 22;
constexpr int kPairBits = 14;
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
  float* exact = inv_q + kQueries;                         // [kTokens]
  uint16_t* candidates = reinterpret_cast<uint16_t*>(exact + kTokens);      // [kTokens][kQueries / 16]
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
    uint32_t deferred = 0u;                              // left to identity_exact_kernel
    uint32_t ph = 0;
    if (tokens) exact[r] = -FLT_MAX;
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
        named_barrier(1, 256);                           // the previous pass no longer reads inv_q and the candidates
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
          if (prm.defer && passes == 1 && at == 0 && r < T) prm.inv_q[txt_off + r] = inv;
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
        const bool tiny = inv_x == 0.f || !(most * inv_x <= 1.2e24f);
        if (!tiny) best = fmaxf(best, top);
        const float limit = tiny ? -INFINITY : best - prm.margin * len_x;
        int found = 0, low = 0, high = 0;                // candidates of the pass, the first and the last of them
#pragma unroll 1
        for (int c0 = 0; c0 < kQueries; c0 += 16) {
          uint32_t bits = 0u;
          if (c0 < cols) {
            float v[16];
            products16(t_lane + c0, v);
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (c0 + e < cols && v[e] * inv_q[c0 + e] >= limit) bits |= 1u << e;
          }
          if (nonfinite || !ok) bits = 0u;
          if (bits && found == 0) low = c0 + __ffs((int)bits) - 1;
          if (bits) high = c0 + 31 - __clz((int)bits);
          found += __popc(bits);
          candidates[r * (kQueries / 16) + (c0 >> 4)] = (uint16_t)bits;
        }
        if (passes == 1 && found >= 1 && found <= prm.defer)
          deferred = kDeferred | (uint32_t)(txt_off + low) | (uint32_t)(high - low) << kPairBits;
        if (deferred) reinterpret_cast<uint4*>(candidates)[r] = make_uint4(0u, 0u, 0u, 0u);
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acc_empty);
      }
      named_barrier(1, 256);                             // the candidates of the pass are known
      for (int t0 = warp; t0 < nrows; t0 += 16) {
        const int t[2] = {t0, min(t0 + 8, nrows - 1)};
        uint4 m[2];
        m[0] = reinterpret_cast<const uint4*>(candidates)[t[0]];
        m[1] = t0 + 8 < nrows ? reinterpret_cast<const uint4*>(candidates)[t[1]] : make_uint4(0u, 0u, 0u, 0u);
        float high[2] = {exact[t[0]], exact[t[1]]};
        for (;;) {
          const int j[2] = {next_candidate(m[0]), next_candidate(m[1])};
          if (j[0] < 0 && j[1] < 0) break;
          const __nv_bfloat16 *xr[2], *qr[2];
          float iq[2], inv[2], dot[2];
#pragma unroll
          for (int p = 0; p < 2; ++p) {                  // a token without one shares the other's loads
            const int tp = j[p] >= 0 ? t[p] : t[1 - p], jp = j[p] >= 0 ? j[p] : j[1 - p];
            xr[p] = prm.x + (size_t)(row0 + tp) * prm.d;
            qr[p] = prm.q + (size_t)(txt_off + pass * prm.n_cols + jp) * prm.d;
            iq[p] = inv_q[jp];
          }
          exact_cosines<2, 4>(xr, qr, iq, prm.d, lane, inv, dot);
#pragma unroll
          for (int p = 0; p < 2; ++p)
            if (j[p] >= 0) {
              high[p] = fmaxf(high[p], dot[p]);
              if (inv[p] == 0.f) m[p] = make_uint4(0u, 0u, 0u, 0u);        // a zero token: 0 with every element
            }
        }
        if (lane == 0) {
          exact[t[0]] = high[0];
          if (t0 + 8 < nrows) exact[t[1]] = high[1];
        }
      }
    }
    named_barrier(1, 256);
    // a wait that gave up leaves NaN, for callers that have no status word to look at
    if (tokens && r < nrows) {
      const uint32_t score = nonfinite || !ok ? 0x7fc00000u : deferred ? deferred : __float_as_uint(exact[r]);
      reinterpret_cast<uint32_t*>(prm.s_query)[row0 + r] = score;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem_base, kColumns);
  if (threadIdx.x == 0 && *abort_flag && prm.status != nullptr) atomicOr(prm.status, kStatusTimeout);
}

// The scores of the tokens that identity_tc_kernel left with one or two candidates; one warp per token, bound by the
// latency and issue of a row's loads and sums (32,768 tokens, d = 3584: about 45 us, 36 of them HBM).
__global__ void __launch_bounds__(256, 4)
identity_exact_kernel(const __nv_bfloat16* __restrict__ x, const __nv_bfloat16* __restrict__ q,
                      const float* __restrict__ inv_q, int d, int pairs, int first, int rows, float* __restrict__ s_query) {
  const int row = (int)(blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)), lane = threadIdx.x & 31;
  wait_for_previous_kernel();
  if (row >= rows) return;
  const uint32_t code = __float_as_uint(s_query[first + row]);
  if ((code & kDeferred) != kDeferred) return;
  const uint32_t low = code & (pairs ? (uint32_t)kPairRows - 1u : ~kDeferred);
  const uint32_t high = low + (pairs ? (code & ~kDeferred) >> kPairBits : 0u);
  const __nv_bfloat16* const xr[1] = {x + (size_t)(first + row) * d};
  float best = -FLT_MAX;
  bool nonfinite = false;
  for (uint32_t j = low;; j = high) {
    const __nv_bfloat16* const qr[1] = {q + (size_t)j * d};
    const float iq[1] = {inv_q[j]};
    float inv[1], dot[1];
    exact_cosines<1, 8>(xr, qr, iq, d, lane, inv, dot);
    best = fmaxf(best, dot[0]);
    nonfinite |= iq[0] != iq[0];
    if (j == high) break;
  }
  if (lane == 0) s_query[first + row] = nonfinite ? __int_as_float(0x7fc00000) : best;
}

}  // namespace ident
}  // namespace covspec
