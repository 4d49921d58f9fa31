// Tensor-core pieces of the low-rank redundancy step (Eq. 13-15): the Gram kernel of the stacked
// preselected tokens, and the shared-memory plan, triangular solve and float64 partial-Gram
// routines of the block power step (the step itself is part of the fused kernel in
// subspace_fused.cuh) with which the subspace iteration reaches the top-r eigenspace.
//
// G = Z_M^T Z_M (Eq. 13-14; its eigenpairs are sigma_k^2 and the right singular vectors of Z_M) is
// produced by tcgen05.mma kind::f16 from the gathered bf16 rows, accumulated in float32 in TMEM and
// stored as two bf16 planes G = G_hi + G_lo (16 mantissa bits), which is the operand format of the
// power step.  One power step computes, per 128-row tile of one request,
//     T      = G[tile, :] * Y                    3 MMAs per k-step: hi*hi + lo*hi + hi*lo
//     Y_next = T * L^-T                          forward substitution per row, L = chol(Y^T Y)
//     B_tile = Y_next[tile]^T Y_next[tile]       float64 partial Gram of the new block
// so that orthonormalising the previous block (Y L^-T) never needs its own pass over memory: the
// triangular factor is applied to the product instead (G (Y L^-T) = (G Y) L^-T).
//
// Layouts.  All requests share 2-D arrays so that one tensor map serves the whole batch:
//   G planes   [sum M_b (+pad), ld]  row presel_off(b) + i, column j          (ld = max M rounded to 64)
//   Y planes   [batch * 160, ld]     row b*160 + basis vector, column = token position (K-major B operand)
//   Yf         [sum M_b, 160]        float32 copy of the last block, one token per row
//   partial    [tiles, 13440]        8 x 8 tiles of the lower triangle in float64 (subspace_fused.cuh)
// Columns of G and Y between M_b and the next multiple of 64 are kept finite / zero respectively so
// that whole 64-wide k-chunks can be multiplied.
#pragma once
#include "tc_common.cuh"

namespace covspec {
namespace sub {

using namespace tc;

constexpr int kTile = 128;                 // rows per tile (UMMA M); Gram column tile (UMMA N)
constexpr int kBK = 64;                    // bf16 elements per k-chunk (one 128-byte swizzle row)
constexpr int kTriMax = kPMax * (kPMax + 1) / 2;          // 12880 packed lower-triangle entries
// Triangular factor as the power step reads it: row i holds L[j][i] for j = (i & ~3) .. P-1 so that
// 8-column blocks are two aligned float4 loads.  Largest size (P = 160) and the per-request stride
// (factor followed by the reciprocal diagonal).
constexpr int kLtFloats = kPMax * kPMax - 8 * (kPMax / 4) * (kPMax / 4 - 1);   // 13120
constexpr int kLbufStride = kLtFloats + kPMax;                                  // 13280

__host__ __device__ __forceinline__ int tri_index(int a, int b) { return a * (a + 1) / 2 + b; }
// Offset of row i of the padded upper-triangular layout for width P (a multiple of 4).
__host__ __device__ __forceinline__ int lt_row_offset(int i, int P) {
  int a = i >> 2, b = i & 3;
  return i * P - 8 * a * (a - 1) - 4 * a * b;
}

__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16& hi, __nv_bfloat16& lo) {
  hi = __float2bfloat16_rn(v);
  lo = __float2bfloat16_rn(v - __bfloat162float(hi));
}

// Row / column tile of the t-th lower-triangle tile (row-major over (ti, tj <= ti)).
__device__ __forceinline__ void tri_decode(int t, int& ti, int& tj) {
  ti = (int)((sqrtf(8.f * (float)t + 1.f) - 1.f) * 0.5f);
  while ((ti + 1) * (ti + 2) / 2 <= t) ++ti;
  while (ti * (ti + 1) / 2 > t) --ti;
  tj = t - ti * (ti + 1) / 2;
}

// ================================================================================================
// Gram kernel
// ================================================================================================
// Items are 128 x 256 blocks of the lower triangle (row tile ti, pair of column tiles 2 tjp and
// 2 tjp + 1, tjp <= ti / 2): per 64-element k-chunk a 16 KB row tile and a 32 KB column tile feed
// 128 x 256 x 64 products, two thirds of the operand bytes per product a square 128 x 128 item
// needs.  On the diagonal only what is needed is loaded and computed: with ti even the 128 x 128 block, with ti
// odd both blocks; where both operands are the same rows (bf16 inputs; float32 inputs have two forms of every
// row) the row tile is taken from the column tiles.
// The mirrored half of the matrix goes through shared memory, transposed, and out in rows of 256 bytes: as
// 2-byte stores straight from the registers it held up the next item (64 ragged requests of 100-1640 rows,
// d = 1536: 216 -> 189 us).
// A stage holds two 64-element chunks: half the barrier rounds of one chunk per stage.  (Polling a barrier costs
// the issuing threads 50-300 cycles while the tensor core reads shared memory; one row tile, d = 2048:
// 16.1 -> 15.6 us.)
constexpr int kGramStages = 2;
constexpr int kGramChunks = 2;
constexpr int kGramN = 2 * kTile;                         // columns of an item
constexpr int kGramBytesA = kTile * kBK * 2;              // 16 KB
constexpr int kGramChunkBytes = kGramBytesA + kGramN * kBK * 2;   // 48 KB
constexpr int kGramStageBytes = kGramChunks * kGramChunkBytes;
constexpr int kGramMirrorBytes = 2 * 32 * kTile * 2;      // 32 mirrored rows of 128 positions, hi and lo plane
constexpr int kGramSmem = kGramStages * kGramStageBytes + 2 * kGramMirrorBytes + 1024 + 1024;
constexpr int kGramTmemCols = 512;                        // two 256-column accumulators
// Items of a request with nt row tiles, and the decoding of an item index.
__host__ __device__ __forceinline__ int gram_items(int nt) {
  int a = nt >> 1;
  return (nt & 1) ? (a + 1) * (a + 1) : a * (a + 1);
}
__device__ __forceinline__ void gram_decode(int t, int& ti, int& tjp) {
  ti = 0;
  for (int cnt = 1; t >= cnt; cnt = (ti >> 1) + 1) { t -= cnt; ++ti; }
  tjp = t;
}

struct GramParams {
  const ReqPlan* plan;
  int batch;
  int n_items;          // lower-triangle tiles over all stage-2 requests
  int k_chunks;         // ceil(d / 64)
  __nv_bfloat16* g_hi;
  __nv_bfloat16* g_lo;
  int ld;
  int same;             // 1: the row and the column operand are the same rows
  int split;            // CTAs that share an item's columns (1, 2 or 4; more than 1: one item per CTA)
  int* status;
};
// A chunk is written to shared memory once and its operands are read once per product, 64 KB for one 128 x 128 item, 512
// cycles at 128 bytes a cycle: 508 measured (within the error of the clock), with two ring stages or six.  Where a call has few items, 2 or 4
// CTAs take the columns of one between them, each with the whole row tile: 64 and 48 KB per chunk instead of 96 for a
// 128 x 256 block (one float32 request 20.4 -> 16.0 us, one bf16 request 16.1 -> 11.7, 16 requests of 288 rows
// 24.2 -> 20.2).  Every element is still summed by one accumulator in the order of the inner dimension.

__global__ void __launch_bounds__(192, 1)
gram_tc_kernel(const __grid_constant__ CUtensorMap map_z,   // row operand [sum M_b, d] bf16, 128-row boxes
               const __grid_constant__ CUtensorMap map_zw,  // column operand, boxes of 256 / split rows
               const __grid_constant__ CUtensorMap map_zd,  // column operand, boxes of 128 / split rows
               const GramParams prm) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  uint8_t* mirror = smem + kGramStages * kGramStageBytes;       // [2][kGramMirrorBytes]
  uint64_t* bars = reinterpret_cast<uint64_t*>(mirror + 2 * kGramMirrorBytes);
  uint64_t* full = bars;                       // [kGramStages]
  uint64_t* empty = bars + kGramStages;        // [kGramStages]
  uint64_t* acc_full = bars + 2 * kGramStages; // [2]
  uint64_t* acc_empty = acc_full + 2;          // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 4);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  const int warp = warp_index(), lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kGramStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 128); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 5) tmem_alloc(tmem_slot, kGramTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  wait_for_previous_kernel();

  const int first_item = blockIdx.x / prm.split, stride = gridDim.x / prm.split, sub = blockIdx.x % prm.split;
  const int same = prm.split == 1 ? prm.same : 0;          // part of the columns holds no whole row tile
  auto decode = [&](int item, ReqPlan& rp, int& ti, int& tjp) {
    int b = find_request(item, prm.batch, [&](int q) { return prm.plan[q].gram_tile_off; });
    rp = prm.plan[b];
    gram_decode(item - rp.gram_tile_off, ti, tjp);
  };

  if (warp == 4) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int item = first_item; item < prm.n_items && ok; item += stride) {
        ReqPlan rp; int ti, tj;
        decode(item, rp, ti, tj);
        // a chunk: row tile, then the pair of column tiles (its first one only where ti = 2 tj)
        const bool first = ti == 2 * tj, load_a = !same || !(first || ti == 2 * tj + 1);
        const int width = (first ? kTile : kGramN) / prm.split, col_row = rp.presel_off + tj * kGramN + sub * width;
        const int bytes = (load_a ? kGramBytesA : 0) + width * kBK * 2;
        for (int kc = 0; kc < prm.k_chunks; kc += kGramChunks, ++it) {
          const int s = it % kGramStages, chunks = min(kGramChunks, prm.k_chunks - kc);
          if (!(ok = mbar_wait(&empty[s], ((it / kGramStages) & 1u) ^ 1u, abort_flag))) break;
          mbar_expect_tx(&full[s], chunks * bytes);
          uint32_t dst = smem_u32(smem + s * kGramStageBytes);
          for (int c = 0; c < chunks; ++c, dst += kGramChunkBytes) {
            if (load_a) tma_load_2d(dst, &map_z, (kc + c) * kBK, rp.presel_off + ti * kTile, &full[s]);
            tma_load_2d(dst + kGramBytesA, first ? &map_zd : &map_zw, (kc + c) * kBK, col_row, &full[s]);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 5) {
    if (lane == 0) {
      uint32_t it = 0, n = 0;
      bool ok = true;
      for (int item = first_item; item < prm.n_items && ok; item += stride, ++n) {
        ReqPlan rp; int ti, tj;
        decode(item, rp, ti, tj);
        const uint32_t idesc = umma_idesc(kTile, (ti == 2 * tj ? kTile : kGramN) / prm.split);
        // where the row tile lies (see the producer)
        const int a_off = !same ? 0 : ti == 2 * tj ? kGramBytesA : ti == 2 * tj + 1 ? 2 * kGramBytesA : 0;
        int buf = n & 1;
        if (!(ok = mbar_wait(&acc_empty[buf], ((n >> 1) & 1u) ^ 1u, abort_flag))) break;
        tc_fence_after();
        for (int kc = 0; kc < prm.k_chunks; kc += kGramChunks, ++it) {
          const int s = it % kGramStages, chunks = min(kGramChunks, prm.k_chunks - kc);
          if (!(ok = mbar_wait(&full[s], (it / kGramStages) & 1u, abort_flag))) break;
          tc_fence_after();
          uint32_t base = smem_u32(smem + s * kGramStageBytes);
#pragma unroll
          for (int c = 0; c < kGramChunks; ++c, base += kGramChunkBytes) {
            if (c >= chunks) break;
            const uint64_t adesc = umma_desc(base + a_off), bdesc = umma_desc(base + kGramBytesA);
#pragma unroll
            for (int k = 0; k < kBK / 16; ++k)
              umma_bf16(tmem_base + buf * kGramN, adesc + 2 * k, bdesc + 2 * k, idesc, (kc | c | k) != 0);
          }
          umma_commit(&empty[s]);
        }
        if (!ok) break;
        umma_commit(&acc_full[buf]);
      }
    }
    __syncwarp();
  } else {
    const int r = warp * 32 + lane;
    const uint32_t t_lane = tmem_base + ((uint32_t)(warp * 32) << 16);
    uint32_t n = 0, rounds = 0;
    bool ok = true;
    for (int item = first_item; item < prm.n_items; item += stride, ++n) {
      ReqPlan rp; int ti, tj;
      decode(item, rp, ti, tj);
      int buf = n & 1;
      ok = ok && mbar_wait(&acc_full[buf], (n >> 1) & 1u, abort_flag);      // a thread that gave up stays for the barriers
      tc_fence_after();
      const int row = ti * kTile + r;                 // row of G inside the request
      const bool row_ok = row < rp.m;
      const size_t ld = (size_t)prm.ld;
      const int groups = (ti == 2 * tj ? kTile : kGramN) / 32 / prm.split, first_group = sub * groups;
#pragma unroll 1
      for (int c4 = first_group; c4 < first_group + groups; ++c4) {
        const int tc = 2 * tj + (c4 >> 2);            // column tile of this group of 32 columns
        float v[32];
        tmem_ld32(t_lane + buf * kGramN + (c4 - first_group) * 32, v);
        const int col0 = tj * kGramN + c4 * 32;
        // entries outside the request's M x M block are stored as zeros: the power step multiplies
        // whole 64-wide k-chunks and must not meet stale non-finite values in the padding
#pragma unroll
        for (int e = 0; e < 32; ++e)
          if (col0 + e >= rp.m || !row_ok) v[e] = 0.f;
        uint32_t ph[16], pl[16];
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          __nv_bfloat162 hi = __floats2bfloat162_rn(v[2 * e], v[2 * e + 1]);
          ph[e] = *reinterpret_cast<uint32_t*>(&hi);
          pl[e] = pack_bf16(v[2 * e] - __low2float(hi), v[2 * e + 1] - __high2float(hi));
        }
        if (ok && row_ok && col0 < prm.ld) {
          size_t o = ((size_t)rp.presel_off + row) * ld + col0;
          uint4* dh = reinterpret_cast<uint4*>(prm.g_hi + o);
          uint4* dl = reinterpret_cast<uint4*>(prm.g_lo + o);
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            dh[q] = make_uint4(ph[4 * q], ph[4 * q + 1], ph[4 * q + 2], ph[4 * q + 3]);
            dl[q] = make_uint4(pl[4 * q], pl[4 * q + 1], pl[4 * q + 2], pl[4 * q + 3]);
          }
        }
        if (ti != tc) {
          // mirrored tile: G[col, row] = G[row, col], 32 rows of it per round; two staging buffers, so that
          // one barrier per round separates the rounds
          unsigned short* st = reinterpret_cast<unsigned short*>(mirror + (rounds & 1u) * kGramMirrorBytes);
          ++rounds;
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const uint32_t wh = ph[e >> 1], wl = pl[e >> 1];
            st[e * kTile + r] = (unsigned short)((e & 1) ? (wh >> 16) : (wh & 0xffffu));
            st[(32 + e) * kTile + r] = (unsigned short)((e & 1) ? (wl >> 16) : (wl & 0xffffu));
          }
          named_barrier(1, 128);
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const int idx = q * 128 + r, e = (idx >> 4) & 31, v = idx & 15;      // plane q / 4, row e, 16-byte vector v
            const int mrow = col0 + e, pos = ti * kTile + v * 8;
            if (ok && mrow < rp.m && pos < prm.ld) {
              const uint4 val = *reinterpret_cast<const uint4*>(st + (size_t)(q >> 2) * 32 * kTile + e * kTile + v * 8);
              __nv_bfloat16* plane = q < 4 ? prm.g_hi : prm.g_lo;
              *reinterpret_cast<uint4*>(plane + ((size_t)rp.presel_off + mrow) * ld + pos) = val;
            }
          }
        }
      }
      tc_fence_before();
      mbar_arrive(&acc_empty[buf]);
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 5) tmem_dealloc(tmem_base, kGramTmemCols);
  if (threadIdx.x == 0 && *abort_flag) atomicOr(prm.status, kStatusTimeout);
}

// Splits a float32 Gram matrix (CUDA-core path, float32 inputs) into the two bf16 planes.
__global__ void __launch_bounds__(256)
split_planes_kernel(const ReqPlan* __restrict__ plan, const float* __restrict__ G,
                    __nv_bfloat16* __restrict__ g_hi, __nv_bfloat16* __restrict__ g_lo, int ld) {
  ReqPlan rp = plan[blockIdx.y];
  if (!rp.stage2) return;
  int cols = (rp.m + 63) & ~63;
  int total = rp.m * cols;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    int i = e / cols, j = e % cols;
    float v = j < rp.m ? G[rp.g_off + (size_t)i * rp.ldm + j] : 0.f;
    __nv_bfloat16 hi, lo;
    split_bf16(v, hi, lo);
    size_t o = ((size_t)rp.presel_off + i) * ld + j;
    g_hi[o] = hi; g_lo[o] = lo;
  }
}

// Start block of the subspace iteration: entries uniform in [-1, 1) from a counter hash of
// (request, basis vector, position); zero in the padding columns and in the unused basis rows
// p .. round_up(p, 16) - 1 of both plane buffers (the MMA reads them, nothing else writes them).
// The same launch resets the per-request words of the fused subspace kernel (three counters and the
// index of the last step per request, then the abort word) and writes zero energies for the requests that skip stage 2.
__global__ void __launch_bounds__(256)
basis_init_kernel(const ReqPlan* __restrict__ plan, __nv_bfloat16* __restrict__ y_hi,
                  __nv_bfloat16* __restrict__ y_lo, __nv_bfloat16* __restrict__ y2_hi,
                  __nv_bfloat16* __restrict__ y2_lo, int ld, float* __restrict__ energy,
                  unsigned* __restrict__ sync, int batch, int last_step) {
  ReqPlan rp = plan[blockIdx.y];
  if (blockIdx.x == 0) {
    if (threadIdx.x < 8) sync[blockIdx.y * 8 + threadIdx.x] = threadIdx.x == 3 ? (unsigned)last_step : 0u;
    if (blockIdx.y == 0 && threadIdx.x >= 32 && threadIdx.x < 36) sync[batch * 8 + threadIdx.x - 32] = 0u;
    if (!rp.stage2)
      for (int i = threadIdx.x; i < rp.m; i += blockDim.x) energy[rp.presel_off + i] = 0.f;
  }
  if (!rp.stage2) return;
  int cols = (rp.m + 63) & ~63;
  int rows = (rp.p + 15) & ~15;
  int total = rows * cols;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < total; e += gridDim.x * blockDim.x) {
    int j = e / cols, i = e % cols;
    float v = 0.f;
    if (j < rp.p && i < rp.m) {
      unsigned h = (unsigned)(j * rp.m + i) * 0x9E3779B1u ^ ((unsigned)blockIdx.y + 1u) * 0x85EBCA77u;
      h ^= h >> 16; h *= 0x7FEB352Du; h ^= h >> 15; h *= 0x846CA68Bu; h ^= h >> 16;
      v = (float)(h >> 8) * (2.0f / 16777216.0f) - 1.0f;
    }
    __nv_bfloat16 hi, lo;
    split_bf16(v, hi, lo);
    size_t o = ((size_t)blockIdx.y * kPMax + j) * ld + i;
    y_hi[o] = hi; y_lo[o] = lo;
    if (j >= rp.p) { y2_hi[o] = hi; y2_lo[o] = lo; }
  }
}

// ================================================================================================
// Power step: shared-memory plan and epilogue routines
// ================================================================================================
constexpr int kPowStages = 2;
constexpr int kPowBytesA = kTile * kBK * 2;              // one plane of the G tile, 16 KB
constexpr int kPowBytesB = kPMax * kBK * 2;              // one plane of the Y tile, 20 KB
constexpr int kPowStageBytes = 2 * kPowBytesA + 2 * kPowBytesB;   // 72 KB
constexpr int kXsLd = kTile + 4;                         // row stride of the staged block (floats)
constexpr int kXsBytes = (kPMax * kXsLd * 4 + 1023) / 1024 * 1024;   // one staged block [kPMax][kXsLd] of float32
// The ring is followed by padding up to two staged blocks: after the MMAs the region holds the new
// block, and either the previous block (last step) or the float64 slabs of the Gram accumulation.
constexpr int kPowRegion = 2 * kXsBytes > kPowStages * kPowStageBytes ? 2 * kXsBytes : kPowStages * kPowStageBytes;
constexpr int kPowSmem = kPowRegion + kLbufStride * 4 + 1024 + 1024;
constexpr int kPowTmemCols = 256;
constexpr int kPowThreads = 320;                         // 8 epilogue warps, TMA producer, MMA issuer
static_assert(kPMax * kXsLd * 4 <= kPowStages * kPowStageBytes, "staged block must fit in the ring");

// Base of the kernel's dynamic shared memory, rounded up to 1024 bytes by an offset (not by integer
// arithmetic on the address), and taken from the array itself in every function that is not inlined: so
// the compiler knows that what it reaches through the result is shared memory.
__device__ __forceinline__ uint8_t* pow_smem() {
  extern __shared__ uint8_t smem_raw[];
  return smem_raw + ((0u - smem_u32(smem_raw)) & 1023u);
}
// ---- T L^-T by super-blocks of 32 columns (x[c * kXsLd + row] holds T and becomes the result) ------
// solve_gemm takes the contributions of the columns before super-block S off its 32 columns: a product
// of (rows) x (32 S) with (32 S) x 32, by the eight warps, RT rows x 4 columns per thread.  A warp
// covers 16 RT rows x 8 columns, so that a column step reads 16 RT + 8 words of shared memory for
// 128 RT products: sixteen multiply-adds per thread when RT = 4, as many cycles as the two loads take.
// Neighbouring lanes share a row group and take different columns: a 16-byte load takes two cycles where neighbours
// read the same address and four where the two halves of the warp read the same addresses (measured), which made
// the first form of this mapping (lane & 15) bound by shared memory.
// solve_diag then solves inside the super-block, one thread per row, the row's 32 values in
// registers.  p = 144, 128 rows: 40 -> 14 k cycles.
// The products enter every sum in ascending column order; `split` (steps before the last one): the
// columns before 32 (S - 1) are summed from zero and T is added to that sum.
template <int RT, int RG>
__device__ __forceinline__ void solve_gemm(float* x, const float* lt, int P, int S, bool split, int nrows, int warp,
                                           int lane) {
  const int rg = warp % RG, row0 = 16 * RT * rg + RT * (lane >> 1);
  const int j0 = 32 * S + 8 * (warp / RG);
  if (16 * RT * rg >= ((nrows + 31) & ~31) || j0 >= P) return;       // whole warp
  const int j = j0 + 4 * (lane & 1);
  float acc[4][RT];
  auto t_at = [&](int c) { return x + (j + c) * kXsLd + row0; };
  auto rows_load = [&](const float* src, float (&v)[RT]) {
    if constexpr (RT == 4) {
      float4 t = *reinterpret_cast<const float4*>(src);
      v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
    } else if constexpr (RT == 2) {
      float2 t = *reinterpret_cast<const float2*>(src);
      v[0] = t.x; v[1] = t.y;
    } else {
      v[0] = *src;
    }
  };
  const float* xp = x + row0;
  const float* lp = lt + j;                // row i of the layout starts at column i & ~3
  int stride = P;                          // rows 4a .. 4a+3 have P - 4a entries
  float xv[2][4][RT];
  float4 lv[2][4];
  auto load = [&](int buf) {               // one group of four columns, then step to the next
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      rows_load(xp + q * kXsLd, xv[buf][q]);
      lv[buf][q] = *reinterpret_cast<const float4*>(lp + q * stride);
    }
    xp += 4 * kXsLd;
    lp += 4 * stride - 4;
    stride -= 4;
  };
  auto apply = [&](int buf) {
#pragma unroll
    for (int q = 0; q < 4; ++q)
#pragma unroll
      for (int e = 0; e < RT; ++e) {
        acc[0][e] -= xv[buf][q][e] * lv[buf][q].x; acc[1][e] -= xv[buf][q][e] * lv[buf][q].y;
        acc[2][e] -= xv[buf][q][e] * lv[buf][q].z; acc[3][e] -= xv[buf][q][e] * lv[buf][q].w;
      }
  };
  // `count` (even) groups; the loads of a group are in flight while the one before is applied.  The
  // group loaded beyond the last one is dropped (its addresses lie inside the staged block and the factor).
  auto groups = [&](int count) {
#pragma unroll 1
    for (int g = 0; g < count; g += 2) {
      load(1);
      apply(0);
      load(0);
      apply(1);
    }
  };
  load(0);
  if (split && S >= 2) {
#pragma unroll
    for (int c = 0; c < 4; ++c)
#pragma unroll
      for (int e = 0; e < RT; ++e) acc[c][e] = 0.f;
    groups(8 * (S - 1));
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      float t[RT];
      rows_load(t_at(c), t);
#pragma unroll
      for (int e = 0; e < RT; ++e) acc[c][e] = t[e] + acc[c][e];
    }
    groups(8);
  } else {
#pragma unroll
    for (int c = 0; c < 4; ++c) rows_load(t_at(c), acc[c]);
    groups(8 * S);
  }
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    if constexpr (RT == 4) *reinterpret_cast<float4*>(t_at(c)) = make_float4(acc[c][0], acc[c][1], acc[c][2], acc[c][3]);
    else if constexpr (RT == 2) *reinterpret_cast<float2*>(t_at(c)) = make_float2(acc[c][0], acc[c][1]);
    else *t_at(c) = acc[c][0];
  }
}
// RT and the split of the eight warps over row groups (RG) and columns: all 32 columns, or at most 16 of them in the
// last super-block (the column groups would otherwise leave half the warps without work).
__device__ __forceinline__ void solve_gemm_any(int tile_rows, float* x, const float* lt, int P, int S, bool split,
                                               int nrows, int warp, int lane) {
  const bool narrow = P - 32 * S <= 16;
  if (tile_rows == kTile) {
    if (narrow) solve_gemm<2, 4>(x, lt, P, S, split, nrows, warp, lane);
    else solve_gemm<4, 2>(x, lt, P, S, split, nrows, warp, lane);
  } else {
    if (narrow) solve_gemm<1, 4>(x, lt, P, S, split, nrows, warp, lane);
    else solve_gemm<2, 2>(x, lt, P, S, split, nrows, warp, lane);
  }
}
// NG: groups of eight columns in the super-block (four but for the last one of a width that is not a multiple of 32).
// One warp per scheduler and a chain from column to column: a column's factor row is loaded while the column before it is
// applied, and two columns are updated by one packed multiply-add.
template <int NG>
__device__ __forceinline__ void solve_diag_n(float* xr, const float* lt, const float* dinv, int P, int S, bool keep) {
  constexpr int W = 8 * NG;
  float acc[W];
  float* xb = xr + 32 * S * kXsLd;
  const int a0 = 8 * S;
  const float* lp = lt + 4 * a0 * P - 8 * a0 * (a0 - 1);      // row 32 S of the layout, at its first column 32 S
  const int stride = P - 32 * S;
  // row i of the factor from the group of four columns that holds i on: P - 32 S - 4 (i / 4) entries a row
  auto row_at = [&](int i) { const int a = i >> 2; return lp + 4 * a * stride - 8 * a * (a - 1) + (i & 3) * (stride - 4 * a); };
  float4 l[2][2 * NG];
  auto load_row = [&](int i, float4 (&dst)[2 * NG]) {
#pragma unroll
    for (int v = 0; v < 2 * NG; ++v)
      if (4 * v + 3 > i) dst[v] = *reinterpret_cast<const float4*>(row_at(i) + 4 * (v - (i >> 2)));
  };
#pragma unroll
  for (int e = 0; e < W; ++e) acc[e] = xb[e * kXsLd];
  float4 d4 = *reinterpret_cast<const float4*>(dinv + 32 * S);
  load_row(0, l[0]);
#pragma unroll
  for (int i = 0; i < W; ++i) {
    const float dv = (i & 3) == 0 ? d4.x : (i & 3) == 1 ? d4.y : (i & 3) == 2 ? d4.z : d4.w;
    const float xi = acc[i] * dv;
    acc[i] = xi;
    if (i + 1 < W) {
      if ((i & 3) == 3) d4 = *reinterpret_cast<const float4*>(dinv + 32 * S + i + 1);
      load_row(i + 1, l[(i + 1) & 1]);
    }
    const f32x2 nx = pack2(-xi, -xi);
#pragma unroll
    for (int v = 0; v < 2 * NG; ++v) {
      if (4 * v + 3 <= i) continue;
      const float lv[4] = {l[i & 1][v].x, l[i & 1][v].y, l[i & 1][v].z, l[i & 1][v].w};
#pragma unroll
      for (int e = 0; e < 4; e += 2) {
        const int j = 4 * v + e;
        if (j > i) {
          const float2 t = unpack2(fma2(nx, pack2(lv[e], lv[e + 1]), pack2(acc[j], acc[j + 1])));
          acc[j] = t.x; acc[j + 1] = t.y;
        } else if (j + 1 > i) {
          acc[j + 1] = fmaf(-xi, lv[e + 1], acc[j + 1]);
        }
      }
    }
  }
#pragma unroll
  for (int e = 0; e < W; ++e) xb[e * kXsLd] = keep ? acc[e] : 0.f;
}
__device__ __forceinline__ void solve_diag(float* xr, const float* lt, const float* dinv, int P, int S, bool keep) {
  const int ng = (P - 32 * S) >> 3;
  if (ng >= 4) solve_diag_n<4>(xr, lt, dinv, P, S, keep);
  else if (ng == 3) solve_diag_n<3>(xr, lt, dinv, P, S, keep);
  else if (ng == 2) solve_diag_n<2>(xr, lt, dinv, P, S, keep);
  else solve_diag_n<1>(xr, lt, dinv, P, S, keep);
}

// The whole solve of a staged block that starts x_off floats behind the base of shared memory, by the eight
// epilogue warps; rows nrows and beyond (and all rows when keep_rows is false) come out as zeros.  Out of
// line: see the rehearsal in subspace_kernel.
__device__ __noinline__ void solve_team(int x_off, int P, int tile_rows, bool split, int nrows, bool keep_rows) {
  float* x = reinterpret_cast<float*>(pow_smem()) + x_off;
  const float* lt = reinterpret_cast<float*>(pow_smem() + kPowRegion);
  const float* dinv = lt + kLtFloats;
  const int et = threadIdx.x, warp = warp_index(), lane = et & 31, nS = (P + 31) >> 5;
#pragma unroll 1
  for (int S = 0; S < nS; ++S) {
    if (S > 0) {
      solve_gemm_any(tile_rows, x, lt, P, S, split, nrows, warp, lane);
      named_barrier(1, 256);
    }
    if (warp < 4 && warp * 32 < nrows) solve_diag(x + et, lt, dinv, P, S, keep_rows && et < nrows);
    named_barrier(1, 256);
  }
}

// C (8x8 float64, two entries per thread) += A (8x4) * B (4x8): one tensor-core instruction.
__device__ __forceinline__ void dmma_8x8x4(double& c0, double& c1, double a, double b) {
  asm volatile("mma.sync.aligned.m8n8k4.row.col.f64.f64.f64.f64 {%0,%1}, {%2}, {%3}, {%0,%1};"
               : "+d"(c0), "+d"(c1)
               : "d"(a), "d"(b));
}

constexpr int kSlabRows = 16;            // the float64 Gram of a block takes its rows in groups of this many

}  // namespace sub
}  // namespace covspec
