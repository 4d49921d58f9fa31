// Segmented top-k selection (preselect the M best fused scores; keep the B_vis largest energies)
// and the row gather used for Z_M (Eq. 13) and for the compacted output.
#pragma once
#include "common.cuh"
#include "score_kernels.cuh"

namespace covspec {

// Monotone map float -> uint32 (larger float = larger key).  -0 is folded onto +0 so that equal
// values share a key; NaN maps to the smallest key.
__device__ __forceinline__ unsigned order_key(float v) {
  if (v != v) return 0u;
  v += 0.0f;
  unsigned u = __float_as_uint(v);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// Block-wide exclusive scan of a small packed counter (blockDim.x multiple of 32, <= 1024).
// Returns the exclusive prefix; *total receives the block sum.
__device__ __forceinline__ unsigned block_exclusive_scan(unsigned v, unsigned* warp_tot,
                                                         unsigned* total) {
  int lane = threadIdx.x & 31, w = warp_index(), nw = blockDim.x >> 5;
  unsigned inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  __syncthreads();
  if (lane == 31) warp_tot[w] = inc;
  __syncthreads();
  if (w == 0) {
    unsigned t = lane < nw ? warp_tot[lane] : 0u, ti = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned u = __shfl_up_sync(0xffffffffu, ti, o);
      if (lane >= o) ti += u;
    }
    if (lane < nw) warp_tot[lane] = ti - t;   // exclusive warp offsets
    if (lane == 31) warp_tot[32] = ti;        // block total
  }
  __syncthreads();
  *total = warp_tot[32];
  return warp_tot[w] + inc - v;
}

// Top-k of n keys: larger key first, then lower index; out[0..k) receives the selected positions in ascending
// order, mapped through `remap` when given.  Two forms:
//   up to kRegKeys keys per thread: the keys stay in registers (thread t holds the positions t,
//   t + blockDim, ...) and the k-th largest key is found two bits at a time, one block-wide count per pair of bits
//   below the prefix that all keys share, ending as soon as a count equals k (about 8 counts of 150-300 cycles for
//   scores).  A radix select through shared-memory histograms took 12 us at 768 keys (scores
//   crowd into a few digit values, whose updates queue up) and ranking every key 18 us.
//   longer segments: an 8-bit-per-pass radix select that re-reads its keys, then an ordered emission.
constexpr int kRegKeys = 16;           // keys per thread the select keeps in registers

// One value per thread -> its block-wide reduction, one barrier.  `slots`: two rows used in turn.
struct CountSlots { unsigned v[2][32]; };

template <int PER>
__device__ __forceinline__ void block_select_regs(const unsigned (&key)[PER], int n, int k, const int* __restrict__ remap,
                                                  int* __restrict__ out, int* status) {
  __shared__ CountSlots slots, slots2;
  __shared__ unsigned counts[PER * 32];
  __shared__ unsigned s_total;
  const int lane = threadIdx.x & 31, warp = warp_index(), nw = blockDim.x >> 5, nt = blockDim.x, tid = threadIdx.x;
  unsigned all_and = 0xffffffffu, all_or = 0u;
#pragma unroll
  for (int j = 0; j < PER; ++j)
    if (tid + j * nt < n) { all_and &= key[j]; all_or |= key[j]; }
  all_and = __reduce_and_sync(0xffffffffu, all_and);
  all_or = __reduce_or_sync(0xffffffffu, all_or);
  if (lane == 0) { slots.v[0][warp] = all_and; slots2.v[0][warp] = all_or; }
  __syncthreads();
  all_and = __reduce_and_sync(0xffffffffu, lane < nw ? slots.v[0][lane] : 0xffffffffu);
  all_or = __reduce_or_sync(0xffffffffu, lane < nw ? slots2.v[0][lane] : 0u);
  const unsigned diff = all_and ^ all_or;
  const int top = 31 - __clz((int)diff);                     // -1: all keys are equal
  unsigned thr = all_and & ~((2u << top) - 1u);              // shared prefix (top = 31: nothing)
  if (top < 0) thr = all_and;
  bool exact = false;                                        // keys >= thr are the answer, no ties
  int buf = 1;
  for (int bit = top; bit >= 0 && !exact; bit -= 2, buf ^= 1) {
    // two bits per round: the largest of three candidates that at least k keys reach (the last round of an odd number of
    // bits has one)
    const int low = max(bit - 1, 0);
    const unsigned step = 1u << low;
    unsigned c12 = 0u, c3 = 0u;                              // keys >= thr + step, >= thr + 2 step (upper half), >= thr + 3 step
#pragma unroll
    for (int j = 0; j < PER; ++j) {                          // positions beyond n hold key 0 < thr + step
      c12 += (key[j] >= thr + step ? 1u : 0u) + (bit > 0 && key[j] >= thr + 2u * step ? 1u << 16 : 0u);
      c3 += bit > 0 && key[j] >= thr + 3u * step;
    }
    c12 = __reduce_add_sync(0xffffffffu, c12);
    c3 = __reduce_add_sync(0xffffffffu, c3);
    if (lane == 0) { slots.v[buf][warp] = c12; slots2.v[buf][warp] = c3; }
    __syncthreads();
    c12 = __reduce_add_sync(0xffffffffu, lane < nw ? slots.v[buf][lane] : 0u);
    c3 = __reduce_add_sync(0xffffffffu, lane < nw ? slots2.v[buf][lane] : 0u);
    const unsigned c1 = c12 & 0xffffu, c2 = c12 >> 16;
    const unsigned take = c3 >= (unsigned)k ? 3u : c2 >= (unsigned)k ? 2u : c1 >= (unsigned)k ? 1u : 0u;
    if (take) { thr += take * step; exact = (take == 3u ? c3 : take == 2u ? c2 : c1) == (unsigned)k; }
  }
  // ordered emission: counts per (j, warp), which is position order, then one scan
  unsigned mg[PER], me[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const bool in = tid + j * nt < n;
    mg[j] = __ballot_sync(0xffffffffu, in && (exact ? key[j] >= thr : key[j] > thr));
    me[j] = __ballot_sync(0xffffffffu, in && !exact && key[j] == thr);
    if (lane == 0) counts[j * nw + warp] = (unsigned)__popc(mg[j]) | (unsigned)__popc(me[j]) << 16;
  }
  __syncthreads();
  if (warp == 0) {
    unsigned v[PER], sum = 0u;                               // PER consecutive entries per lane (nw <= 32)
#pragma unroll
    for (int j = 0; j < PER; ++j) {
      v[j] = sum;
      if (lane * PER + j < PER * nw) sum += counts[lane * PER + j];
    }
    unsigned inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      unsigned t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
#pragma unroll
    for (int j = 0; j < PER; ++j)
      if (lane * PER + j < PER * nw) counts[lane * PER + j] = inc - sum + v[j];
    if (lane == 31) s_total = inc;
  }
  __syncthreads();
  const unsigned kk = (unsigned)k - (s_total & 0xffffu);     // how many keys equal to the threshold are taken
  const unsigned below = (1u << lane) - 1u;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const bool g = mg[j] >> lane & 1u, e = me[j] >> lane & 1u;
    if (!g && !e) continue;
    const unsigned before = counts[j * nw + warp];
    const unsigned gt_before = (before & 0xffffu) + __popc(mg[j] & below), eq_before = (before >> 16) + __popc(me[j] & below);
    const unsigned pos = gt_before + min(eq_before, kk);
    if ((g || eq_before < kk) && COVSPEC_IN_BOUNDS(pos, k, status)) {
      const int i = tid + j * nt;
      out[pos] = remap ? remap[i] : i;
    }
  }
}

// One digit of the radix select, by the first warp: with `kk` keys still to take among those that
// match the digits fixed so far, the largest digit value d such that the keys with a larger digit
// number fewer than kk (digit 0 when none does); *sel_k = kk minus those keys.  Lane l sums the
// eight histogram bins 8 l .. 8 l + 7; a suffix scan over the lanes finds the lane that holds d.
__device__ __forceinline__ void select_digit(const unsigned* hist, unsigned kk, unsigned prefix, int shift,
                                             unsigned* sel_prefix, unsigned* sel_k) {
  const int lane = threadIdx.x & 31;
  if (kk == 0u) {                             // nothing left to take: no key is above the top digit
    if (lane == 0) { *sel_prefix = prefix | (255u << shift); *sel_k = 0u; }
    return;
  }
  unsigned h[8], mine = 0u;
#pragma unroll
  for (int e = 0; e < 8; ++e) { h[e] = hist[8 * lane + e]; mine += h[e]; }
  unsigned above = mine;                      // inclusive suffix sum over lanes >= this one
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    unsigned t = __shfl_down_sync(0xffffffffu, above, o);
    if (lane + o < 32) above += t;
  }
  above -= mine;                              // keys in the bins of higher lanes
  const unsigned holds = __ballot_sync(0xffffffffu, above < kk && above + mine >= kk);
  const int owner = holds ? 31 - __clz(holds) : 0;
  if (lane == owner) {
    unsigned c = above;
    int e = 7;
    for (; e > 0; --e) {
      if (c + h[e] >= kk) break;
      c += h[e];
    }
    if (!holds) {                             // fewer matching keys than kk: digit 0 takes the rest
      e = 0;
      c = above + mine - h[0];
    }
    *sel_prefix = prefix | ((unsigned)(8 * lane + e) << shift);
    *sel_k = kk - c;
  }
}

// The select on up to PER keys per thread; `load(i)` returns key i as a float.
template <int PER, typename LoadF>
__device__ __forceinline__ void block_topk_regs(LoadF load, int n, int k, bool all_equal, const int* __restrict__ remap,
                                                int* __restrict__ out, int* status) {
  unsigned key[PER];
  bool bad = false;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = (int)threadIdx.x + j * (int)blockDim.x;
    key[j] = 0u;
    if (i < n && !all_equal) {
      const float v = load(i);
      bad |= !(fabsf(v) <= 3.402823466e38f);
      key[j] = order_key(v);
    }
  }
  if (bad && status != nullptr) atomicOr(status, kStatusNonFinite);
  block_select_regs<PER>(key, n, k, remap, out, status);
}

// `load(i)` returns key i as a float; `status` may be nullptr (non-finite keys are then not reported).
// `all_equal` treats every key as equal (selects the first k positions).
template <typename LoadF>
__device__ void block_topk_by(LoadF load, int n, int k, bool all_equal,
                              const int* __restrict__ remap, int* __restrict__ out, int* status) {
  const int per = (n + (int)blockDim.x - 1) / (int)blockDim.x;
  if (per <= 1) { block_topk_regs<1>(load, n, k, all_equal, remap, out, status); return; }
  if (per <= 4) { block_topk_regs<4>(load, n, k, all_equal, remap, out, status); return; }
  if (per <= kRegKeys) { block_topk_regs<kRegKeys>(load, n, k, all_equal, remap, out, status); return; }
  __shared__ unsigned hist[256];
  __shared__ unsigned sel_prefix, sel_k;
  __shared__ unsigned warp_tot[33];
  unsigned prefix = 0u, mask = 0u, kk = (unsigned)k;
  if (!all_equal) {
    bool bad = false;
    for (int shift = 24; shift >= 0; shift -= 8) {
      for (int i = threadIdx.x; i < 256; i += blockDim.x) hist[i] = 0u;
      __syncthreads();
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        float v = load(i);
        if (shift == 24) bad |= !(fabsf(v) <= 3.402823466e38f);
        unsigned key = order_key(v);
        if ((key & mask) == prefix) atomicAdd(&hist[(key >> shift) & 255u], 1u);
      }
      __syncthreads();
      if (warp_index() == 0) select_digit(hist, kk, prefix, shift, &sel_prefix, &sel_k);
      __syncthreads();
      prefix = sel_prefix;
      kk = sel_k;
      mask |= 255u << shift;
    }
    if (bad && status != nullptr) atomicOr(status, kStatusNonFinite);
  }
  // Ordered emission.  kk = how many elements equal to the threshold are taken.
  unsigned run_gt = 0u, run_eq = 0u;
  for (int base = 0; base < n; base += blockDim.x) {
    int i = base + threadIdx.x;
    unsigned gt = 0u, eq = 0u;
    if (i < n) {
      if (all_equal) eq = 1u;
      else {
        unsigned key = order_key(load(i));
        gt = key > prefix; eq = key == prefix;
      }
    }
    unsigned tot;
    unsigned ex = block_exclusive_scan(gt | (eq << 16), warp_tot, &tot);
    unsigned gt_before = run_gt + (ex & 0xffffu), eq_before = run_eq + (ex >> 16);
    if (gt || (eq && eq_before < kk)) {
      unsigned pos = gt_before + min(eq_before, kk);
      if (COVSPEC_IN_BOUNDS(pos, k, status)) out[pos] = remap ? remap[i] : i;
    }
    run_gt += tot & 0xffffu;
    run_eq += tot >> 16;
  }
}

__device__ __forceinline__ void block_topk(const float* __restrict__ keys, int n, int k, bool all_equal,
                                           const int* __restrict__ remap, int* __restrict__ out, int* status) {
  block_topk_by([&](int i) { return keys[i]; }, n, k, all_equal, remap, out, status);
}

// Preselection: one block per request, the M best fused scores -> presel (ascending token index).
__global__ void __launch_bounds__(1024)
preselect_kernel(const float* __restrict__ s_fused, const ReqPlan* __restrict__ plan,
                 int* __restrict__ presel, int* status) {
  ReqPlan rp = plan[blockIdx.x];
  block_topk(s_fused + rp.vis_off, rp.n, rp.m, false, nullptr, presel + rp.presel_off, status);
}

// Eq. 12 and the preselection in one launch (the fused call): the block that fused a request's scores selects
// its M best right away.  Up to kRegKeys tokens per thread both scores, the fused score and its keys stay in
// registers from the one read of the scores to the selection; longer requests go through memory.
template <int PER>
__device__ __forceinline__ void fuse_select_regs(const ReqPlan& rp, const float* __restrict__ s_query,
                                                 const float* __restrict__ s_act, float lambda, int mode,
                                                 float* __restrict__ s_fused, int* __restrict__ presel, float* scratch,
                                                 int* status) {
  const int n = rp.n, tid = threadIdx.x, nt = blockDim.x;
  float q[PER], a[PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = tid + j * nt;
    q[j] = i < n ? s_query[rp.vis_off + i] : 0.f;
    a[j] = i < n && s_act != nullptr ? s_act[rp.vis_off + i] : 0.f;
  }
  const NormParams nq = norm_params_by<PER>([&](int j) { return q[j]; }, n, mode, scratch, status);
  NormParams na{0.f, 1.f};
  if (s_act != nullptr) na = norm_params_by<PER>([&](int j) { return a[j]; }, n, mode, scratch, status);
  unsigned key[PER];
  bool bad = false;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int i = tid + j * nt;
    key[j] = 0u;
    if (i < n) {
      const float f = s_act == nullptr ? (q[j] - nq.shift) * nq.scale
                                       : lambda * ((q[j] - nq.shift) * nq.scale) + (1.f - lambda) * ((a[j] - na.shift) * na.scale);
      s_fused[rp.vis_off + i] = f;
      bad |= !(fabsf(f) <= 3.402823466e38f);
      key[j] = order_key(f);
    }
  }
  if (bad) atomicOr(status, kStatusNonFinite);
  block_select_regs<PER>(key, n, rp.m, nullptr, presel + rp.presel_off, status);
}

__global__ void __launch_bounds__(1024)
fuse_preselect_kernel(const float* __restrict__ s_query, const float* __restrict__ s_act,
                      const ReqPlan* __restrict__ plan, float lambda, int mode,
                      float* __restrict__ s_fused, int* __restrict__ presel, int* status) {
  __shared__ float scratch[32];
  const ReqPlan rp = plan[blockIdx.x];
  if (rp.n <= 1024) fuse_select_regs<1>(rp, s_query, s_act, lambda, mode, s_fused, presel, scratch, status);
  else if (rp.n <= 4 * 1024) fuse_select_regs<4>(rp, s_query, s_act, lambda, mode, s_fused, presel, scratch, status);
  else if (rp.n <= kRegKeys * 1024) fuse_select_regs<kRegKeys>(rp, s_query, s_act, lambda, mode, s_fused, presel, scratch, status);
  else {
    fuse_request(rp, s_query, s_act, lambda, mode, s_fused, scratch, status);
    __syncthreads();                                  // the block's own global writes are visible to it
    block_topk(s_fused + rp.vis_off, rp.n, rp.m, false, nullptr, presel + rp.presel_off, status);
  }
}

// Final selection: one block per request, the B_vis largest energies among the M preselected
// tokens -> keep_idx (token indices, ascending).  Requests whose stage 2 is skipped keep their
// whole preselected set (B_vis == M).
__global__ void __launch_bounds__(1024)
final_select_kernel(const float* __restrict__ energy, const int* __restrict__ presel,
                    const ReqPlan* __restrict__ plan, int* __restrict__ keep_idx, int* status) {
  wait_for_previous_kernel();
  ReqPlan rp = plan[blockIdx.x];
  block_topk(energy + rp.presel_off, rp.m, rp.b_vis, rp.stage2 == 0, presel + rp.presel_off,
             keep_idx + rp.keep_off, status);
}

// out[row, :] = src[vis_off(b) + idx[row], :] as 16-byte vectors; one warp per output row (its
// first lane looks the request up), four vectors per lane in flight.
// `use_presel` selects which plan offsets delimit the rows of a request (presel_off / keep_off).
constexpr int kGatherWarps = 8;
__global__ void __launch_bounds__(kGatherWarps * 32)
gather_rows_kernel(const uint4* __restrict__ src, const int* __restrict__ idx,
                   const ReqPlan* __restrict__ plan, int batch, int use_presel, int row_vec16, int rows,
                   uint4* __restrict__ dst, int* __restrict__ out_pos, int* status) {
  const int lane = threadIdx.x & 31;
  const int row = blockIdx.x * kGatherWarps + (threadIdx.x >> 5);
  wait_for_previous_kernel();
  if (row >= rows) return;
  long long first = 0;
  int tok = 0;
  if (lane == 0) {
    int b = find_request(row, batch, [&](int q) {
      return use_presel ? plan[q].presel_off : plan[q].keep_off;
    });
    tok = idx[row];
    // checked build: a token index outside its request is reported and the row is skipped
    first = COVSPEC_IN_BOUNDS(tok, plan[b].n, status) ? (long long)plan[b].vis_off + tok : -1;
    if (out_pos != nullptr) out_pos[row] = tok;
  }
  first = __shfl_sync(0xffffffffu, first, 0);
  if (first < 0) return;
  const uint4* s = src + (size_t)first * row_vec16;
  uint4* d = dst + (size_t)row * row_vec16;
  int v = lane;
  for (; v + 96 < row_vec16; v += 128) {
    uint4 a = __ldg(s + v), b2 = __ldg(s + v + 32), c = __ldg(s + v + 64), e = __ldg(s + v + 96);
    d[v] = a; d[v + 32] = b2; d[v + 64] = c; d[v + 96] = e;
  }
  for (; v < row_vec16; v += 32) d[v] = __ldg(s + v);
}

inline unsigned gather_grid(long long rows) { return (unsigned)((rows + kGatherWarps - 1) / kGatherWarps); }

}  // namespace covspec
