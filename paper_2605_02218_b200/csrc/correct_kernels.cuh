// Device-side gating and correction over the vocabulary (Eq. 2, 4, 5, 6, 16, 17; Sec. III-C.2):
// from the draft logits and the target logits of one position, the draft distribution's top-2 margin
// and gate, the acceptance probability of the drafted token, the residual distribution
// max(p_t - p_d, 0) / mass and a token drawn from it by inverse CDF with a uniform number supplied by
// the caller.
//
// One cluster of CTAs per position.  Both logit rows (2 * W * elem bytes, ~600 KB at W = 152 k
// in 16 bits) are read from HBM once; the second sweep (residual mass) and the short third one (the
// cumulative sum inside the one warp segment that contains the sample) find them in L2.  Each warp
// owns a contiguous segment of the row and reads it with coalesced 16-byte vectors, so the order of
// the cumulative sum is (segment, vector, lane, element).  The method needs two exponentials per
// vocabulary entry for the denominators and two more for the residual; they run on the
// special-function units (16 per clock per SM), which bound the kernel before HBM does.
#pragma once
#include <cuda_fp16.h>

#include <atomic>

#include "common.cuh"
#include "select_kernels.cuh"

namespace covspec {
namespace corr {

constexpr int kThreads = 512;
constexpr int kWarps = kThreads / 32;
constexpr int kCtasPerSm = 2;                         // resident CTAs per SM the register budget allows
constexpr int kSegs = 32;                            // segments of a row, one warp's work with two CTAs per position
constexpr int kMaxChunks = 256;                      // chunks of a segment whose totals fit in shared memory

__device__ __forceinline__ float cvt(float v) { return v; }
__device__ __forceinline__ float cvt(__half v) { return __half2float(v); }
__device__ __forceinline__ float cvt(__nv_bfloat16 v) { return __bfloat162float(v); }

template <typename T> struct Vec;           // 16-byte vector of logits
template <> struct Vec<float> { static constexpr int N = 4; };
template <> struct Vec<__half> { static constexpr int N = 8; };
template <> struct Vec<__nv_bfloat16> { static constexpr int N = 8; };

constexpr float kLog2e = 1.4426950408889634f;

// 2^x on the special-function unit, results below the normal range flushed to zero (a probability
// under 1e-38): one instruction, where the denormal-preserving form takes four.
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// 16 bytes of logits: the largest element and the N values as floats.  Elements at or beyond `w`
// read as -inf (probability zero).  The row base is 16-byte aligned.
__device__ __forceinline__ void unpack(const uint4& raw, float (&v)[4], const float*) {
  v[0] = __uint_as_float(raw.x); v[1] = __uint_as_float(raw.y);
  v[2] = __uint_as_float(raw.z); v[3] = __uint_as_float(raw.w);
}
__device__ __forceinline__ void unpack(const uint4& raw, float (&v)[8], const __half*) {
  const __half2* h = reinterpret_cast<const __half2*>(&raw);
#pragma unroll
  for (int k = 0; k < 4; ++k) { float2 f = __half22float2(h[k]); v[2 * k] = f.x; v[2 * k + 1] = f.y; }
}
__device__ __forceinline__ void unpack(const uint4& raw, float (&v)[8], const __nv_bfloat16*) {
  const uint32_t u[4] = {raw.x, raw.y, raw.z, raw.w};
#pragma unroll
  for (int k = 0; k < 4; ++k) { v[2 * k] = __uint_as_float(u[k] << 16); v[2 * k + 1] = __uint_as_float(u[k] & 0xffff0000u); }
}
__device__ __forceinline__ float vec_max(const uint4& raw, const float*) {
  return fmaxf(fmaxf(__uint_as_float(raw.x), __uint_as_float(raw.y)),
               fmaxf(__uint_as_float(raw.z), __uint_as_float(raw.w)));
}
__device__ __forceinline__ float vec_max(const uint4& raw, const __half*) {
  const __half2* h = reinterpret_cast<const __half2*>(&raw);
  __half2 m = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));       // exact: a maximum rounds nothing
  return __half2float(__hmax(__low2half(m), __high2half(m)));
}
__device__ __forceinline__ float vec_max(const uint4& raw, const __nv_bfloat16*) {
  const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
  __nv_bfloat162 m = __hmax2(__hmax2(h[0], h[1]), __hmax2(h[2], h[3]));
  return __bfloat162float(__hmax(__low2bfloat16(m), __high2bfloat16(m)));
}

// The N consecutive logits that start at element `i` (a multiple of N) of `row`, as raw bits; the
// tail vector of a row whose length is not a multiple of N is completed with -inf.
template <typename T>
__device__ __forceinline__ uint4 load_raw(const T* __restrict__ row, int i, int w) {
  constexpr int N = Vec<T>::N;
  if (i + N <= w) return *reinterpret_cast<const uint4*>(row + i);
  T e[N];
#pragma unroll
  for (int k = 0; k < N; ++k) e[k] = i + k < w ? row[i + k] : (T)(-INFINITY);
  return *reinterpret_cast<const uint4*>(e);
}
template <typename T>
__device__ __forceinline__ void load_vec(const T* __restrict__ row, int i, int w, float (&v)[Vec<T>::N]) {
  unpack(load_raw(row, i, w), v, (const T*)nullptr);
}

// Running (max, sum of exp(z - max)) pair of a softmax denominator.
struct MaxSum {
  float m, s;
  // Branch-free: in a reduction by shuffles half of the lanes take either side, and the code for both
  // sides of five steps, run once per position, was fetched line by line (11 k cycles for four steps).
  __device__ __forceinline__ void merge(const MaxSum& o) {
    const bool up = o.m > m;
    const float hm = up ? o.m : m, hs = up ? o.s : s, lm = up ? m : o.m, ls = up ? s : o.s;
    m = hm;
    s = lm > -INFINITY ? fmaf(ls, __expf(lm - hm), hs) : hs;
  }
};
__device__ __forceinline__ MaxSum shfl_xor(const MaxSum& a, int o) {
  MaxSum r;
  r.m = __shfl_xor_sync(0xffffffffu, a.m, o);
  r.s = __shfl_xor_sync(0xffffffffu, a.s, o);
  return r;
}

// Probability of one logit: 2^(z log2(e) - c) with c = log2(e) max + log2(sum of exp(z - max)), one
// fused multiply-add and one special-function instruction.  Draft and target rows go through the
// same instructions, so identical rows give a residual of exactly zero.
__device__ __forceinline__ float prob(float z, float neg_c) { return ex2(fmaf(z, kLog2e, neg_c)); }

// Two largest values of a multiset.
struct Top2 {
  float a, b;   // a >= b
  __device__ __forceinline__ void add(float z) {
    if (z > a) { b = a; a = z; } else if (z > b) b = z;
  }
  __device__ __forceinline__ void merge(const Top2& o) {
    b = fmaxf(fminf(a, o.a), fmaxf(b, o.b));
    a = fmaxf(a, o.a);
  }
};

// Branch-free trackers of the two largest logits of the vectors one thread sees.  The 16-bit types
// keep two independent (largest, second) pairs, one per half of a packed register, on the raw bits:
// three packed min / max instructions per two logits, exact because a maximum rounds nothing.
template <typename T> struct Top2Run;
template <> struct Top2Run<float> {
  float a = -INFINITY, b = -INFINITY;
  __device__ __forceinline__ void add(const uint4& raw) {
    const float z[4] = {__uint_as_float(raw.x), __uint_as_float(raw.y), __uint_as_float(raw.z), __uint_as_float(raw.w)};
#pragma unroll
    for (int k = 0; k < 4; ++k) { b = fmaxf(b, fminf(a, z[k])); a = fmaxf(a, z[k]); }
  }
  __device__ __forceinline__ Top2 result() const { return Top2{a, b}; }
};
template <> struct Top2Run<__half> {
  __half2 a = __half2half2(__ushort_as_half((unsigned short)0xfc00)), b = a;       // -inf
  __device__ __forceinline__ void add(const uint4& raw) {
    const __half2* h = reinterpret_cast<const __half2*>(&raw);
#pragma unroll
    for (int k = 0; k < 4; ++k) { b = __hmax2(b, __hmin2(a, h[k])); a = __hmax2(a, h[k]); }
  }
  __device__ __forceinline__ Top2 result() const {
    Top2 t{__low2float(a), __low2float(b)};
    t.add(__high2float(a)); t.add(__high2float(b));
    return t;
  }
};
template <> struct Top2Run<__nv_bfloat16> {
  __nv_bfloat162 a = __bfloat162bfloat162(__ushort_as_bfloat16((unsigned short)0xff80)), b = a;   // -inf
  __device__ __forceinline__ void add(const uint4& raw) {
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&raw);
#pragma unroll
    for (int k = 0; k < 4; ++k) { b = __hmax2(b, __hmin2(a, h[k])); a = __hmax2(a, h[k]); }
  }
  __device__ __forceinline__ Top2 result() const {
    Top2 t{__low2float(a), __low2float(b)};
    t.add(__high2float(a)); t.add(__high2float(b));
    return t;
  }
};

// How far above the reference of a running sum a logit may lie before the sum is moved to a new
// reference: exp(60) ~ 1e26 leaves room for a whole vocabulary of such terms in float32.
constexpr float kRefSlack = 60.f;
// Lowest reference.  Masked entries (the type's lowest value, -1e30, ...) may open a lane's share of the row; relative
// to such a reference the exponent's rounding alone is beyond the range (1.44e9, for a reference of -1e9, is
// rounded by up to 64), the sum becomes infinite and the next move of the reference makes it NaN.  Entries this low
// weigh nothing beside an ordinary logit.
constexpr float kRefFloor = -1e9f;

// ---- thread-block cluster helpers (a position is shared by the CTAs of a cluster) ----
__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The address `p` (shared memory of this CTA) has in CTA `cta` of the cluster.
__device__ __forceinline__ unsigned peer_addr(const void* p, unsigned cta) {
  unsigned local = (unsigned)__cvta_generic_to_shared(p), remote;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(local), "r"(cta));
  return remote;
}
// Partial results are pushed into every CTA's shared memory ahead of a cluster barrier: a warp that
// fetches 32 scattered values of a peer waits 1.5-2 k cycles per load.
__device__ __forceinline__ void peer_store(unsigned addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void peer_store(unsigned addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void peer_store(unsigned addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}

// rows: positions; w: vocabulary size; ldz: elements between consecutive rows (multiple of 16 bytes).
//
// The row is cut into kSegs = 32 contiguous segments of whole 16-byte vectors; lane l of a segment owns its
// vectors l, l + 32, ... and adds their sums up in that order, whatever the number of warps that share the
// work, so that a result does not depend on how many positions a call has.
//   CL = 2: one cluster of two CTAs per position, one warp per segment, two CTAs resident per SM: the sweep
//           that streams the rows from HBM in one CTA overlaps the sweeps that re-read them from L2
//           (special-function bound) in the other CTA of the SM, while the positions in flight (one per
//           cluster) still fit in L2.
//   CL = 4, 8: 2 or 4 warps per segment, for calls with too few positions to fill the SMs: chunks of 32
//           vectors are dealt over the warps of the segment, the vector sums go through shared memory and
//           one warp adds them up.
// Partial results cross the cluster through distributed shared memory.  With `store` the residual sums of
// the vectors stay in shared memory: the draw then only scans them and evaluates one chunk of 32 vectors
// again, instead of the whole segment.
template <typename T, int CL>
__global__ void __launch_bounds__(kThreads, kCtasPerSm)
correct_kernel(const T* __restrict__ zd, const T* __restrict__ zt, long long ldz, int w,
               const int* __restrict__ drafted, const float* __restrict__ uniforms, float gamma,
               float* __restrict__ margin, int* __restrict__ gate, float* __restrict__ accept,
               float* __restrict__ resid_mass, int* __restrict__ token, int store) {
  constexpr int N = Vec<T>::N;
  constexpr int WPS = CL * kWarps / kSegs;         // warps per segment
  constexpr int SPC = kSegs / CL;                  // segments per CTA
  extern __shared__ float vec_sums[];              // [SPC][chunks][32] (store), [2][SPC][chunks][32] (WPS > 1)
  // results of the whole cluster, filled in by every CTA
  __shared__ float4 sh_seg[kSegs];                 // per segment: (max, sum) pairs of the draft and the target row
  __shared__ float2 sh_top[CL * kWarps];           // per warp: two largest draft logits
  __shared__ float sh_mass[2][kSegs];              // segment masses in row order (residual pass, p_t pass)
  __shared__ float sh_chunk[kMaxChunks];           // totals of the 32-vector chunks of the segment that holds the sample
  const unsigned crank = cluster_rank();
  const int row = blockIdx.x / CL, tid = threadIdx.x, lane = tid & 31, warp = warp_index();
  const int ls = warp / WPS, sub = warp % WPS;     // segment inside the CTA, warp inside the segment
  const int seg_id = (int)crank * SPC + ls;
  const T* rd = zd + (size_t)row * ldz;
  const T* rt = zt + (size_t)row * ldz;
  const T* const tag = nullptr;
  // peers may be written to once they have started: waited for after the first sweep
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  // scalars of the position, requested now so that their latency hides behind the first sweep
  const float x_uniform = __ldg(uniforms + row);
  float zd_y = 0.f, zt_y = 0.f;
  const bool has_y = accept != nullptr && drafted != nullptr;
  if (has_y && tid == 0 && crank == 0) {
    const int y = __ldg(drafted + row);
    zd_y = cvt(rd[y]);
    zt_y = cvt(rt[y]);
  }
  // contiguous segment of this warp, in whole vectors
  const int nvec = (w + N - 1) / N;
  const int vec_per_seg = (nvec + kSegs - 1) / kSegs;
  const int chunks = (vec_per_seg + 31) >> 5;
  const int v0 = min(nvec, seg_id * vec_per_seg), v1 = min(nvec, v0 + vec_per_seg);
  // vectors that lie wholly inside the row, then the one that straddles its end (if any)
  const int nfull = w / N, f1 = min(v1, nfull);
  const bool owns_tail = nfull < nvec && nfull >= v0 && nfull < v1 && ((nfull - v0) & 31) == lane;
  float* my_sums = vec_sums + (size_t)ls * chunks * 32 + lane;                       // + 32 * chunk
  float* my_sums2 = my_sums + (size_t)SPC * chunks * 32;

  // ---- sweep 1: softmax denominators of both rows (Eq. 2, 4), two largest draft logits (Eq. 16) ----
  // The sums run relative to a reference logit of this lane, in the base-2 domain:
  // exp(z - m) = 2^(z log2(e) - m log2(e)).  The reference is the largest logit of the first vector
  // and moves only when a logit lies more than kRefSlack above it (any reference gives the same
  // quotient; the slack keeps the terms inside the float32 range), so the branch is rarely taken.
  MaxSum md{-INFINITY, 0.f}, mt{-INFINITY, 0.f};
  float nd = 0.f, nt = 0.f;                     // -m log2(e) of the two references
  float thr_d = -INFINITY, thr_t = -INFINITY;   // reference + slack
  Top2Run<T> top_run;
  // sum of exp over one vector of either row, terms in element order
  auto exp_sums = [&](const uint4& ra, const uint4& rb) {
    float a[N], b[N];
    unpack(ra, a, tag);
    unpack(rb, b, tag);
    float sa = 0.f, sb = 0.f;
#pragma unroll
    for (int k = 0; k < N; ++k) {
      sa += ex2(fmaf(a[k], kLog2e, nd));
      sb += ex2(fmaf(b[k], kLog2e, nt));
    }
    return make_float2(sa, sb);
  };
  auto move_reference = [&](float va, float vb) {
    if (va > thr_d) {
      const float m = fmaxf(va, kRefFloor);
      md.s *= __expf(md.m - m); md.m = m; nd = -m * kLog2e; thr_d = m + kRefSlack;
    }
    if (vb > thr_t) {
      const float m = fmaxf(vb, kRefFloor);
      mt.s *= __expf(mt.m - m); mt.m = m; nt = -m * kLog2e; thr_t = m + kRefSlack;
    }
  };
  auto sweep1 = [&](const uint4& ra, const uint4& rb) {
    // every vector holds at least one element of the vocabulary; 2^(-inf) = 0 takes care of padding
    move_reference(vec_max(ra, tag), vec_max(rb, tag));
    const float2 s = exp_sums(ra, rb);
    md.s += s.x;
    mt.s += s.y;
  };
  auto sweep1_segment = [&]() {                 // the whole segment by one warp
    const uint4* pa = reinterpret_cast<const uint4*>(rd) + v0 + lane;
    const uint4* pb = reinterpret_cast<const uint4*>(rt) + v0 + lane;
#pragma unroll 2
    for (int v = v0 + lane; v < f1; v += 32, pa += 32, pb += 32) {
      const uint4 ra = __ldg(pa), rb = __ldg(pb);
      sweep1(ra, rb);
      if (WPS == 1) top_run.add(ra);
    }
    if (owns_tail) {
      const uint4 ra = load_raw(rd, nfull * N, w);
      sweep1(ra, load_raw(rt, nfull * N, w));
      if (WPS == 1) top_run.add(ra);
    }
  };
  if constexpr (WPS == 1) {
    sweep1_segment();
  } else {
    // the lane's reference is that of its first vector; a warp that meets a logit too far above it makes
    // one warp go through the segment again in order
    const int vref = v0 + lane < v1 ? v0 + lane : -1;
    if (vref >= 0) move_reference(vec_max(load_raw(rd, vref * N, w), tag), vec_max(load_raw(rt, vref * N, w), tag));
    bool moved = false;
#pragma unroll 2
    for (int c = sub; c < chunks; c += WPS) {
      const int v = v0 + 32 * c + lane;
      if (v < v1) {
        const uint4 ra = load_raw(rd, v * N, w), rb = load_raw(rt, v * N, w);
        moved |= vec_max(ra, tag) > thr_d || vec_max(rb, tag) > thr_t;
        const float2 s = exp_sums(ra, rb);
        my_sums[32 * c] = s.x;
        my_sums2[32 * c] = s.y;
        top_run.add(ra);
      }
    }
    const int again = __syncthreads_or(moved);
    if (sub == 0) {
      if (again) {
        md = MaxSum{-INFINITY, 0.f}; mt = md;
        thr_d = thr_t = -INFINITY;
        sweep1_segment();
      } else {
#pragma unroll 4
        for (int c = 0; c < chunks; ++c)
          if (v0 + 32 * c + lane < v1) { md.s += my_sums[32 * c]; mt.s += my_sums2[32 * c]; }
      }
    }
  }
  Top2 top = top_run.result();
#pragma unroll 1
  for (int o = 16; o > 0; o >>= 1) {
    if (sub == 0) { md.merge(shfl_xor(md, o)); mt.merge(shfl_xor(mt, o)); }
    Top2 other{__shfl_xor_sync(0xffffffffu, top.a, o), __shfl_xor_sync(0xffffffffu, top.b, o)};
    top.merge(other);
  }
  __syncwarp();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  if (lane < CL) {
    if (sub == 0) peer_store(peer_addr(&sh_seg[seg_id], (unsigned)lane), make_float4(md.m, md.s, mt.m, mt.s));
    peer_store(peer_addr(&sh_top[(int)crank * kWarps + warp], (unsigned)lane), make_float2(top.a, top.b));
  }
  cluster_sync();                               // every CTA has all partial results
  // the same merge in every warp of the cluster: lane q holds segment q; each half of the segments is
  // merged in a butterfly of its own, then the two halves
  const float4 mine_seg = sh_seg[lane];
  MaxSum sd{mine_seg.x, mine_seg.y}, st{mine_seg.z, mine_seg.w};
  top = Top2{-INFINITY, -INFINITY};
#pragma unroll
  for (int q = 0; q < WPS; ++q) {
    const float2 o = sh_top[lane * WPS + q];
    top.merge(Top2{o.x, o.y});
  }
#pragma unroll 1
  for (int o = 8; o > 0; o >>= 1) {             // inside the halves
    sd.merge(shfl_xor(sd, o)); st.merge(shfl_xor(st, o));
    Top2 other{__shfl_xor_sync(0xffffffffu, top.a, o), __shfl_xor_sync(0xffffffffu, top.b, o)};
    top.merge(other);
  }
  {
    Top2 other{__shfl_xor_sync(0xffffffffu, top.a, 16), __shfl_xor_sync(0xffffffffu, top.b, 16)};
    top.merge(other);
  }
  // the lower half's result, then the upper half's, in every lane
  md = MaxSum{__shfl_sync(0xffffffffu, sd.m, 0), __shfl_sync(0xffffffffu, sd.s, 0)};
  mt = MaxSum{__shfl_sync(0xffffffffu, st.m, 0), __shfl_sync(0xffffffffu, st.s, 0)};
  md.merge(MaxSum{__shfl_sync(0xffffffffu, sd.m, 16), __shfl_sync(0xffffffffu, sd.s, 16)});
  mt.merge(MaxSum{__shfl_sync(0xffffffffu, st.m, 16), __shfl_sync(0xffffffffu, st.s, 16)});
  // exponent offsets of the two distributions: p = 2^(z log2(e) + offset)
  const float cd = -(md.m * kLog2e + log2f(md.s)), ct = -(mt.m * kLog2e + log2f(mt.s));
  if (crank == 0 && tid == 0) {                 // off the critical path of the other warps
    float m = (1.f - (top.b > -INFINITY ? __expf(top.b - top.a) : 0.f)) * __expf(top.a - md.m) / md.s;
    margin[row] = m;
    gate[row] = m < gamma ? 1 : 0;                                       // Eq. 17
    if (accept != nullptr) {
      float al = 1.f;
      if (has_y) {
        float pd = __expf(zd_y - md.m) / md.s, pt = __expf(zt_y - mt.m) / mt.s;
        al = pd > 0.f ? fminf(1.f, pt / pd) : 1.f;                       // Eq. 5
      }
      accept[row] = al;
    }
  }

  // ---- sweep 2: residual mass per segment (Eq. 6 denominator) ----
  // use_pt: the residual is identically zero (the two distributions coincide): draw from p_t.
  for (int use_pt = 0; use_pt < 2; ++use_pt) {
    float part = 0.f;
    if (!use_pt) {
      auto residual = [&](const uint4& ra, const uint4& rb) {         // summed over one vector, in element order
        float a[N], b[N];
        unpack(ra, a, tag);
        unpack(rb, b, tag);
        float acc = 0.f;
#pragma unroll
        for (int k = 0; k < N; ++k) acc += fmaxf(prob(b[k], ct) - prob(a[k], cd), 0.f);
        return acc;
      };
      if constexpr (WPS == 1) {
        const uint4* pa = reinterpret_cast<const uint4*>(rd) + v0 + lane;
        const uint4* pb = reinterpret_cast<const uint4*>(rt) + v0 + lane;
        float* keep = my_sums;
#pragma unroll 2
        for (int v = v0 + lane; v < f1; v += 32, pa += 32, pb += 32, keep += 32) {
          const float acc = residual(__ldg(pa), __ldg(pb));
          if (store) *keep = acc;
          part += acc;
        }
        if (owns_tail) {
          const float acc = residual(load_raw(rd, nfull * N, w), load_raw(rt, nfull * N, w));
          if (store) my_sums[nfull - v0 - lane] = acc;
          part += acc;
        }
      } else {
#pragma unroll 2
        for (int c = sub; c < chunks; c += WPS) {
          const int v = v0 + 32 * c + lane;
          if (v < v1) my_sums[32 * c] = residual(load_raw(rd, v * N, w), load_raw(rt, v * N, w));
        }
        __syncthreads();
        if (sub == 0)
#pragma unroll 4
          for (int c = 0; c < chunks; ++c)
            if (v0 + 32 * c + lane < v1) part += my_sums[32 * c];
      }
    } else if (sub == 0) {
      for (int v = v0 + lane; v < v1; v += 32) {
        float b[N];
        load_vec(rt, v * N, w, b);
#pragma unroll
        for (int k = 0; k < N; ++k) part += prob(b[k], ct);
      }
    }
    part = warp_sum(part);
    if (sub == 0 && lane < CL) peer_store(peer_addr(&sh_mass[use_pt][seg_id], (unsigned)lane), part);
    cluster_sync();                             // every CTA has all segment masses (the last access to a peer)
    const float* sh_all = sh_mass[use_pt];
    float mass = 0.f;
#pragma unroll
    for (int q = 0; q < kSegs; ++q) mass += sh_all[q];                    // same order in every thread
    if (!use_pt && crank == 0 && tid == 0 && resid_mass != nullptr) resid_mass[row] = mass;
    if (mass > 0.f || use_pt) {
      // ---- sweep 3: the warp whose segment contains x * mass walks it in order ----
      const float target = x_uniform * mass;
      float before = 0.f;
      int seg = -1;
#pragma unroll
      for (int q = 0; q < kSegs; ++q) {
        const float next = before + sh_all[q];
        if (seg < 0 && next > target) seg = q;
        if (seg < 0) before = next;
      }
      float tgt = target;
      if (seg < 0) {
        // rounding left x * mass at or above the total: the last token with positive probability,
        // i.e. the walk below never crosses and reports the last positive entry of this segment
        seg = kSegs - 1;
        while (seg > 0 && !(sh_all[seg] > 0.f)) --seg;
        tgt = INFINITY;
      }
      if (seg / SPC != (int)crank) break;       // another CTA's segment
      // The segment is walked in chunks of 32 vectors.  The warps of the CTA that owns it first
      // sum the chunks in parallel; the walk then starts at the first chunk whose running total
      // passes the target (running totals added up in chunk order, as the walk itself would).
      const int sv0 = min(nvec, seg * vec_per_seg), sv1 = min(nvec, sv0 + vec_per_seg);
      const int nchunks = (sv1 - sv0 + 31) >> 5;
      const bool skip_ahead = nchunks <= kMaxChunks && tgt != INFINITY;
      auto chunk_values = [&](int v, float (&r)[N]) -> float {
        float lsum = 0.f;
        if (v < sv1) {
          float a[N], b[N];
          load_vec(rd, v * N, w, a);
          load_vec(rt, v * N, w, b);
#pragma unroll
          for (int k = 0; k < N; ++k) {
            float pt = prob(b[k], ct), pd = prob(a[k], cd);
            r[k] = use_pt ? pt : fmaxf(pt - pd, 0.f);
            lsum += r[k];
          }
        } else {
#pragma unroll
          for (int k = 0; k < N; ++k) r[k] = 0.f;
        }
        return lsum;
      };
      if (skip_ahead) {
        const float* kept = vec_sums + (size_t)(seg - (int)crank * SPC) * chunks * 32 + lane;
        for (int c = warp; c < nchunks; c += kWarps) {
          float r[N], inc;
          if (store && !use_pt) inc = sv0 + 32 * c + lane < sv1 ? kept[32 * c] : 0.f;
          else inc = chunk_values(sv0 + 32 * c + lane, r);
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {          // the same inclusive scan the walk uses
            float t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
          }
          if (lane == 31) sh_chunk[c] = inc;
        }
      }
      __syncthreads();
      if (seg_id == seg && sub == 0) {
        float run = before;
        int first_chunk = 0;
        if (skip_ahead) {
          while (first_chunk + 1 < nchunks && !(run + sh_chunk[first_chunk] > tgt)) run += sh_chunk[first_chunk++];
        }
        int found = -1, last_pos = -1;
        for (int vb = v0 + 32 * first_chunk; vb < v1; vb += 32) {
          int v = vb + lane;
          float r[N];
          float lsum = chunk_values(v, r);
          // exclusive prefix over lanes
          float inc = lsum;
#pragma unroll
          for (int o = 1; o < 32; o <<= 1) {
            float t = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += t;
          }
          float acc = run + inc - lsum;
          int mine = -1, mylast = -1;
#pragma unroll
          for (int k = 0; k < N; ++k) {
            if (r[k] > 0.f) mylast = v * N + k;
            acc += r[k];
            if (mine < 0 && r[k] > 0.f && acc > tgt) mine = v * N + k;
          }
          // first lane that crossed; last positive element seen so far
          unsigned hit = __ballot_sync(0xffffffffu, mine >= 0);
          unsigned pos = __ballot_sync(0xffffffffu, mylast >= 0);
          if (pos) last_pos = __shfl_sync(0xffffffffu, mylast, 31 - __clz(pos));
          if (hit) { found = __shfl_sync(0xffffffffu, mine, __ffs(hit) - 1); break; }
          run += __shfl_sync(0xffffffffu, inc, 31);
        }
        int tk = found >= 0 ? found : last_pos;
        if (tk < 0 && lane == 0) {
          // the chosen segment held no positive entry at all (possible only through rounding):
          // scan back for the last positive probability in the whole row
          for (int i = w - 1; i >= 0 && tk < 0; --i) {
            float pt = prob(cvt(rt[i]), ct), pd = prob(cvt(rd[i]), cd);
            if ((use_pt ? pt : pt - pd) > 0.f) tk = i;
          }
        }
        if (lane == 0) token[row] = tk;
      }
      break;
    }
    __syncthreads();
  }
}

// CTAs per position.  Few positions are spread over up to eight CTAs each, so that a drafted block of eight positions uses
// 64 SMs instead of 16, for as long as every CTA gets an SM to itself: 128 CTAs of clusters of 4 or 8 do on 148 SMs
// (a cluster stays inside one GPC, so not every SM can be had); beyond that two CTAs of one SM take their
// sweeps in turn and splitting costs more than it gives.  151,674 float16 logits, calls back to back in a graph,
// clusters of 8 / 4 / 2: 8 positions 13.0 / 16.8 / 19.1 us, 16: 16.8 / 17.0 / 19.1, 32: 19.7 / 17.4 / 19.4,
// 38: 27.3 / 23.3 / 19.3, 74: 41.5 / 34.9 / 19.7.  float32 rows (twice the bytes): 8: 16.1 / 21.8 / 22.8,
// 24: 20.7 / 22.0 / 22.9, 32: 22.3 / 22.4 / 23.4, 38: 33.0 / 28.4 / 23.4; clusters of 8 all the way.
constexpr int kSpreadCtas = 128;
template <typename T>
int cluster_ctas(int rows) {
  if (4 * rows > kSpreadCtas) return 2;
  return 8 * rows <= kSpreadCtas || sizeof(T) == 4 ? 8 : 4;
}
constexpr size_t kSumsMost = 96 * 1024;              // shared memory for the vector sums: two CTAs per SM
// Dynamic shared memory of a CTA: one sum per vector of its segments, two where several warps share one.
template <typename T>
size_t sums_bytes(int cl, int w) {
  const int nvec = (w + Vec<T>::N - 1) / Vec<T>::N, chunks = ((nvec + kSegs - 1) / kSegs + 31) / 32;
  return (size_t)(kSegs / cl) * chunks * 32 * sizeof(float) * (cl > 2 ? 2 : 1);
}

template <typename T, int CL>
cudaError_t launch_correct_n(int rows, const T* zd, const T* zt, long long ldz, int w, const int* drafted,
                             const float* uniforms, float gamma, float* margin, int* gate, float* accept,
                             float* resid_mass, int* token, cudaStream_t s) {
  static std::atomic<unsigned long long> configured{0};   // bit per device; setting the attribute twice is harmless
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev >= 64 || !(configured.load(std::memory_order_acquire) >> dev & 1ull)) {
    e = cudaFuncSetAttribute(correct_kernel<T, CL>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSumsMost);
    if (e != cudaSuccess) return e;
    if (dev < 64) configured.fetch_or(1ull << dev, std::memory_order_release);
  }
  const size_t bytes = sums_bytes<T>(CL, w);
  const bool store = bytes <= kSumsMost;
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((unsigned)rows * CL);
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = store ? bytes : 0;
  cfg.stream = s;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeClusterDimension;
  attr.val.clusterDim.x = CL;
  attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
  cfg.attrs = &attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, correct_kernel<T, CL>, zd, zt, ldz, w, drafted, uniforms, gamma, margin, gate, accept,
                            resid_mass, token, store ? 1 : 0);
}
template <typename T>
cudaError_t launch_correct(int rows, const T* zd, const T* zt, long long ldz, int w, const int* drafted,
                           const float* uniforms, float gamma, float* margin, int* gate, float* accept,
                           float* resid_mass, int* token, cudaStream_t s) {
  int cl = cluster_ctas<T>(rows);
  if (sums_bytes<T>(cl, w) > kSumsMost) cl = 2;       // a row too long for sums in shared memory: two CTAs need none
  const auto f = cl == 2 ? launch_correct_n<T, 2> : cl == 4 ? launch_correct_n<T, 4> : launch_correct_n<T, 8>;
  return f(rows, zd, zt, ldz, w, drafted, uniforms, gamma, margin, gate, accept, resid_mass, token, s);
}

// Logit i of a row as the candidate selections see it: the drafted token `y` comes last, behind entries masked with -inf
// (NaN has the smallest key).
template <typename T>
__device__ __forceinline__ float entry(const T* __restrict__ r, int i, int y) {
  return i == y ? __int_as_float(0x7fc00000) : cvt(r[i]);
}

// Bonus-token candidates of the parallel branching (Sec. III-C.1, Eq. 23): for every position the
// F_j largest draft logits, the token drafted at that position excluded; ties go to the lower
// token id; ids are written in ascending order at cand[cand_offsets[row] ...].  One block per
// position (segmented radix select over the logit row, which stays in L2 between its passes).
template <typename T>
__global__ void __launch_bounds__(1024)
branch_candidates_kernel(const T* __restrict__ zd, long long ldz, int w, const int* __restrict__ drafted,
                         const int* __restrict__ cand_offsets, int* __restrict__ cand) {
  const int row = blockIdx.x;
  const int off = cand_offsets[row], f = cand_offsets[row + 1] - off;
  if (f <= 0) return;
  const T* r = zd + (size_t)row * ldz;
  const int y = drafted != nullptr ? drafted[row] : -1;
  block_topk_by([&](int i) { return entry(r, i, y); }, w, min(f, w), false, nullptr,
                cand + off, nullptr);
}

// The same for small fan-outs (the usual case: F_j = ceil(F_0 rho^j) of a handful): one cluster of eight
// CTAs per position streams the row once.  The F_j-th largest of the 128 warps' maxima bounds the F_j-th
// largest key of the row from below, so only the few threads that saw a key that large look at
// their vectors again, and what they find (F_j entries and a few more) is ranked by one CTA.  One block
// per position with five passes over the row read it at one SM's rate: 32 positions x 151,674 float16
// logits 290 us.
constexpr int kFastFanout = 64;                      // largest fan-out of this kernel
constexpr int kFastCtas = 8, kFastThreads = 512;
constexpr int kFastWarps = kFastCtas * kFastThreads / 32;
constexpr int kFastMinVec = 32 * kFastFanout;        // shorter rows give fewer warps with a vector than F_j may ask for
constexpr int kFastList = 1024;                      // entries that are ranked directly
constexpr int kFastRows = 512;                       // positions per launch: their offsets travel as kernel arguments
struct FanOffsets { int v[kFastRows + 1]; };

// The F_j first of the n listed entries in (larger key, lower id) order, written by ascending id.
__device__ __forceinline__ void write_ranked(const unsigned* list_key, const int* list_id, int n, int f, unsigned* chosen,
                                             int* __restrict__ cand) {
  for (int q = (int)threadIdx.x; q < kFastList / 32; q += kFastThreads) chosen[q] = 0u;
  __syncthreads();
  for (int e = (int)threadIdx.x; e < n; e += kFastThreads) {
    const unsigned k = list_key[e];
    const int id = list_id[e];
    int rank = 0;
    for (int j = 0; j < n; ++j) rank += list_key[j] > k || (list_key[j] == k && list_id[j] < id);
    if (rank < f) atomicOr(&chosen[e >> 5], 1u << (e & 31));
  }
  __syncthreads();
  for (int e = (int)threadIdx.x; e < n; e += kFastThreads) {
    if (!(chosen[e >> 5] >> (e & 31) & 1u)) continue;
    const int id = list_id[e];
    int pos = 0;
    for (int j = 0; j < n; ++j) pos += (chosen[j >> 5] >> (j & 31) & 1u) && list_id[j] < id;
    cand[pos] = id;
  }
}

// The general selection.
template <typename T>
__device__ __forceinline__ void select_row(const T* __restrict__ r, int w, int y, int f, int* __restrict__ cand) {
  block_topk_by([&](int i) { return entry(r, i, y); }, w, f, false, nullptr, cand, nullptr);
}

// Mass ties: a row masked down to fewer tokens than F_j, say, whose F_j-th largest key (the threshold) is the mask, so
// that more entries reach it than are ranked directly.  One CTA lists what lies above the threshold (raising it while
// that is more than the list holds), takes ties in the order of their ids until it has F_j, and writes the candidates.  A row
// of 151,674 float16 logits with 15 of them unmasked, F_j = 32, eight rows: 26 us (499 with every thread that saw a tie
// at the counter and the general selection behind it).  In line: a call, although hardly ever taken, made the
// usual path 4 % longer.
template <typename T>
__device__ __forceinline__ void list_ties(const T* __restrict__ r, int w, int y, int f, unsigned threshold, unsigned* count,
                                          unsigned* list_key, int* list_id, unsigned* chosen, int* __restrict__ cand) {
  constexpr int N = Vec<T>::N;
  __shared__ unsigned scan_totals[33];
  __shared__ unsigned raised;
  const int tid = threadIdx.x, nvec = (w + N - 1) / N;
  __syncthreads();                                   // everybody has read the count
  if (tid == 0) *count = 0u;
  __syncthreads();
  auto special = [&](int v) { return (v + 1) * N > w || (y >= v * N && y < (v + 1) * N); };
  auto each = [&](int v, auto take) {                // (id, key) of every entry of vector v
    if (special(v)) {
      for (int i = v * N; i < min(w, (v + 1) * N); ++i) take(i, order_key(entry(r, i, y)));
    } else {
      float e[N];
      unpack(__ldg(reinterpret_cast<const uint4*>(r) + v), e, (const T*)nullptr);
#pragma unroll
      for (int q = 0; q < N; ++q) take(v * N + q, order_key(e[q]));
    }
  };
  int n = 0;
  for (int round = 0;; ++round) {
#pragma unroll 4
    for (int v = tid; v < nvec; v += kFastThreads) {
      if (!special(v) && order_key(vec_max(__ldg(reinterpret_cast<const uint4*>(r) + v), (const T*)nullptr)) <= threshold) continue;
      each(v, [&](int i, unsigned k) {
        if (k <= threshold) return;
        const unsigned at = atomicAdd(count, 1u);
        if (at < (unsigned)kFastList) { list_key[at] = k; list_id[at] = i; }
      });
    }
    __syncthreads();
    n = (int)min(*count, (unsigned)(kFastList + 1));
    if (n <= kFastList) break;
    if (round == 3) {
      select_row<T>(r, w, y, f, cand);
      return;
    }
    // more than the list holds: the F_j-th largest of those it holds is a higher threshold that F_j entries reach
    for (int e = tid; e < kFastList; e += kFastThreads) {
      const unsigned k = list_key[e];
      int above = 0, reach = 0;
      for (int j = 0; j < kFastList; ++j) { above += list_key[j] > k; reach += list_key[j] >= k; }
      if (above < f && f <= reach) raised = k;
    }
    __syncthreads();
    threshold = raised;
    if (tid == 0) *count = 0u;
    __syncthreads();
  }
  for (int v0 = 0; n < f && v0 < nvec; v0 += kFastThreads) {         // n: the same in all threads
    const int v = v0 + tid;
    unsigned ties = 0u, total;
    if (v < nvec) each(v, [&](int, unsigned k) { ties += k == threshold; });
    int at = n + (int)block_exclusive_scan(ties, scan_totals, &total);
    if (ties != 0u)
      each(v, [&](int i, unsigned k) {
        if (k != threshold) return;
        if (at < f) { list_key[at] = k; list_id[at] = i; }
        ++at;
      });
    n = min(f, n + (int)total);
  }
  __syncthreads();
  write_ranked(list_key, list_id, n, f, chosen, cand);
}

template <typename T>
__global__ void __cluster_dims__(kFastCtas, 1, 1) __launch_bounds__(kFastThreads)
branch_fast_kernel(const T* __restrict__ zd, long long ldz, int w, const int* __restrict__ drafted,
                   const int* __restrict__ dev_offsets, const __grid_constant__ FanOffsets host_offsets,
                   int* __restrict__ cand) {
  constexpr int N = Vec<T>::N;
  __shared__ __align__(16) unsigned keys[kFastWarps];
  __shared__ unsigned warp_best[kFastThreads / 32];
  __shared__ unsigned s_threshold, s_count;
  __shared__ unsigned list_key[kFastList];
  __shared__ int list_id[kFastList];
  __shared__ unsigned chosen[kFastList / 32];
  const unsigned crank = cluster_rank();
  const int row = blockIdx.x / kFastCtas, tid = threadIdx.x;
  const int off = dev_offsets != nullptr ? dev_offsets[row] : host_offsets.v[row];
  const int f = min((dev_offsets != nullptr ? dev_offsets[row + 1] : host_offsets.v[row + 1]) - off, w);
  if (f <= 0) return;                                // the whole cluster
  const T* r = zd + (size_t)row * ldz;
  const int y = drafted != nullptr ? __ldg(drafted + row) : -1;
  if (f > kFastFanout) {                             // offsets that ask for more than max_fanout said (again the whole cluster)
    if (crank == 0) select_row<T>(r, w, y, f, cand + off);
    return;
  }
  const int nvec = (w + N - 1) / N, first = (int)crank * kFastThreads + tid;
  constexpr int kStep = kFastCtas * kFastThreads;
  if (tid == 0) s_count = 0u;
  auto key_at = [&](int i) { return order_key(entry(r, i, y)); };
  auto special = [&](int v) { return (v + 1) * N > w || (y >= v * N && y < (v + 1) * N); };   // row end, drafted token
  unsigned mine = 0u;
#pragma unroll 4
  for (int v = first; v < nvec; v += kStep) {
    if (special(v)) {
      for (int i = v * N; i < min(w, (v + 1) * N); ++i) mine = max(mine, key_at(i));
    } else {
      mine = max(mine, order_key(vec_max(__ldg(reinterpret_cast<const uint4*>(r) + v), (const T*)nullptr)));
    }
  }
  {
    const unsigned m = __reduce_max_sync(0xffffffffu, mine);
    if ((tid & 31) == 0) warp_best[tid >> 5] = m;
  }
  cluster_sync();                                    // every CTA's maxima are in its shared memory
  if (tid < kFastWarps) {
    unsigned k;
    const unsigned a = peer_addr(&warp_best[tid & (kFastThreads / 32 - 1)], (unsigned)(tid / (kFastThreads / 32)));
    asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(k) : "r"(a) : "memory");
    keys[tid] = k;
  }
  __syncthreads();
  if (tid < kFastWarps) {
    const unsigned k = keys[tid];
    int rank = 0;                                    // maxima before this one in (larger, earlier) order
#pragma unroll 8
    for (int j = 0; j < kFastWarps; j += 4) {
      const uint4 q = *reinterpret_cast<const uint4*>(keys + j);
      rank += (q.x > k || (q.x == k && j < tid)) + (q.y > k || (q.y == k && j + 1 < tid)) +
              (q.z > k || (q.z == k && j + 2 < tid)) + (q.w > k || (q.w == k && j + 3 < tid));
    }
    if (rank == f - 1) s_threshold = k;
  }
  __syncthreads();
  const unsigned threshold = s_threshold;
  // far more warps at the threshold than F_j: mass ties, which CTA 0 takes up by itself (thousands of threads would
  // queue up at its counter)
  bool push = __any_sync(0xffffffffu, mine >= threshold);
  if (push) {
    const uint4 q = *reinterpret_cast<const uint4*>(keys + 4 * (tid & 31));
    push = __reduce_add_sync(0xffffffffu, (q.x >= threshold) + (q.y >= threshold) + (q.z >= threshold) + (q.w >= threshold)) <=
           f + kFastWarps / 4;
  }
  if (push && mine >= threshold) {
    auto take = [&](int i, unsigned k) {
      if (k < threshold) return;
      unsigned at;
      asm volatile("atom.shared::cluster.add.u32 %0, [%1], 1;" : "=r"(at) : "r"(peer_addr(&s_count, 0u)) : "memory");
      if (at < (unsigned)kFastList) {
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(&list_key[at], 0u)), "r"(k) : "memory");
        asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_addr(&list_id[at], 0u)), "r"(i) : "memory");
      }
    };
#pragma unroll 1
    for (int v = first; v < nvec; v += kStep) {
      if (special(v)) {
        for (int i = v * N; i < min(w, (v + 1) * N); ++i) take(i, key_at(i));
      } else {
        const uint4 raw = __ldg(reinterpret_cast<const uint4*>(r) + v);
        if (order_key(vec_max(raw, (const T*)nullptr)) < threshold) continue;
        float e[N];
        unpack(raw, e, (const T*)nullptr);
#pragma unroll
        for (int q = 0; q < N; ++q) take(v * N + q, order_key(e[q]));
      }
    }
  }
  cluster_sync();                                    // the list is complete in CTA 0
  if (crank != 0) return;
  const int n = (int)min(s_count, (unsigned)(kFastList + 1));
  if (n < f || n > kFastList) {                      // nothing was pushed, or too much
    list_ties<T>(r, w, y, f, threshold, &s_count, list_key, list_id, chosen, cand + off);
    return;
  }
  write_ranked(list_key, list_id, n, f, chosen, cand + off);
}

}  // namespace corr
}  // namespace covspec
