// Small dense building blocks of the top-r subspace solver behind Eq. 14-15 (used by the fused
// kernel in subspace_fused.cuh).
//
// The energies c_i = sum_{k<=r} lambda_k V_ik^2 are the diagonal of the best rank-r approximation of
// the Gram matrix G = Z_M^T Z_M (lambda_k = sigma_k^2, V = right singular vectors of Z_M).  The
// library reaches the top-r eigenspace of G by block subspace iteration with p = r + oversample
// vectors.  Every step leaves the float64 Gram matrix B = Y^T Y of the new block as per-tile partial
// sums; its Cholesky factor L makes Q = Y L^-T an orthonormal basis.  After the last step
// Y' = G Q^T: Rayleigh-Ritz for G^2 on the span of the last `win` basis vectors, whose Ritz matrix
// is the trailing win x win block of B' = Y'^T Y' = Q G^2 Q^T.  Its Cholesky factor is diagonalised
// by one-sided Jacobi rotations (this file); the eigenvectors u_k of the p - r smallest Ritz values
// are kept.  For an orthonormal basis of a G-invariant subspace, sum_k lambda_k V_ik^2 =
// sum_j Y'_ij Q_ij; the energy in the top-r subspace is that total over all p basis vectors minus
// the part of the p - r smallest Ritz pairs,
//   c_i = sum_j Y'_ij Q_ij - sum_k (Y'_i,win u_k)(Q_i,win u_k).
// Only the Ritz pairs next to the cut at r have to be resolved individually: basis vectors more
// than 16 places above the cut are separated from the discarded ones by the same eigenvalue ratios
// that drive the subspace iteration itself, so the window has p - r + min(16, r) vectors (all p when
// the problem is small).
#pragma once
#include "subspace_tc.cuh"

namespace covspec {

using sub::kLbufStride;
using sub::kLtFloats;
using sub::kTriMax;
using sub::kXsLd;
using sub::lt_row_offset;
using sub::tri_index;

// Bytes of shared memory the blocked Cholesky factorisation needs for an n x n matrix (8 x 8 tiles
// of the lower triangle in float64, the original diagonal and the reciprocal pivots).
__host__ __device__ constexpr size_t cholesky_smem_bytes(int n) {
  int nb = (n + 7) / 8;
  return ((size_t)nb * (nb + 1) / 2 * 64 + 16 * nb) * sizeof(double);
}

// One-sided Jacobi on the w columns C[c * ldc + row] (w <= 4 * ROWS): rotate column pairs until
// they are mutually orthogonal.  Round-robin ordering, w/2 disjoint pairs per round, one 4-lane
// group per pair with the two columns held in registers between the inner products and the
// rotation, so that a round is a short instruction stream on few warps and the barrier between
// rounds spans only those warps (named barrier 1 over `nact` threads, a multiple of 32; the caller guarantees
// that exactly the threads tid < nact enter).  A pair is left alone when its inner product g is
// negligible against the two norms (g^2 <= 1e-12 |a|^2 |b|^2) or so small that the energies move by
// less than ~2e-5 of the problem's scale s1 (g^2 <= (2e-5 s1)^2 min(|a|^2, |b|^2)).  Returns false
// when max_sweeps sweeps did not reach a sweep without rotations.
template <int ROWS>
__device__ __forceinline__ bool jacobi_sweeps(float* C, int ldc, int w, float s1, int max_sweeps,
                                              int nact, volatile int* flag) {
  const int tid = threadIdx.x;
  const int np = (w + 1) & ~1, half = np >> 1;
  const int g = tid >> 2, gl = tid & 3;
  const float abs2 = (2e-5f * s1) * (2e-5f * s1);
  bool converged = w < 2;
  for (int sweep = 0; sweep < max_sweeps && !converged; ++sweep) {
    int rotated = 0;
    for (int round = 0; round < np - 1; ++round) {
      // windows of more than nact / 2 columns have more pairs than groups: the groups go round again (the pairs of
      // a round are disjoint, so their order does not matter)
      for (int g0 = 0; g0 < half; g0 += nact >> 2) {
        const int pair = g0 + g;
        int a = 0, b = 0;
        bool active = pair < half;
        if (active) {
          a = round + pair; if (a >= np - 1) a -= np - 1;
          b = round - pair; if (b < 0) b += np - 1;
          if (pair == 0) { a = round; b = np - 1; }
          if (a > b) { int t = a; a = b; b = t; }
          active = b < w;
        }
        float* ca = C + a * ldc;
        float* cb = C + b * ldc;
        float xa[ROWS], xb[ROWS];
        float al = 0.f, be = 0.f, ga = 0.f;
#pragma unroll
        for (int q = 0; q < ROWS; ++q) {
          int row = gl + 4 * q;
          bool in = active && row < w;
          xa[q] = in ? ca[row] : 0.f;
          xb[q] = in ? cb[row] : 0.f;
          al += xa[q] * xa[q]; be += xb[q] * xb[q]; ga += xa[q] * xb[q];
        }
#pragma unroll
        for (int o = 2; o > 0; o >>= 1) {
          al += __shfl_xor_sync(0xffffffffu, al, o);
          be += __shfl_xor_sync(0xffffffffu, be, o);
          ga += __shfl_xor_sync(0xffffffffu, ga, o);
        }
        float g2 = ga * ga;
        float thr2 = fmaxf(1e-12f * al * be, abs2 * fminf(al, be));
        if (active && g2 > thr2 && g2 > 1e-37f) {
          // tan of the rotation angle: t = sign(d g) 2|g| / (|d| + sqrt(d^2 + 4 g^2)), d = |b|^2 - |a|^2
          float d = be - al;
          float t = __fdividef(2.f * ga, fabsf(d) + __fsqrt_rn(d * d + 4.f * g2));
          if (d < 0.f) t = -t;
          float c = rsqrtf(t * t + 1.f), sn = t * c;
#pragma unroll
          for (int q = 0; q < ROWS; ++q) {
            int row = gl + 4 * q;
            if (row < w) {
              ca[row] = c * xa[q] - sn * xb[q];
              cb[row] = sn * xa[q] + c * xb[q];
            }
          }
          rotated = 1;
        }
      }
      sub::named_barrier(1, nact);
    }
    if (rotated) *flag = 1;
    sub::named_barrier(1, nact);
    converged = *flag == 0;
    sub::named_barrier(1, nact);
    if (tid == 0) *flag = 0;
    sub::named_barrier(1, nact);
  }
  return converged;
}

// The same rotations for w <= 32 (the usual window), same pairs in the same order and the same sums in
// the same order, by one warp: two lanes per pair, the rows of a column dealt over them as the four
// partial sums above want it (lane h adds up the rows 4 q + h, then the rows 4 q + h + 2), so that one
// shuffle joins the sums and no barrier separates the rounds.  The search ends as soon as np - 1
// consecutive rounds (every pair once) have passed without a rotation, wherever in a sweep that
// happens.  A round is a chain of shared load, eight-term sums, shuffle, threshold and, where a pair
// rotates, two reciprocal roots and store: w = 32 took 640 cycles a round on two warps with a
// barrier per round, 485 with root, quotient and reciprocal root, 445 now (packed sums as well: 505, their chain is the longer).
__host__ __device__ __forceinline__ int ritz_row(int row) {      // place of a row inside its column
  return (row & 1) * 16 + (row & 2) * 4 + (row >> 2);
}
constexpr int kRitzLd32 = 36;            // column stride: the columns of neighbouring pairs hit distinct banks
// c_off: place of C in the kernel's shared memory (floats from the base).  Out of line: see the rehearsal in
// subspace_kernel.
__device__ __noinline__ bool jacobi_warp32(int c_off, int w, float s1, int max_sweeps) {
  float* C = reinterpret_cast<float*>(sub::pow_smem()) + c_off;
  const int lane = threadIdx.x & 31, g = lane >> 1, h = lane & 1;
  const int np = (w + 1) & ~1, half = np >> 1;
  const float abs2 = (2e-5f * s1) * (2e-5f * s1);
  if (w < 2) return true;
  const int limit = max_sweeps * (np - 1);
  int quiet = 0;                         // rounds since the last rotation
  // columns of this group's pair, one step of the round-robin further each round: ra runs upwards and rb
  // with it through 0 .. np - 2 (their sum is 2 round modulo np - 1), column np - 1 stays with group 0
  int ra = g, rb = g == 0 ? np - 1 : np - 1 - g;
  for (int it = 0; it < limit; ++it) {
    const int a = min(ra, rb), b = max(ra, rb);
    const bool active = g < half && b < w;
    float4* ca = reinterpret_cast<float4*>(C + (active ? a : 0) * kRitzLd32 + h * 16);
    float4* cb = reinterpret_cast<float4*>(C + (active ? b : 0) * kRitzLd32 + h * 16);
    float xa[16], xb[16];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const float4 u = ca[q], v = cb[q];
      xa[4 * q] = u.x; xa[4 * q + 1] = u.y; xa[4 * q + 2] = u.z; xa[4 * q + 3] = u.w;
      xb[4 * q] = v.x; xb[4 * q + 1] = v.y; xb[4 * q + 2] = v.z; xb[4 * q + 3] = v.w;
    }
    float al = 0.f, be = 0.f, ga = 0.f, al2 = 0.f, be2 = 0.f, ga2 = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      al += xa[q] * xa[q]; be += xb[q] * xb[q]; ga += xa[q] * xb[q];
      al2 += xa[q + 8] * xa[q + 8]; be2 += xb[q + 8] * xb[q + 8]; ga2 += xa[q + 8] * xb[q + 8];
    }
    al += al2; be += be2; ga += ga2;
    al += __shfl_xor_sync(0xffffffffu, al, 1);
    be += __shfl_xor_sync(0xffffffffu, be, 1);
    ga += __shfl_xor_sync(0xffffffffu, ga, 1);
    if (++ra == np - 1) ra = 0;
    if (g != 0 && ++rb == np - 1) rb = 0;
    const float g2 = ga * ga;
    const float thr2 = fmaxf(1e-12f * al * be, abs2 * fminf(al, be));
    const bool rotate = active && g2 > thr2 && g2 > 1e-37f;
    if (__any_sync(0xffffffffu, rotate)) {
      // with d = |b|^2 - |a|^2 and theta the smaller of the two angles that make the columns orthogonal:
      // cos 2 theta = |d| / sqrt(d^2 + 4 g^2), sin 2 theta = sign(d) 2 g / sqrt(d^2 + 4 g^2), then the half-angle formulas
      // (hardware reciprocal roots, a few units in the last place each: the rotation is orthogonal to float32
      // accuracy up to those, and the columns' lengths are taken again when the vectors are written)
      const float d = be - al;
      float ih, ic;
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ih) : "f"(fmaf(d, d, 4.f * g2)));
      const float c2 = ih > 0.f ? fmaf(0.5f * fabsf(d), ih, 0.5f) : 1.f;      // 0: the root is beyond the float32 range
      asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(ic) : "f"(c2));
      const float c = c2 * ic, sn = (d < 0.f ? -ga : ga) * ih * ic;
      if (rotate) {
        const f32x2 cc = pack2(c, c), ss = pack2(sn, sn), ns = pack2(-sn, -sn);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          float2 a01, a23, b01, b23;
          const f32x2 x0 = pack2(xa[4 * q], xa[4 * q + 1]), x1 = pack2(xa[4 * q + 2], xa[4 * q + 3]);
          const f32x2 y0 = pack2(xb[4 * q], xb[4 * q + 1]), y1 = pack2(xb[4 * q + 2], xb[4 * q + 3]);
          a01 = unpack2(fma2(ns, y0, mul2(cc, x0))); a23 = unpack2(fma2(ns, y1, mul2(cc, x1)));
          b01 = unpack2(fma2(cc, y0, mul2(ss, x0))); b23 = unpack2(fma2(cc, y1, mul2(ss, x1)));
          ca[q] = make_float4(a01.x, a01.y, a23.x, a23.y);
          cb[q] = make_float4(b01.x, b01.y, b23.x, b23.y);
        }
      }
      __syncwarp();
      quiet = 0;
    } else if (++quiet >= np - 1) {
      return true;
    }
  }
  return false;
}

// Column stride of the window factor in shared memory: >= w and congruent to 4 modulo 32, so that
// the eight 4-lane groups of a warp, which hold consecutive columns, hit distinct banks.
__host__ __device__ constexpr int ritz_ldc(int w) { return (w + 27) / 32 * 32 + 4; }
// Bytes of shared memory the Rayleigh-Ritz step takes for a window of w vectors.
__host__ __device__ constexpr size_t ritz_smem_bytes(int w) {
  return ((((size_t)w * ritz_ldc(w) + w + 1) & ~(size_t)1)) * sizeof(float) + cholesky_smem_bytes(w);
}

}  // namespace covspec
