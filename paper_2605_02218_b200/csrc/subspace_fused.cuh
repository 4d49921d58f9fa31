// The whole subspace iteration behind Eq. 14-15 in one persistent kernel.
//
// Work items are the 128-row tiles of the stage-2 requests (the same items and per-CTA lists as the
// power step had as a kernel of its own); every CTA walks its list once per multiplication by G.
// What used to be kernel boundaries are per-request counters in global memory:
//   arrive[b]   tiles of request b that have finished a step (their slab of the new block is in the
//               bf16 planes, their float64 partial Gram matrix is in `partial`); step k of a tile may
//               start loading the block once arrive[b] >= tiles(b) * k
//   factor[b]   number of triangular factors published for request b; the epilogue of step k needs
//               factor[b] >= k
//   ritz[b]     1 once the Rayleigh-Ritz vectors of the last block are published
//   last[b]     index of the request's last step: eig_iters on entry; the tile that factors step k
//               lowers it to k + 1 when the Ritz value estimates say that the energies will have
//               settled by then (see team_cholesky).  It only ever decreases and is written before
//               factor[b] = k + 1 is published: the epilogue of step k + 1, which waits for that
//               factor, reads "is this the last step?" with it, and the producer and MMA roles, which
//               only ask "is step s skipped?", can first be affected at step k + 2, whose start
//               every tile's arrival of step k + 1 precedes
//   summed[b]   CTAs of request b that have added up their slice of the partial Gram matrices of a
//               step (CTAs of request b, only when every CTA holds tiles of one request, see spread_sum)
// With SMs to spare the grid carries one more CTA per request that holds no tile and only factors for
// that request (n_servers); otherwise
// the tile that makes arrive[b] reach tiles(b) * (k + 1) (an atomic ticket; nobody waits for it to be
// a particular CTA) sums the partial Gram matrices in tile order and factors the sum right there: a
// Cholesky factorisation after the first steps, the Rayleigh-Ritz solve of the window next to the cut
// after the last one.  All CTAs are resident at the same time (cooperative launch, one CTA per SM),
// every wait is bounded and a CTA that gives up raises a global abort word that ends the others'
// waits too.  After the last step every CTA evaluates the energies (Eq. 15) of its own tiles.
//
// Data that crosses CTAs inside the kernel (partial sums, factors, Ritz vectors, the float32 window
// columns, the bf16 planes the last step re-reads) is read with L1-bypassing loads; the operand
// tiles of the bf16 planes are read by TMA, behind a proxy fence.
#pragma once
#include "eig_kernels.cuh"

namespace covspec {
namespace sub {

constexpr int kSyncStride = 8;           // unsigned words per request: arrive, factor, ritz, last, summed

struct FusedParams {
  const ReqPlan* plan;
  int batch;
  int n_items;              // row tiles over all stage-2 requests
  int tile_rows;            // rows of a tile: 128, or 64 (the MMA still computes 128 rows; the upper half is dropped)
  const int* sched;         // [gridDim.x + 1] offsets, the item lists of every CTA, [gridDim.x] place among the CTAs of the
                            // request: index | count << 16
  int steps;                // multiplications by G (eig_iters + 1, >= 2)
  float* lbuf;              // [batch][kLbufStride] triangular factor + reciprocal diagonal
  __nv_bfloat16* y_hi[2];   // plane buffers: step k reads [k & 1], writes [(k & 1) ^ 1]
  __nv_bfloat16* y_lo[2];
  int ld;
  float* yf[2];             // [sum M_b * kPMax], window columns only: the orthonormal basis Q of the block
                            // before the last multiplication, and the block after it (Eq. 15); the tile that
                            // starts at row i owns the floats from i * kPMax on, as [window column][row of the tile]
  double* partial;          // [tiles][kTileDoubles], see tile_offset
  float* ub;                // [batch][kPMax * kPMax] Ritz vectors of the discarded pairs
  float* energy;            // [sum M_b] (out)
  unsigned* sync;           // [batch][kSyncStride] counters (zero on entry), then the abort word
  int spread_sum;           // every CTA holds tiles of one request only: the CTAs of a request can add up the partial
                            // matrices together (the schedule then carries every CTA's place among them)
  int n_tile_ctas;          // CTAs that carry tiles: blockIdx.x < n_tile_ctas
  int n_servers;            // CTAs after those, one per stage-2 request, that only factor (0: the last tile to
                            // finish a step factors)
  int max_sweeps;
  float conv_tol;           // bound on the estimated energy error before NOCONVERGE is raised
  int early_stop;           // 1: requests whose estimate is far below conv_tol stop before `steps`
  int* status;
};

__device__ __forceinline__ unsigned ld_acquire_u32(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_u32(unsigned* p, unsigned v) {
  asm volatile("st.release.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
__device__ __forceinline__ void fence_proxy_async_all() {
  asm volatile("fence.proxy.async;" ::: "memory");
}

constexpr uint32_t kFlagSpinLimit = 1u << 21;       // polls of ~100 ns: gives up after a fraction of a second

// One thread waits until *ctr >= target.  Returns false when the limit expired (raises the global
// abort word) or another CTA gave up.
__device__ __forceinline__ bool flag_wait_ge(const unsigned* ctr, unsigned target, unsigned* gabort,
                                             volatile int* abort_flag) {
  for (uint32_t i = 0; i < kFlagSpinLimit; ++i) {
    if (ld_acquire_u32(ctr) >= target) return true;
    if ((i & 15u) == 15u && (ld_acquire_u32(gabort) != 0u || *abort_flag)) { *abort_flag = 1; return false; }
    __nanosleep(64);
  }
  *abort_flag = 1;
  atomicExch(gabort, 1u);
  return false;
}

// One thread decides whether step `step` (>= 1) of a request runs, and waits until it can: returns
// 1 when every tile has finished step - 1 (run; *last_out = the request's last step as known now),
// 0 when the request's last step is before `step` (skip), -1 when the wait was given up.  `last` is
// examined before `arrive`: after the request's final step arrive reaches the count the skipped
// next step would wait for.
__device__ __forceinline__ int step_decide(const unsigned* sync_b, unsigned nt, int step, unsigned* gabort,
                                           volatile int* abort_flag, int* last_out) {
  for (uint32_t i = 0; i < kFlagSpinLimit; ++i) {
    const unsigned arrived = ld_acquire_u32(sync_b);
    const int last = (int)ld_acquire_u32(sync_b + 3);
    if (last < step) return 0;
    if (arrived >= nt * (unsigned)step) { *last_out = last; return 1; }
    if ((i & 15u) == 15u && (ld_acquire_u32(gabort) != 0u || *abort_flag)) { *abort_flag = 1; return -1; }
    __nanosleep(64);
  }
  *abort_flag = 1;
  atomicExch(gabort, 1u);
  return -1;
}

// Layout of a partial Gram matrix in global memory: the 8 x 8 tiles of the lower triangle, tile
// (I, J <= I) at tri_index(I, J) * 64, row-major inside (diagonal tiles hold all 64 entries) - the
// layout the blocked factorisation works on, so that summing the tiles' partial matrices is an
// element-wise sum of contiguous arrays.
constexpr int kTileDoubles = (kPMax / 8) * (kPMax / 8 + 1) / 2 * 64;      // 13440
__device__ __forceinline__ int tile_offset(int i, int j) {                 // i >= j
  return tri_index(i >> 3, j >> 3) * 64 + (i & 7) * 8 + (j & 7);
}
// One entry summed over the tiles of a request in tile order (L1-bypassing loads, 8 in flight).
__device__ __forceinline__ double gram_entry_cg(int ntile, const double* src) {
  double s = 0.0;
  for (int t0 = 0; t0 < ntile; t0 += 8) {
    double v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = __ldcg(src + (size_t)min(t0 + q, ntile - 1) * kTileDoubles);
#pragma unroll
    for (int q = 0; q < 8; ++q) s += t0 + q < ntile ? v[q] : 0.0;
  }
  return s;
}
// T[0 .. count) = sum over the request's tiles (tile order: deterministic) of their partial
// matrices; count a multiple of 64.  Coalesced 16-byte loads, 32 of them in flight per thread.
__device__ __forceinline__ void team_sum_partials(double* T, const double* pbase, int ntile, int count,
                                                  int tid, int nthreads) {
  const int pairs = count >> 1;
  if (ntile == 1) {
    // one matrix (already summed, or a one-tile request): a plain copy, eight loads in flight per thread
    const double2* src = reinterpret_cast<const double2*>(pbase);
    for (int e0 = tid; e0 < pairs; e0 += 8 * nthreads) {
      double2 v[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) v[u] = __ldcg(src + min(e0 + u * nthreads, pairs - 1));
#pragma unroll
      for (int u = 0; u < 8; ++u)
        if (e0 + u * nthreads < pairs) reinterpret_cast<double2*>(T)[e0 + u * nthreads] = v[u];
    }
    return;
  }
  for (int e0 = tid; e0 < pairs; e0 += 4 * nthreads) {
    int e[4];
    double2 s[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      e[u] = e0 + u * nthreads < pairs ? e0 + u * nthreads : e0;
      s[u] = make_double2(0.0, 0.0);
    }
    for (int t0 = 0; t0 < ntile; t0 += 8) {
      double2 v[4][8];
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        const double2* src = reinterpret_cast<const double2*>(pbase + (size_t)min(t0 + q, ntile - 1) * kTileDoubles);
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u][q] = __ldcg(src + e[u]);
      }
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (t0 + q < ntile) {
#pragma unroll
          for (int u = 0; u < 4; ++u) { s[u].x += v[u][q].x; s[u].y += v[u][q].y; }
        }
      }
    }
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (e0 + u * nthreads < pairs) reinterpret_cast<double2*>(T)[e0 + u * nthreads] = s[u];
  }
}

// 1 / sqrt(x) for x > 0: float32 estimate of 1 / sqrt(x) refined in float32 and by one Newton step in
// float64.  kScale: x = m 4^k with m in [1, 4) first (integer operations on the exponent field) and the
// result scaled by 2^-k, for pivots beyond the float32 range; the result is the same, bit for bit, where
// both forms apply (every operation scales by a power of two).  Subnormal or non-finite x give a
// meaningless value; the caller clamps pivots to a positive floor.
template <bool kScale>
__device__ __forceinline__ double rsqrt_f64(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  const int k = kScale ? ((((hi >> 20) & 0x7ff) - 1023)) >> 1 : 0;
  const double m = kScale ? __hiloint2double(hi - (k << 21), lo) : x;
  const float xf = (float)m;
  float yf;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(yf) : "f"(xf));
  yf = yf * (1.5f - 0.5f * xf * yf * yf);
  double y = (double)yf;
  const double e = fma(-0.5 * m * y, y, 0.5);
  y = fma(y, e, y);
  return kScale ? __hiloint2double(__double2hiint(y) - (k << 20), __double2loint(y)) : y;
}

// Diagonal 8 x 8 tile, factored by one thread in registers: measured faster than a lane-per-row
// version (64-bit shuffles cost more than the arithmetic they save).  Two columns at a time: for the
// leading 2 x 2 block [[al, be], [be, ga]] the factor is l11 = sqrt(al), l21 = be / l11,
// l22 = sqrt(de / al) with de = al ga - be^2, so the two reciprocal square roots (of al and de) run
// side by side instead of one after the other.  The chain of dependent pivots is the critical path
// of the whole factorisation.  A pivot below 1e-12 of its original diagonal entry (a numerically
// dependent direction) is clamped there; the next multiplication by G restores the direction.  The
// tests for that, and for pivots whose reciprocal root needs the scaled form, stay off the chain:
// the roots are taken first and taken again where a test fails.
__device__ __forceinline__ void factor_diag_thread(double* D, const double* d0, double* rd) {
  double a[8][8], fl[8];
#pragma unroll
  for (int l = 0; l < 8; ++l) {
#pragma unroll
    for (int m = 0; m <= l; m += 2) {
      const double2 v = *reinterpret_cast<const double2*>(D + l * 8 + m);
      a[l][m] = v.x;
      if (m < l) a[l][m + 1] = v.y;
    }
    fl[l] = 1e-12 * d0[l];
  }
#pragma unroll
  for (int c = 0; c < 8; c += 2) {
    double al = a[c][c];
    const double be = a[c + 1][c], ga = a[c + 1][c + 1];
    double de = fma(al, ga, -be * be);                  // al * (second pivot)
    double ra = rsqrt_f64<false>(al), rq = rsqrt_f64<false>(de);
    // 2^-100 < al, de < 2^100 by the exponent fields (a negative value's field is out of range too)
    const unsigned ea = (unsigned)__double2hiint(al) - (923u << 20), ed = (unsigned)__double2hiint(de) - (923u << 20);
    if (!(al > fl[c]) || !(de > fl[c + 1] * al) || ea >= (200u << 20) || ed >= (200u << 20)) {
      if (!(al > fl[c])) al = fl[c] > 0.0 ? fl[c] : 1.0;
      de = fma(al, ga, -be * be);
      const double fd = fl[c + 1] * al;
      if (!(de > fd)) de = fd > 0.0 ? fd : al;
      ra = rsqrt_f64<true>(al);
      rq = rsqrt_f64<true>(de);
    }
    const double l11 = al * ra, l21 = be * ra, inv22 = rq * l11, l22 = de * rq * ra;
    a[c][c] = l11; a[c + 1][c] = l21; a[c + 1][c + 1] = l22;
    rd[c] = ra; rd[c + 1] = inv22;
#pragma unroll
    for (int l = c + 2; l < 8; ++l) {
      const double x1 = a[l][c] * ra;
      a[l][c + 1] = (a[l][c + 1] - x1 * l21) * inv22;
      a[l][c] = x1;
    }
#pragma unroll
    for (int l = c + 2; l < 8; ++l)
#pragma unroll
      for (int m = c + 2; m <= l; ++m) a[l][m] -= a[l][c] * a[m][c] + a[l][c + 1] * a[m][c + 1];
  }
#pragma unroll
  for (int l = 0; l < 8; ++l)
#pragma unroll
    for (int m = 0; m <= l; m += 2)
      if (m < l) *reinterpret_cast<double2*>(D + l * 8 + m) = make_double2(a[l][m], a[l][m + 1]);
      else D[l * 8 + m] = a[l][m];
}

constexpr int kEpiThreads = 256;         // warps 0-7

// What the kernel needs to know of a tile.  Every role looks its tiles up once per step; the search through the requests is a
// chain of loads that the acquiring loads of the counters send to L2 each time (64 requests: 3.3 k cycles a tile and step
// in the epilogue alone), so a CTA's first kCachedTiles tiles are looked up once per launch.
struct TileItem {
  int b, tile;              // request, tile of the request
  int m, p, r, win, presel_off, ptile_off;
};
constexpr int kCachedTiles = 16;
static_assert(8 * 8 + 8 * 4 + sizeof(TileItem) * kCachedTiles <= 1024, "barriers, single words and tiles lie in the last KB of the tail");

// The part behind the ring: the triangular factor, its reciprocal diagonal (a scratch array of p floats
// while a factor is being made), barriers, then single words.
struct PowTail {
  float *lt, *dinv;
  uint64_t* bars;
  uint32_t* tmem_slot;
  volatile int *abort_flag, *s_word;     // s_word: [2] broadcast slots of the epilogue
  int* s_flag;                           // Jacobi rotation flag
  float* s_scale;
  TileItem* tiles;                       // [kCachedTiles]
};
__device__ __forceinline__ PowTail pow_tail() {
  PowTail t;
  t.lt = reinterpret_cast<float*>(pow_smem() + kPowRegion);
  t.dinv = t.lt + kLtFloats;
  t.bars = reinterpret_cast<uint64_t*>(t.lt + kLbufStride);
  t.tmem_slot = reinterpret_cast<uint32_t*>(t.bars + 8);
  t.abort_flag = reinterpret_cast<volatile int*>(t.tmem_slot + 1);
  t.s_word = reinterpret_cast<volatile int*>(t.tmem_slot + 2);
  t.s_flag = reinterpret_cast<int*>(t.tmem_slot + 4);
  t.s_scale = reinterpret_cast<float*>(t.tmem_slot + 6);
  t.tiles = reinterpret_cast<TileItem*>(t.tmem_slot + 8);
  return t;
}

// float64 Gram matrix of the staged block (columns coff .. coff + 8 nb8 - 1, 16 nslab rows) on the FP64
// tensor cores, by the eight epilogue warps.  A warp takes 16 x 16 blocks of the lower triangle (dealt
// round-robin, `first` = the warp's place in the deal) and runs through all rows of a block before it
// starts the next: the four fragments of four rows (two per block row / column, one shared-memory word
// and one conversion per lane each) feed four instructions, so that nothing is staged and the warps
// never wait for one another.  Rows enter in ascending groups of four, whatever the split.  Bound by the
// FP64 pipe (16 cycles an instruction and scheduler): p = 144, 128 rows 68 -> 29 k cycles against
// float64 slabs in shared memory with a barrier every 16 rows; p = 48, 64 rows 12.5 -> 3 k.
constexpr int kEpiWarps = kEpiThreads / 32;
__device__ __forceinline__ void gram_tile_f64(const float* xs, int coff, int nb8, int nslab, int first, int lane,
                                              double* __restrict__ out) {
  const int fr = lane >> 2, fk = lane & 3;
  const int nb = (nb8 + 1) >> 1, nblk = nb * (nb + 1) / 2, t0 = coff >> 3;
  for (int q = first; q < nblk; q += kEpiWarps) {
    int bi, bj;
    tri_decode(q, bi, bj);
    // an odd number of tiles leaves half of the last block row unused: its reads are turned to the first half
    const bool hi_i = 2 * bi + 1 < nb8, hi_j = 2 * bj + 1 < nb8, off_diag = bi != bj;
    const float* a0 = xs + (size_t)(coff + bi * 16 + fr) * kXsLd + fk;
    const float* b0 = xs + (size_t)(coff + bj * 16 + fr) * kXsLd + fk;
    const float* a1 = a0 + (hi_i ? 8 * kXsLd : 0);
    const float* b1 = b0 + (hi_j ? 8 * kXsLd : 0);
    double c00[2] = {0.0, 0.0}, c10[2] = {0.0, 0.0}, c11[2] = {0.0, 0.0}, c01[2] = {0.0, 0.0};
    for (int sl = 0; sl < nslab; ++sl) {
#pragma unroll
      for (int ks = 0; ks < kSlabRows / 4; ++ks) {
        const int o = sl * kSlabRows + 4 * ks;
        const double x0 = (double)a0[o], x1 = (double)a1[o], y0 = (double)b0[o], y1 = (double)b1[o];
        dmma_8x8x4(c00[0], c00[1], x0, y0);
        if (hi_i) {
          dmma_8x8x4(c10[0], c10[1], x1, y0);
          dmma_8x8x4(c11[0], c11[1], x1, y1);
        }
        if (off_diag) dmma_8x8x4(c01[0], c01[1], x0, y1);
      }
    }
    auto put = [&](int I, int J, const double (&c)[2]) {
      *reinterpret_cast<double2*>(out + tri_index(t0 + I, t0 + J) * 64 + fr * 8 + 2 * fk) = make_double2(c[0], c[1]);
    };
    put(2 * bi, 2 * bj, c00);
    if (hi_i) { put(2 * bi + 1, 2 * bj, c10); put(2 * bi + 1, 2 * bj + 1, c11); }
    if (off_diag) put(2 * bi, 2 * bj + 1, c01);
  }
}

template <int N> struct IntTag { static constexpr int value = N; };

// Blocked right-looking Cholesky factorisation in float64 by the eight epilogue warps.  The matrix is
// already in shared memory, t_off doubles behind the base (tile layout, see tile_offset; 16-byte
// aligned), followed by room for 16 nb doubles (original diagonal, reciprocal pivots); entries beyond n
// inside the last row of tiles are replaced by the identity here.  out != nullptr: the factor goes to
// global memory in the layout the triangular solve reads (see lt_row_offset) with the reciprocal
// diagonal behind it, panel by panel while the later ones are factored.  One function for the
// factor and for the Rayleigh-Ritz window, kept out of line: code that runs once per launch is fetched
// from L2, and the window's factorisation finds this code where the steps before it left it.
__device__ __noinline__ void cholesky_team(int n, int t_off, float* out) {
  double* T = reinterpret_cast<double*>(pow_smem()) + t_off;
  const int tid = threadIdx.x, lane = tid & 31, warp = warp_index();
  auto sync = [&]() { named_barrier(1, kEpiThreads); };
  const int nb = (n + 7) >> 3;
  double* aux = T + nb * (nb + 1) / 2 * 64;
  double* d0 = aux;                 // original diagonal
  double* rd = aux + 8 * nb;        // 1 / L[j][j]
  // identity padding of rows / columns n .. 8 nb - 1 (last row of tiles), then the diagonal
  for (int e = tid; e < nb * 64; e += kEpiThreads) {
    const int J = e >> 6, i = 8 * (nb - 1) + ((e >> 3) & 7), j = 8 * J + (e & 7);
    if (i >= n || j >= n) T[tri_index(nb - 1, J) * 64 + (e & 63)] = (i == j) ? 1.0 : 0.0;
  }
  sync();
  for (int i = tid; i < 8 * nb; i += kEpiThreads) d0[i] = T[tile_offset(i, i)];
  sync();
  const int fr = lane >> 2, fk = lane & 3;
  auto update_tile = [&](int J, int I, int K) {
    const double* XI = T + tri_index(I, J) * 64 + fr * 8 + fk;
    const double* XK = T + tri_index(K, J) * 64 + fr * 8 + fk;
    double* C = T + tri_index(I, K) * 64 + fr * 8 + 2 * fk;
    double c0 = C[0], c1 = C[1];
    dmma_8x8x4(c0, c1, -XI[0], XK[0]);
    dmma_8x8x4(c0, c1, -XI[4], XK[4]);
    C[0] = c0; C[1] = c1;
  };
  // row `i` of the tile (I, J) <- row * L_JJ^-T (forward substitution over the 8 columns)
  auto solve_row = [&](int J, int i, double (&x)[8]) {
    const double2* D = reinterpret_cast<const double2*>(T + tri_index(J, J) * 64);
    double2* row = reinterpret_cast<double2*>(T + tri_index(i >> 3, J) * 64 + (i & 7) * 8);
    double r[8];
#pragma unroll
    for (int c = 0; c < 4; ++c) {
      const double2 v = row[c], q = reinterpret_cast<const double2*>(rd + 8 * J)[c];
      x[2 * c] = v.x; x[2 * c + 1] = v.y;
      r[2 * c] = q.x; r[2 * c + 1] = q.y;
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) {
      double v = x[c];
#pragma unroll
      for (int k = 0; k < c; k += 2) {
        const double2 l = D[c * 4 + (k >> 1)];
        v -= x[k] * l.x;
        if (k + 1 < c) v -= x[k + 1] * l.y;
      }
      x[c] = v * r[c];
    }
#pragma unroll
    for (int c = 0; c < 4; ++c) row[c] = make_double2(x[2 * c], x[2 * c + 1]);
  };
  // NT tiles (I, K), (I + step, K), ... -= sum over the panels 0 .. J of X_I X_K^T, accumulators in registers
  auto accumulate = [&](auto nt_tag, int J, int I, int step, int K) {
    constexpr int NT = decltype(nt_tag)::value;
    double c[NT][2];
#pragma unroll
    for (int u = 0; u < NT; ++u) {
      const double2 v = *reinterpret_cast<const double2*>(T + tri_index(I + u * step, K) * 64 + fr * 8 + 2 * fk);
      c[u][0] = v.x; c[u][1] = v.y;
    }
    const double* XK = T + tri_index(K, 0) * 64 + fr * 8 + fk;
    const double* XI = T + tri_index(I, 0) * 64 + fr * 8 + fk;
    int skip[NT];                                        // from tile (I, .) to tile (I + u step, .)
#pragma unroll
    for (int u = 0; u < NT; ++u) skip[u] = (tri_index(I + u * step, 0) - tri_index(I, 0)) * 64;
    double k0[2], k4[2], x0[2][NT], x4[2][NT];           // fragments of two panels: one in flight, one in use
    auto load = [&](int buf) {
      k0[buf] = XK[0]; k4[buf] = XK[4];
#pragma unroll
      for (int u = 0; u < NT; ++u) { x0[buf][u] = XI[skip[u]]; x4[buf][u] = XI[skip[u] + 4]; }
      XK += 64; XI += 64;
    };
    auto apply = [&](int buf) {
#pragma unroll
      for (int u = 0; u < NT; ++u) dmma_8x8x4(c[u][0], c[u][1], -x0[buf][u], k0[buf]);
#pragma unroll
      for (int u = 0; u < NT; ++u) dmma_8x8x4(c[u][0], c[u][1], -x4[buf][u], k4[buf]);
    };
    load(0);
#pragma unroll 1
    for (int q = 0; q <= J; q += 2) {                    // (the loads beyond panel J stay inside the matrix)
      load(1);
      apply(0);
      if (q + 1 > J) break;
      load(0);
      apply(1);
    }
#pragma unroll
    for (int u = 0; u < NT; ++u)
      *reinterpret_cast<double2*>(T + tri_index(I + u * step, K) * 64 + fr * 8 + 2 * fk) = make_double2(c[u][0], c[u][1]);
  };
  // Factor entries in the layout of the triangular solve (row j holds L[i][j] for i >= (j & ~3)): the
  // tiles (J, J) and (J + 1, J) with the reciprocal diagonal by one warp, the rows below by the threads
  // that solved them (consecutive rows, so a column is one coalesced store).
  const int P8 = nb * 8;
  auto column = [&](int j) { return out + lt_row_offset(j, P8) - (j & ~3); };
  auto store_tiles = [&](int J) {
    const int jl = lane >> 2, j = 8 * J + jl;
    if (j >= n) return;
    float* dst = column(j);
    for (int I = J; I < min(J + 2, nb); ++I)
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int i0 = (lane & 3) * 2 + q, i = 8 * I + i0;
        if (i >= j && i < n) dst[i] = (float)T[tri_index(I, J) * 64 + i0 * 8 + jl];
      }
    if ((lane & 3) == 0) out[kLtFloats + j] = (float)rd[j];
  };
  auto store_row = [&](int J, int i, const double (&x)[8]) {
    if (i >= n) return;
#pragma unroll
    for (int c = 0; c < 8; ++c) column(8 * J + c)[i] = (float)x[c];
  };
  if (tid == 0) factor_diag_thread(T, d0, rd);
  sync();
  // One barrier of the whole team per 8-column panel.  The chain that bounds the factorisation -
  // panel J's diagonal tile -> tile (J+1, J) -> its update of tile (J+1, J+1) -> that tile's eight
  // dependent pivots - runs on warp 0 alone; the warps of the other three schedulers (the FP64 pipe
  // is per scheduler: warp w issues on scheduler w & 3, so warp 4 stays idle) meanwhile solve the rest of
  // panel J and bring the columns J+1 and J+2 up to date.  They look two columns ahead: column J+2 takes
  // its contributions of all panels up to J in one go, with the tile in registers, and column J+1 only
  // that of panel J (it had the others an iteration before).  Updating the whole trailing matrix after
  // every panel, every tile through shared memory, made the first half of the panels wait for it
  // (n = 144: 80-100 k cycles); now every panel takes what its pivot chain takes.  The bulk warps need
  // tile (J+1, J) for column J+1: warp 0 arrives on barrier 4 once it is solved.
  const bool bulk = (warp & 3) != 0;
  const int me = warp - (warp >> 2) - 1;                                     // bulk warps, in order
  constexpr int nbulk = kEpiWarps - (kEpiWarps + 3) / 4, bulk_threads = nbulk * 32;
  const int btid = me * 32 + lane;
  for (int J = 0; J + 1 < nb; ++J) {
    if (warp == 0) {
      double x[8];
      if (lane < 8) solve_row(J, 8 * (J + 1) + lane, x);
      __syncwarp();
      asm volatile("bar.arrive 4, %0;" ::"r"(bulk_threads + 32) : "memory");
      update_tile(J, J + 1, J + 1);
      __syncwarp();
      if (lane == 0) factor_diag_thread(T + tri_index(J + 1, J + 1) * 64, d0 + 8 * (J + 1), rd + 8 * (J + 1));
      __syncwarp();
    } else if (bulk) {
      const int i = 8 * (J + 2) + btid;              // at most 18 tiles below: fewer rows than bulk threads
      double x[8];
      if (i < 8 * nb) solve_row(J, i, x);
      asm volatile("bar.sync 4, %0;" ::"r"(bulk_threads + 32) : "memory");
      if (out != nullptr && i < 8 * nb) store_row(J, i, x);
      for (int I = J + 2 + me; I < nb; I += nbulk) update_tile(J, I, J + 1);
      // column J + 2: the tiles are dealt from the other end, so that the warps with one tile less
      // above come first here
      for (int I = J + 2 + (nbulk - 1 - me); I < nb; I += 3 * nbulk) {
        if (I + 2 * nbulk < nb) accumulate(IntTag<3>{}, J, I, nbulk, J + 2);
        else if (I + nbulk < nb) accumulate(IntTag<2>{}, J, I, nbulk, J + 2);
        else accumulate(IntTag<1>{}, J, I, nbulk, J + 2);
      }
    } else if (out != nullptr && warp == 4 && J >= 1) {
      store_tiles(J - 1);                        // final since the last barrier
    }
    sync();
  }
  if (out != nullptr) {
    if (nb >= 2 && warp == 1) store_tiles(nb - 2);
    if (warp == 2) store_tiles(nb - 1);
  }
}

// ---- work of the tile that finishes a step last (all 256 epilogue threads) ----------------------
// Kept out of line: the tile epilogue is register-bound, and these run once per request and step.

// Cholesky factor of the summed Gram matrix, written in the layout the triangular solve reads
// (see lt_row_offset) followed by the reciprocal diagonal.  Uses the operand ring as scratch.
// Returns (to every thread) whether the next step may be the last one: from the diagonal of
// the summed Gram matrix B = Y'^T Y' (theta_i = sqrt(B_ii) estimates the i-th eigenvalue of G once the
// basis has started to order itself) the energy error after q_final multiplications is predicted as
// max_i 2 (theta_i / theta_1) (theta_min / theta_i)^q_final over the kept directions i < r that the
// cut can tell apart from the discarded ones (theta_i - theta_min > 1e-3 theta_1), the estimate
// team_ritz reports at the end; stop_below is the bound it has to stay under (0: never stop early).
// pad: also write the entries of the layout that no factor touches (the first factorisation of a
// launch does; they stay as they are for the later ones).
__device__ __noinline__ bool team_cholesky(const double* pbase, int nt, int p, int r, float* out, int q_final,
                                           float stop_below, bool pad) {
  double* Tm = reinterpret_cast<double*>(pow_smem());
  float* dg = pow_tail().dinv;
  volatile int* s_word = pow_tail().s_word;
  const int et = threadIdx.x, warp = warp_index(), lane = et & 31;
  const int P = (p + 7) & ~7, nb = (p + 7) >> 3;
  auto epi_sync = [&]() { named_barrier(1, kEpiThreads); };
  // identity padding of the layout rows / columns p .. P-1 and the entries left of the diagonal
  for (int i = warp; pad && i < P; i += 8) {
    int j0 = i & ~3;
    float* row = out + lt_row_offset(i, P) - j0;
    for (int j = j0 + lane; j < P; j += 32)
      if (j < i || i >= p || j >= p) row[j] = (i == j) ? 1.f : 0.f;
  }
  for (int j = p + et; pad && j < P; j += kEpiThreads) out[kLtFloats + j] = 1.f;
  team_sum_partials(Tm, pbase, nt, nb * (nb + 1) / 2 * 64, et, kEpiThreads);
  epi_sync();
  if (stop_below > 0.f) {
    for (int i = et; i < p; i += kEpiThreads) dg[i] = sqrtf(fmaxf((float)Tm[tile_offset(i, i)], 0.f));
    if (et == 0) *s_word = 0;
    epi_sync();
    if (warp == 0) {
      float tmin = 3.0e38f, tmax = 0.f;
      for (int i = lane; i < p; i += 32) { tmin = fminf(tmin, dg[i]); tmax = fmaxf(tmax, dg[i]); }
      tmin = warp_min(tmin); tmax = warp_max(tmax);
      float worst = 0.f;
      for (int i = lane; i < r; i += 32) {
        float th = dg[i];
        if (th - tmin > 1e-3f * tmax && th > 0.f) worst = fmaxf(worst, 2.f * (th / tmax) * __powf(tmin / th, (float)q_final));
      }
      worst = warp_max(worst);
      if (lane == 0 && tmax > 0.f && worst < stop_below) *s_word = 1;
    }
    epi_sync();
  }
  const bool stop = stop_below > 0.f && *s_word != 0;
  cholesky_team(p, 0, out);
  return stop;
}

// Rayleigh-Ritz on the window next to the cut (see eig_kernels.cuh) and the convergence estimate.
// Uses the operand ring and the factor's place behind it as scratch: the window factor C, the float64 window block
// and its two diagonals end before the reciprocal diagonal, which serves as `dg`, for every window.  (At the
// start of the factor's place `dg` lay inside the float64 block of windows of 136 and more.)
static_assert(ritz_smem_bytes(kPMax) + 16 <= kPowRegion + kLtFloats * sizeof(float), "scratch of team_ritz");
__device__ __noinline__ void team_ritz(const double* pbase, int nt, int p, int w, int r, int m, float* out_u,
                                       int max_sweeps, float conv_tol, int steps, int* status) {
  float* C = reinterpret_cast<float*>(pow_smem());
  float* dg = pow_tail().dinv;
  float* s_scale = pow_tail().s_scale;
  int* s_flag = pow_tail().s_flag;
  const int et = threadIdx.x, warp = warp_index(), lane = et & 31;
  auto epi_sync = [&]() { named_barrier(1, kEpiThreads); };
  const int w0 = p - w, nbot = p - r;
  const bool small = w <= 32;            // the usual window: see jacobi_warp32 for the row order of a column
  const int ldc = small ? kRitzLd32 : ritz_ldc(w);
  auto at = [&](int col, int row) { return col * ldc + (small ? ritz_row(row) : row); };
  float* sig = C + (size_t)w * ldc;
  for (int e = et; e < w * ldc; e += kEpiThreads) C[e] = 0.f;
  if (et == 0) *s_scale = 0.f;
  epi_sync();
  {
    float mx = 0.f;
    for (int i = et; i < p; i += kEpiThreads) {
      float v = (float)gram_entry_cg(nt, pbase + tile_offset(i, i));
      dg[i] = sqrtf(fmaxf(v, 0.f));                      // sqrt of the diagonal of B'
      mx = fmaxf(mx, v);
    }
    mx = warp_max(mx);
    if (lane == 0 && mx > 0.f) atomicMax(reinterpret_cast<int*>(s_scale), __float_as_int(mx));
  }
  {
    // the window block of B' (rows / columns w0 .. p-1), gathered into a tile layout of its own
    const int nbw = (w + 7) >> 3, cnt = nbw * (nbw + 1) / 2 * 64;
    const int tw_off = (w * ldc + w + 3) / 4 * 2;          // doubles from the base, a multiple of two
    double* Tw = reinterpret_cast<double*>(C) + tw_off;
    for (int e = et; e < cnt; e += kEpiThreads) {
      int I, J;
      tri_decode(e >> 6, I, J);
      int i = 8 * I + ((e >> 3) & 7), j = 8 * J + (e & 7);
      double v = 0.0;
      if (i < w && j < w) v = gram_entry_cg(nt, pbase + tile_offset(w0 + max(i, j), w0 + min(i, j)));
      Tw[e] = v;
    }
    epi_sync();
    cholesky_team(w, tw_off, nullptr);
    epi_sync();
    for (int e = et; e < cnt; e += kEpiThreads) {
      int I, J;
      tri_decode(e >> 6, I, J);
      const int i = 8 * I + ((e >> 3) & 7), j = 8 * J + (e & 7);
      if (i < w && j <= i) C[at(j, i)] = (float)Tw[e];
    }
  }
  epi_sync();
  const float s1 = sqrtf(*s_scale);
  // `first` .. : the threads that look at the estimate
  auto settled = [&](int first, int count) {
    if (!(conv_tol > 0.f) || p >= m) return;
    // Has the iteration settled?  The basis vectors converge to eigenvectors in order, so
    // theta_k ~ sqrt(B'_kk) estimates the k-th eigenvalue of G and theta_min the first one left
    // out of the basis.  After q multiplications a kept direction k still carries about
    // (theta_min / theta_k)^q of the directions outside the basis, which moves the energies by
    // about 2 theta_k (theta_min / theta_k)^q; relative to the scale theta_1 of the energies, and
    // only for directions that the cut can tell apart from the discarded ones (more than
    // 1e-3 theta_1 above theta_min; closer ones may mix freely, Eq. 15 is not unique there).
    float tmin = 3.0e38f;
    for (int i = lane; i < p; i += 32) tmin = fminf(tmin, dg[i]);
    tmin = warp_min(tmin);
    float worst = 0.f;
    for (int i = et - first; i < r; i += count) {
      float th = dg[i];
      if (th - tmin > 1e-3f * s1 && th > 0.f)
        worst = fmaxf(worst, 2.f * (th / s1) * __powf(tmin / th, (float)steps));
    }
    worst = warp_max(worst);
    if (lane == 0 && worst > conv_tol) atomicOr(status, kStatusNoConverge);
  };
  const int nact = small ? 32 : min(kEpiThreads, ((((w + 1) >> 1) * 4) + 31) & ~31);
  if (et == 0) *s_flag = 0;
  epi_sync();
  if (et < nact) {
    bool converged;
    if (small) converged = jacobi_warp32(0, w, s1, max_sweeps);
    else if (w <= 64) converged = jacobi_sweeps<16>(C, ldc, w, s1, max_sweeps, nact, s_flag);
    else if (w <= 96) converged = jacobi_sweeps<24>(C, ldc, w, s1, max_sweeps, nact, s_flag);
    else converged = jacobi_sweeps<(kPMax + 3) / 4>(C, ldc, w, s1, max_sweeps, nact, s_flag);
    if (!converged && et == 0) atomicOr(status, kStatusNoConverge);
    if (!small) settled(0, nact);
  } else if (small) {
    settled(32, kEpiThreads - 32);               // beside the rotations, which are one warp's
  }
  named_barrier(3, kEpiThreads);
  for (int k = warp; k < w; k += 8) {
    float sm = 0.f;
    for (int row = lane; row < w; row += 32) { float x = C[at(k, row)]; sm += x * x; }
    sm = warp_sum(sm);
    if (lane == 0) sig[k] = sqrtf(sm);
  }
  epi_sync();
  // rank the columns by singular value (ascending, ties by larger index first); the nbot smallest
  // become unit vectors out_u[j * nbot + rank]
  for (int k = warp; k < w; k += 8) {
    float sk = sig[k];
    int rank = 0;
    for (int q = lane; q < w; q += 32) {
      float sq = sig[q];
      rank += (sq < sk) || (sq == sk && q > k);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
    if (rank < nbot) {
      float scale = sk > 0.f ? 1.f / sk : 0.f;
      for (int j = lane; j < w; j += 32) out_u[j * nbot + rank] = C[at(k, j)] * scale;
    }
  }
}

__global__ void __launch_bounds__(kPowThreads, 1)
subspace_kernel(const __grid_constant__ CUtensorMap map_gh, const __grid_constant__ CUtensorMap map_gl,
                const __grid_constant__ CUtensorMap map_y0h, const __grid_constant__ CUtensorMap map_y0l,
                const __grid_constant__ CUtensorMap map_y1h, const __grid_constant__ CUtensorMap map_y1l,
                const FusedParams prm) {
  uint8_t* smem = pow_smem();
  float* xs = reinterpret_cast<float*>(smem);                       // aliases the ring after the MMAs
  float* xq = reinterpret_cast<float*>(smem + kXsBytes);            // previous block (last step)
  const PowTail tail = pow_tail();
  float *lt = tail.lt, *dinv = tail.dinv;
  uint64_t* full = tail.bars;            // [2]
  uint64_t* empty = tail.bars + 2;       // [2]
  uint64_t* acc_full = tail.bars + 4;
  uint64_t* acc_empty = tail.bars + 5;
  uint64_t* epi_done = tail.bars + 6;    // the region no longer belongs to the epilogue
  uint32_t* tmem_slot = tail.tmem_slot;
  volatile int* abort_flag = tail.abort_flag;
  volatile int* s_word = tail.s_word;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  unsigned* gabort = prm.sync + (size_t)prm.batch * kSyncStride;

  if (threadIdx.x == 0) {
    for (int s = 0; s < kPowStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 128);
    mbar_init(epi_done, kEpiThreads);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  const int s_begin = prm.sched[blockIdx.x], s_end = prm.sched[blockIdx.x + 1];
  const int* s_items = prm.sched + gridDim.x + 1;
  const int my_group = prm.sched[gridDim.x + 1 + prm.n_items + blockIdx.x] & 0xffff;
  const int n_groups = prm.sched[gridDim.x + 1 + prm.n_items + blockIdx.x] >> 16;
  const int last_step = prm.steps - 1;
  const int R = prm.tile_rows;
  auto look_up = [&](int item) {
    const int b = find_request(item, prm.batch, [&](int q) { return prm.plan[q].ptile_off; });
    const ReqPlan& rp = prm.plan[b];
    return TileItem{b, item - rp.ptile_off, rp.m, rp.p, rp.r, rp.win, rp.presel_off, rp.ptile_off};
  };
  if (threadIdx.x < min(kCachedTiles, s_end - s_begin)) tail.tiles[threadIdx.x] = look_up(s_items[s_begin + threadIdx.x]);
  if (warp == 9) tmem_alloc(tmem_slot, kPowTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // the CTA's si-th tile
  auto tile_at = [&](int si) { return si - s_begin < kCachedTiles ? tail.tiles[si - s_begin] : look_up(s_items[si]); };

  // request of the factor server with this index: the index-th one that has a stage 2
  auto server_request = [&](int index) -> int {
    for (int q = 0; q < prm.batch; ++q)
      if (prm.plan[q].stage2 && index-- == 0) return q;
    return -1;
  };

  if (warp == 8) {
    // ------------------------------------------------------------ TMA producer
    if (lane == 0) {
      uint32_t it = 0, n = 0;
      bool ok = true;
      for (int step = 0; step <= last_step && ok; ++step) {
        const CUtensorMap* myh = (step & 1) ? &map_y1h : &map_y0h;
        const CUtensorMap* myl = (step & 1) ? &map_y1l : &map_y0l;
        for (int si = s_begin; si < s_end && ok; ++si, ++n) {
          const TileItem rp = tile_at(si);
          const int b = rp.b;
          if (step > 0) {
            // every tile of the request has written its slab of the block this step multiplies,
            // unless the request has already had its last step
            const unsigned nt = (unsigned)((rp.m + R - 1) / R);
            int last_b;
            const int go = step_decide(prm.sync + (size_t)b * kSyncStride, nt, step, gabort, abort_flag, &last_b);
            if (go < 0) { ok = false; break; }
            if (go == 0) { --n; continue; }
            fence_proxy_async_all();
          }
          // the previous item's staged block (and whatever its last tile factored) lives in the
          // ring until its epilogue is done
          if (n > 0 && !(ok = mbar_wait(epi_done, (n - 1) & 1u, abort_flag))) break;
          int k_chunks = (rp.m + kBK - 1) / kBK;
          for (int kc = 0; kc < k_chunks; ++kc, ++it) {
            int s = it % kPowStages;
            if (!(ok = mbar_wait(&empty[s], ((it / kPowStages) & 1u) ^ 1u, abort_flag))) break;
            mbar_expect_tx(&full[s], kPowStageBytes);
            uint32_t dst = smem_u32(smem + s * kPowStageBytes);
            int grow = rp.presel_off + rp.tile * R;
            tma_load_2d(dst, &map_gh, kc * kBK, grow, &full[s]);
            tma_load_2d(dst + kPowBytesA, &map_gl, kc * kBK, grow, &full[s]);
            tma_load_2d(dst + 2 * kPowBytesA, myh, kc * kBK, b * kPMax, &full[s]);
            tma_load_2d(dst + 2 * kPowBytesA + kPowBytesB, myl, kc * kBK, b * kPMax, &full[s]);
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 9 && prm.n_servers > 0 && (int)blockIdx.x >= prm.n_tile_ctas) {
    // ------------------------------------------------------------ rehearsal (factor servers)
    // A server has nothing to multiply.  While it waits for the tiles this warp runs the eigenvalue
    // rotations of the Ritz window once on a made-up matrix, in the part of the ring that the team
    // does not use: the code is then in the SM's instruction cache when the last step needs it, instead of
    // being fetched line by line from L2 in the middle of the request's critical path.  Nothing orders the team behind
    // this warp, so the place must be one that no phase of the team's work reaches: the factorisation and windows of
    // up to 32 end below it; wider windows do not take this code.
    constexpr int kOff = (kPowRegion - 32 * kRitzLd32 * 4) / 4;
    static_assert(cholesky_smem_bytes(kPMax) <= kOff * 4 && ritz_smem_bytes(32) <= kOff * 4, "place of the rehearsal");
    const int served = server_request((int)blockIdx.x - prm.n_tile_ctas);
    if (served >= 0 && prm.plan[served].win <= 32) {
      float* C = reinterpret_cast<float*>(smem) + kOff;
      for (int e = lane; e < 32 * kRitzLd32; e += 32) C[e] = 0.f;
      __syncwarp();
      C[lane * kRitzLd32 + ritz_row(lane)] = 1.f;
      if (lane == 0) C[ritz_row(1)] = 0.5f;
      __syncwarp();
      jacobi_warp32(kOff, 32, 1.f, 1);
    }
  } else if (warp == 9) {
    // ------------------------------------------------------------ MMA issuer
    if (lane == 0) {
      uint32_t it = 0, n = 0;
      bool ok = true;
      for (int step = 0; step <= last_step && ok; ++step) {
        for (int si = s_begin; si < s_end && ok; ++si, ++n) {
          const TileItem rp = tile_at(si);
          const int b = rp.b;
          const uint32_t idesc = umma_idesc(kTile, (rp.p + 15) & ~15);
          if (step > 0) {
            const unsigned nt = (unsigned)((rp.m + R - 1) / R);
            int last_b;
            const int go = step_decide(prm.sync + (size_t)b * kSyncStride, nt, step, gabort, abort_flag, &last_b);
            if (go < 0) { ok = false; break; }
            if (go == 0) { --n; continue; }
          }
          if (!(ok = mbar_wait(acc_empty, (n & 1u) ^ 1u, abort_flag))) break;
          tc_fence_after();
          int k_chunks = (rp.m + kBK - 1) / kBK;
          bool ready = false;
          for (int kc = 0; kc < k_chunks; ++kc, ++it) {
            int s = it % kPowStages;
            if (!ready && !(ok = mbar_wait(&full[s], (it / kPowStages) & 1u, abort_flag))) break;
            tc_fence_after();
            uint32_t base = smem_u32(smem + s * kPowStageBytes);
            ready = kc + 1 < k_chunks && mbar_peek(&full[(it + 1) % kPowStages], ((it + 1) / kPowStages) & 1u);
            // T += G_hi Y_hi + G_lo Y_hi + G_hi Y_lo
#pragma unroll
            for (int term = 0; term < 3; ++term) {
              uint64_t adesc = umma_desc(base + (term == 1 ? kPowBytesA : 0));
              uint64_t bdesc = umma_desc(base + 2 * kPowBytesA + (term == 2 ? kPowBytesB : 0));
#pragma unroll
              for (int k = 0; k < kBK / 16; ++k)
                umma_bf16(tmem_base, adesc + 2 * k, bdesc + 2 * k, idesc, (kc | term | k) != 0);
            }
            umma_commit(&empty[s]);
          }
          if (!ok) break;
          umma_commit(acc_full);
        }
      }
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue, warps 0-7
    const int et = threadIdx.x;                    // 0 .. 255
    const int r = (warp & 3) * 32 + lane;          // TMEM lane = row of the tile (warps 0-3 solve)
    const uint32_t t_lane = tmem_base + ((uint32_t)((warp & 3) * 32) << 16);
    auto epi_sync = [&]() { named_barrier(1, kEpiThreads); };
    // thread 0 waits for a counter; everybody learns the outcome
    auto team_wait = [&](const unsigned* ctr, unsigned target) -> bool {
      epi_sync();
      if (et == 0) *s_word = flag_wait_ge(ctr, target, gabort, abort_flag) ? 1 : 0;
      epi_sync();
      return *s_word != 0;
    };
    // Do the CTAs of a request with nt tiles add up its partial matrices slice by slice?  One CTA reads
    // about 64 bytes a cycle, the two more rounds through L2 that sharing takes cost 5-6 k cycles: worth it
    // from 48 k entries over all tiles on (12 tiles at p = 88, 5 at p = 144), and only if there is somebody
    // to share with (a server's request has one CTA per tile).
    auto spread_of = [&](int nt, int P) {
      return prm.spread_sum && nt * ((P >> 3) * ((P >> 3) + 1) / 2 * 64) > 48000 && (prm.n_servers > 0 || n_groups > 1);
    };
    uint32_t n = 0;
    int cached_b = -1, cached_step = -1;
    bool ok = true;
    // Factors the summed Gram matrix of request b after step `step` (Cholesky, or the Rayleigh-Ritz
    // solve after the last step) and publishes the result; returns whether the next step was
    // declared the last one.  Uses the operand ring as scratch.
    auto factor_request = [&](int b, const auto& rp, unsigned* sync_b, int step, bool is_last, int last_b,
                              int nt_sum) -> bool {
      const int p = rp.p;
      const double* pbase = prm.partial + (size_t)rp.ptile_off * kTileDoubles;
      bool stop = false;
      if (!is_last) {
        // after the second multiplication and later: may the next step be the last one?  (asked with a
        // margin of 8 under the tolerance, 64 at the first opportunity: the estimate is rough while
        // the basis is still mixing)
        const bool may_stop = prm.early_stop && step >= 1 && step + 1 < last_b && p < rp.m;
        const float margin = step == 1 ? 0.015625f : 0.125f;
        stop = team_cholesky(pbase, nt_sum, p, rp.r, prm.lbuf + (size_t)b * kLbufStride, step + 2,
                             may_stop ? margin * prm.conv_tol : 0.f, step == 0);
        epi_sync();                                // then one fence for the team's stores (it is cumulative)
        if (et == 0) {
          __threadfence();
          if (stop) st_release_u32(sync_b + 3, (unsigned)(step + 1));
          st_release_u32(sync_b + 1, (unsigned)(step + 1));
        }
      } else {
        team_ritz(pbase, nt_sum, p, rp.win, rp.r, rp.m, prm.ub + (size_t)b * kPMax * kPMax,
                  prm.max_sweeps, prm.conv_tol, step + 1, prm.status);
        epi_sync();
        if (et == 0) { __threadfence(); st_release_u32(sync_b + 2, 1u); }
      }
      return stop;
    };
    if (prm.n_servers > 0 && (int)blockIdx.x >= prm.n_tile_ctas) {
      // ------------------------------------------------------------ factor server
      // This CTA carries no tile.  It factors for one request: on a CTA that also carries a tile the
      // factorisation, which needs the operand ring as scratch, would delay that tile's next
      // multiplication, and with it the request's next step.
      const int b = server_request((int)blockIdx.x - prm.n_tile_ctas);
      if (b >= 0) {
        const ReqPlan rp = prm.plan[b];
        unsigned* sync_b = prm.sync + (size_t)b * kSyncStride;
        const unsigned nt = (unsigned)((rp.m + R - 1) / R);
        const bool summed = spread_of((int)nt, (rp.p + 7) & ~7);   // the tiles have added up the partial matrices
        int last_b = last_step;
        for (int step = 0; step <= last_b; ++step) {
          if (!team_wait(summed ? sync_b + 4 : sync_b, nt * (unsigned)(step + 1))) break;
          if (factor_request(b, rp, sync_b, step, step == last_b, last_b, summed ? 1 : (int)nt)) last_b = step + 1;
        }
      }
    }
    for (int step = 0; step <= last_step; ++step) {
      const bool identity = step == 0;
      __nv_bfloat16* y_hi = prm.y_hi[(step & 1) ^ 1];
      __nv_bfloat16* y_lo = prm.y_lo[(step & 1) ^ 1];
      for (int si = s_begin; si < s_end; ++si, ++n) {
        const TileItem rp = tile_at(si);
        const int b = rp.b, tile = rp.tile;
        const int p = rp.p, P = (p + 7) & ~7;
        unsigned* sync_b = prm.sync + (size_t)b * kSyncStride;
        const unsigned nt = (unsigned)((rp.m + R - 1) / R);
        // does the request still run this step, and is it its last one?  (one answer for the team)
        int last_b = last_step;
        if (!identity) {
          epi_sync();
          if (et == 0) {
            int lb = last_step;
            const int go = step_decide(sync_b, nt, step, gabort, abort_flag, &lb);
            s_word[0] = go; s_word[1] = lb;
          }
          epi_sync();
          const int go = s_word[0];
          last_b = s_word[1];
          if (go == 0) { --n; continue; }
          if (go < 0) ok = false;
        }
        if (!identity && (b != cached_b || step != cached_step)) {
          // the factor of the previous block, published by whichever tile finished that step last
          ok = team_wait(sync_b + 1, (unsigned)step) && ok;
          if (ok) {
            const float4* src = reinterpret_cast<const float4*>(prm.lbuf + (size_t)b * kLbufStride);
            float4* dst = reinterpret_cast<float4*>(lt);
            const int n4 = (lt_row_offset(P, P) + 3) / 4;    // 16-byte vectors the P-wide layout takes, eight in flight
            for (int e0 = et; e0 < n4; e0 += 8 * kEpiThreads) {
              float4 v[8];
#pragma unroll
              for (int u = 0; u < 8; ++u) v[u] = __ldcg(src + min(e0 + u * kEpiThreads, n4 - 1));
#pragma unroll
              for (int u = 0; u < 8; ++u)
                if (e0 + u * kEpiThreads < n4) dst[e0 + u * kEpiThreads] = v[u];
            }
            const float* dsrc = prm.lbuf + (size_t)b * kLbufStride + kLtFloats;
            for (int e = et; e < P; e += kEpiThreads) dinv[e] = __ldcg(dsrc + e);
          }
          epi_sync();
          cached_b = b; cached_step = step;
        }
        // whether this is the request's last step is known once the previous step's factor has been
        // published: the tile that computed it may have declared this step the last one
        if (!identity) {
          if (et == 0) s_word[1] = (int)ld_acquire_u32(sync_b + 3);
          epi_sync();
          last_b = s_word[1];
          epi_sync();
        }
        const bool is_last = step == last_b;
        float* yf = is_last ? prm.yf[1] : nullptr;
        float* qprev = is_last ? prm.yf[0] : nullptr;
        const int nrows = min(R, rp.m - tile * R);
        // ---- Y_next = T L^-T (forward substitution), staged as xs[c][r]; see solve_gemm / solve_diag ----
        const int nS = (P + 31) >> 5;
        const bool row_ok = r < nrows;
        // 32-row groups that lie wholly beyond the tile's rows (64-row tiles, ragged last tiles) are left
        // out; their rows of the staged block stay unwritten and are not read below
        const bool active = (warp & 3) * 32 < nrows;
        if (warp < 4) {
          ok = ok && mbar_wait(acc_full, n & 1u, abort_flag);
          tc_fence_after();
          if (active) {
#pragma unroll 1
            for (int S = 0; S < nS; ++S) {
              float v[32];
              tmem_ld32(t_lane + S * 32, v);
#pragma unroll
              for (int e = 0; e < 32; ++e)
                if (S * 32 + (e & ~7) < P) xs[(S * 32 + e) * kXsLd + r] = (row_ok && ok) ? v[e] : 0.f;
            }
          }
          tc_fence_before();
          mbar_arrive(acc_empty);
        } else if (is_last) {
          // last step, warps 4-7: the block this step multiplied, from its two bf16 planes (eight rows of a
          // column per vector), becomes Q = Y L^-T
          ok = ok && mbar_wait(acc_full, n & 1u, abort_flag);      // the ring is no longer read
          const int t4 = et - 128, chunks = (nrows + 7) >> 3;
          const size_t base = (size_t)b * kPMax * prm.ld + tile * R;
          const int ch = t4 & 15;
          if (ch < chunks) {
#pragma unroll 4
            for (int c = t4 >> 4; c < P; c += 8) {
              uint4 h = make_uint4(0u, 0u, 0u, 0u), l = h;
              if (c < p) {
                h = __ldcg(reinterpret_cast<const uint4*>(prm.y_hi[step & 1] + base + (size_t)c * prm.ld) + ch);
                l = __ldcg(reinterpret_cast<const uint4*>(prm.y_lo[step & 1] + base + (size_t)c * prm.ld) + ch);
              }
              const uint32_t uh[4] = {h.x, h.y, h.z, h.w}, ul[4] = {l.x, l.y, l.z, l.w};
              float f[8];
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                f[2 * e] = __uint_as_float(uh[e] << 16) + __uint_as_float(ul[e] << 16);
                f[2 * e + 1] = __uint_as_float(uh[e] & 0xffff0000u) + __uint_as_float(ul[e] & 0xffff0000u);
              }
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (ch * 8 + e >= nrows) f[e] = 0.f;
              float4* dst = reinterpret_cast<float4*>(xq + c * kXsLd + ch * 8);
              dst[0] = make_float4(f[0], f[1], f[2], f[3]);
              dst[1] = make_float4(f[4], f[5], f[6], f[7]);
            }
          }
          // 32-row groups that the diagonal solves touch are complete
          if (active && chunks * 8 + (t4 & 31) < ((nrows + 31) & ~31) && t4 < 32)
            for (int c = 0; c < P; ++c) xq[c * kXsLd + chunks * 8 + t4] = 0.f;
        }
        if (!identity) {
          for (int q = 0; q < (is_last ? 2 : 1); ++q) {     // the block, then (last step) Q
            if (is_last) epi_sync();
            solve_team(q * (kXsBytes / 4), P, R, !is_last, nrows, ok);
          }
        }
        if (is_last) {
          // only the window columns of Q are read again (second half of Eq. 15)
          float* qrows = qprev + ((size_t)rp.presel_off + tile * R) * kPMax;      // [win][nrows]
          for (int c = warp; c < rp.win; c += 8)
            for (int rr = lane; rr < nrows; rr += 32) qrows[c * nrows + rr] = xq[(p - rp.win + c) * kXsLd + rr];
        }
        epi_sync();                                  // the staged block is complete
        if (is_last && et < nrows) {
          // first half of Eq. 15 while both blocks are on chip: sum_j Y'_ij Q_ij, parked in the
          // energy array until the Ritz vectors of the request are known
          float total = 0.f;
          for (int c = 0; c < p; ++c) total += xs[c * kXsLd + et] * xq[c * kXsLd + et];
          prm.energy[(size_t)rp.presel_off + tile * R + et] = total;
        }
        // ---- bf16 planes of the new block (K-major operand of the next step): 8 positions per thread
        if (!is_last) {
          const int cols = (rp.m + kBK - 1) / kBK * kBK;
          const int cshift = R == 64 ? 3 : 4;          // 8-position chunks per row of the tile: 2^cshift
          for (int wi = et; wi < (p << cshift); wi += kEpiThreads) {
            int c = wi >> cshift, ch = wi & ((1 << cshift) - 1);
            int pos = tile * R + ch * 8;
            if (pos >= cols) continue;
            const float4* xp = reinterpret_cast<const float4*>(xs + c * kXsLd + ch * 8);
            float4 a = xp[0], d = xp[1];
            float f[8] = {a.x, a.y, a.z, a.w, d.x, d.y, d.z, d.w};
            if (ch * 8 + 8 > nrows) {                  // padding positions up to the k-chunk boundary are zero
#pragma unroll
              for (int e = 0; e < 8; ++e)
                if (ch * 8 + e >= nrows) f[e] = 0.f;
            }
            uint32_t ph[4], pl[4];
#pragma unroll
            for (int e = 0; e < 4; ++e) {
              __nv_bfloat162 hi = __floats2bfloat162_rn(f[2 * e], f[2 * e + 1]);
              ph[e] = *reinterpret_cast<uint32_t*>(&hi);
              pl[e] = pack_bf16(f[2 * e] - __low2float(hi), f[2 * e + 1] - __high2float(hi));
            }
            size_t o = ((size_t)b * kPMax + c) * prm.ld + pos;
            *reinterpret_cast<uint4*>(y_hi + o) = make_uint4(ph[0], ph[1], ph[2], ph[3]);
            *reinterpret_cast<uint4*>(y_lo + o) = make_uint4(pl[0], pl[1], pl[2], pl[3]);
          }
        }
        if (yf != nullptr) {
          // float32 window columns of the final block (second half of Eq. 15)
          float* yrows = yf + ((size_t)rp.presel_off + tile * R) * kPMax;          // [win][nrows]
          for (int c = warp; c < rp.win; c += 8)
            for (int rr = lane; rr < nrows; rr += 32) yrows[c * nrows + rr] = xs[(p - rp.win + c) * kXsLd + rr];
        }
        // ---- float64 partial Gram of the tile on the FP64 tensor cores ----
        const int coff = is_last ? ((p - rp.win) & ~7) : 0;
        {
          // The last step only feeds the Rayleigh-Ritz window: the trailing block of columns from
          // coff on, plus the diagonal of the leading columns (the scale of the problem).
          double* out = prm.partial + (size_t)(rp.ptile_off + tile) * kTileDoubles;
          for (int c = et; c < coff; c += kEpiThreads) {
            double sq = 0.0;
            for (int rr = 0; rr < nrows; ++rr) { double x = (double)xs[c * kXsLd + rr]; sq += x * x; }
            out[tile_offset(c, c)] = sq;
          }
          gram_tile_f64(xs, coff, (p - coff + 7) >> 3, (nrows + kSlabRows - 1) / kSlabRows, kEpiWarps - 1 - warp, lane, out);
        }
        // ---- arrival: this tile's slab and partial sums are published -------------------------
        // (one thread's fence covers what the others wrote before the barrier; a fence of every thread
        // cost 2-3 k cycles more)
        fence_proxy_async_all();
        epi_sync();
        int nt_sum = (int)nt;                        // partial matrices the factoring tile has to add up
        const bool spread = spread_of((int)nt, P);
        if (spread && si + 1 == s_end) {
          // All tiles of the request are being worked on at the same time, one group of them per CTA:
          // instead of leaving the sum of the partial matrices to one CTA, every CTA waits for the last
          // of the tiles and adds up its own slice of the matrix (in tile order, into the slot of
          // tile 0); the last one to finish its slice factors the summed matrix.
          if (et == 0) { __threadfence(); atomicAdd(sync_b, 1u); }
          ok = team_wait(sync_b, nt * (unsigned)(step + 1)) && ok;
          double* sum0 = prm.partial + (size_t)rp.ptile_off * kTileDoubles;
          const int used = (P >> 3) * ((P >> 3) + 1) / 2 * 64;
          const int chunk = ((used + n_groups - 1) / n_groups + 1) & ~1;
          const int e1 = min(used, (my_group + 1) * chunk);
          if (ok) {
            for (int e = my_group * chunk + 2 * et; e < e1; e += 2 * kEpiThreads) {
              double2 acc = make_double2(0.0, 0.0);
              for (int t0 = 0; t0 < (int)nt; t0 += 8) {
                double2 v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q)
                  v[q] = __ldcg(reinterpret_cast<const double2*>(sum0 + (size_t)min(t0 + q, (int)nt - 1) * kTileDoubles + e));
#pragma unroll
                for (int q = 0; q < 8; ++q)
                  if (t0 + q < (int)nt) { acc.x += v[q].x; acc.y += v[q].y; }
              }
              *reinterpret_cast<double2*>(sum0 + e) = acc;
            }
          }
          epi_sync();
          if (et == 0) {
            __threadfence();
            unsigned old = atomicAdd(sync_b + 4, 1u);
            __threadfence();
            *s_word = (old + 1u == (unsigned)n_groups * (unsigned)(step + 1) && !*abort_flag) ? 1 : 0;
          }
          nt_sum = 1;
        } else if (et == 0) {
          __threadfence();
          unsigned old = atomicAdd(sync_b, 1u);
          __threadfence();
          // one decision for the whole team (a CTA that has given up factors nothing)
          *s_word = (!spread && old + 1u == nt * (unsigned)(step + 1) && !*abort_flag) ? 1 : 0;
        }
        epi_sync();
        if (*s_word && prm.n_servers == 0) {
          // ---- the last tile of the request to finish this step factors the summed Gram matrix ----
          factor_request(b, rp, sync_b, step, is_last, last_b, nt_sum);
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        mbar_arrive(epi_done);
        if (identity && prm.n_servers > 0) {
          // Rehearsal: this CTA's only tile now waits for the first factor.  The solve runs once on whatever
          // the factor's place holds (a narrow block with the same remainder of columns, so that the same
          // code runs): it is in the instruction cache when the factor arrives, instead of being fetched line
          // by line from L2 on the critical path (batch of 16 requests: 27 -> 11 k cycles).
          const int dry = P <= 95 ? P : 64 + (P & 31);
          solve_team(kPowRegion / 4, dry, R, true, nrows, true);
        }
      }
    }
    // ------------------------------------------------------------ Eq. 15 for this CTA's tiles
    // c_i = sum_j Y'_ij Q_ij - sum_k (Y'_{i,win} u_k)(Q_{i,win} u_k)  (see eig_kernels.cuh)
    // The discarded Ritz pairs take only the window columns of the two blocks, which lie column by
    // column in global memory (coalesced over the rows; one token per row of 640 bytes took a sector
    // for every value: 28-40 k cycles a tile, now about 4 k).  Two threads share a row: of every
    // sixteen Ritz vectors the first projects the row on eight and the second on the next eight; the
    // products are added up in the order of the vectors, the second thread going on from the
    // first's sum.
    {
      float* us = reinterpret_cast<float*>(smem);                      // [w][nb8], zero-padded columns
      float* part = us + kPMax * kPMax;                                // [128] running sums
      int cached_u = -1;
      for (int si = s_begin; si < s_end; ++si) {
        const TileItem rp = tile_at(si);
        const int b = rp.b, tile = rp.tile;
        const int p = rp.p, w = rp.win, nbot = p - rp.r, nb8 = (nbot + 7) & ~7;
        const int nrows = min(R, rp.m - tile * R);
        const int rr = et & 127, second = et >> 7;
        const size_t grow = (size_t)rp.presel_off + tile * R;
        const float* yw = prm.yf[1] + grow * kPMax + rr;
        const float* qw = prm.yf[0] + grow * kPMax + rr;
        const bool have = rr < nrows;
        float yv[32], qv[32];
        auto load_chunk = [&](int j0) {
#pragma unroll
          for (int jj = 0; jj < 32; ++jj) {
            const bool in = have && j0 + jj < w;
            yv[jj] = in ? __ldcg(yw + (j0 + jj) * nrows) : 0.f;
            qv[jj] = in ? __ldcg(qw + (j0 + jj) * nrows) : 0.f;
          }
        };
        load_chunk(0);                                 // this CTA's own rows: before the wait for the Ritz vectors
        float total = have && !second ? __ldcg(prm.energy + grow + rr) : 0.f;
        if (b != cached_u) {
          ok = team_wait(prm.sync + (size_t)b * kSyncStride + 2, 1u) && ok;
          const float* usrc = prm.ub + (size_t)b * kPMax * kPMax;
          for (int e = et; e < w * nb8; e += kEpiThreads) {
            const int j = e / nb8, k = e - j * nb8;
            us[e] = ok && k < nbot ? __ldcg(usrc + j * nbot + k) : 0.f;
          }
          epi_sync();
          cached_u = b;
        }
        float sub_ = 0.f;
        for (int k0 = 0; k0 < nbot; k0 += 16) {
          const int kk = k0 + 8 * second;
          float ya[8], qa[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) { ya[u] = 0.f; qa[u] = 0.f; }
          if (have && kk < nbot) {
            for (int j0 = 0; j0 < w; j0 += 32) {
              if (w > 32) load_chunk(j0);
#pragma unroll
              for (int jj = 0; jj < 32; ++jj) {
                if (j0 + jj < w) {
                  const float4* ur = reinterpret_cast<const float4*>(us + (j0 + jj) * nb8 + kk);
                  const float4 u0 = ur[0], u1 = ur[1];
                  const float uu[8] = {u0.x, u0.y, u0.z, u0.w, u1.x, u1.y, u1.z, u1.w};
#pragma unroll
                  for (int u = 0; u < 8; ++u) { ya[u] += yv[jj] * uu[u]; qa[u] += qv[jj] * uu[u]; }
                }
              }
            }
          }
          if (!second) {
#pragma unroll
            for (int u = 0; u < 8; ++u) sub_ += ya[u] * qa[u];
            part[rr] = sub_;
          }
          epi_sync();
          if (second) {
            sub_ = part[rr];
#pragma unroll
            for (int u = 0; u < 8; ++u) sub_ += ya[u] * qa[u];
            part[rr] = sub_;
          }
          epi_sync();
          if (!second) sub_ = part[rr];
        }
        if (have && !second) prm.energy[grow + rr] = fmaxf((ok ? total : 0.f) - sub_, 0.f);
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 9) tmem_dealloc(tmem_base, kPowTmemCols);
  if (threadIdx.x == 0 && *abort_flag) atomicOr(prm.status, kStatusTimeout);
}

}  // namespace sub
}  // namespace covspec
