// The reduced power mode (QFS_POWER_REDUCED) as a kernel of its own, for p <= 7 in the dp4a form.  Per quartic: the chain
// to f~^p mod p^2, Delta_1(f), then
//     theta(F) = - f^(p-2) u(F Delta_1(f))   (mod p)
// for the iterates F (whose witness coefficient is zero; qfs_engine.cuh has the derivation), each followed by the
// height test.
//
// Every form of a quartic is small (degree 4p at most: 4,495 bytes at p = 7), so a CTA of four warps keeps them all in
// shared memory (by rows, qfs_rows.cuh) and works through the quartics that passed the height-1 screen.  Both the chain
// and the last step of theta are products with a quartic: f~, or - u(F Delta_1(f)).
//
// u(F Delta_1(f))[r] = sum_c Delta_1(f)[p r + (p-1)1 - c] F[c], r of degree 4: one warp per r, one row of F per lane.  F is
// kept reversed (byte j of row s: F[s - j]), so that a row's terms are a run of Delta_1(f) against a run of F; the rows
// of Delta_1(f) have zero guards on both sides instead of bounds checks.
//
// Bound by the latency of its small stages: four CTAs of 56 KB per SM at p = 7, so 16 warps, which issue in 61 % of the
// cycles (per issue: fixed latency 2.2, branches 0.7, barrier 0.5); no DRAM traffic to speak of.  262,144 dense quartics at p = 7, of
// which 37,224 reach it: 4.9 ms, against 13.8 ms in the fused kernel, where 256 threads with 128 registers and 92 KB run
// the same stages through device memory.
#include <cuda_runtime.h>

#include "../../include/qfs.h"
#include "qfs_reduced.cuh"
#include "qfs_rows.cuh"

namespace qfs {
namespace {

constexpr int kRThreads = 128;
constexpr int kRWarps = kRThreads / 32;

// Sizes and shared-memory layout (word offsets) for prime P.
template <int P>
struct Red {
  static constexpr int d = 4 * (P - 1), d1 = 4 * P, dm = 4 * (P - 2);   // f^(p-1), f^p and Delta_1(f), f^(p-2)
  static constexpr int pitch = rows::pitch_of(d1);
  static constexpr int guard = (d + 3) / 4 + 1;                // zero words before a row of Delta_1(f) ...
  static constexpr int dpitch = guard + d1 / 4 + 1;            // ... whose end meets the next row's
  static constexpr int d_words = tri(d1 + 1) * dpitch + guard + 1, g_words = (tri(d + 1) + 1) * pitch;
  static constexpr int x_words = d_words > g_words ? d_words : g_words;   // f~^(p-1), later Delta_1(f)
  static constexpr int y_words = (tri(d1 + 1) + 1) * pitch;               // f~^(p-2), f~^p
  static constexpr int m_words = (tri(dm + 1) + 1) * pitch;               // f^(p-2) mod p
  static constexpr int r_words = rows::items_of(d);                       // the iterate, rows reversed
  static constexpr int o_x = 0, o_y = x_words, o_m = o_y + y_words, o_r = o_m + m_words, o_items = o_r + r_words,
                       o_slice = o_items + (rows::items_of(d1) + 1) / 2, words = o_slice + d1 + 2;
};

struct RSmem {
  int taps[35];
  int q[35];
  rows::TapWords T;
  int powp[8];         // c^p mod p^2
  int64_t item;
};

// Tap words of the 35 values `a`, between two barriers.
__device__ __forceinline__ void build_taps(RSmem &S, const int *a) {
  __syncthreads();
  if (threadIdx.x < 15) S.T.tw[threadIdx.x] = rows::tap_word(a, threadIdx.x);
  if (threadIdx.x == 32) S.T.a44 = (uint32_t)a[34];
  __syncthreads();
}

template <int P>
__device__ int reduced_quartic(const uint8_t *__restrict__ f35, int max_h, RSmem &S, uint32_t *mem, uint32_t *status,
                               int &steps) {
  using Q = Red<P>;
  using Pr = Prime<P>;
  constexpr int pitch = Q::pitch, d = Q::d, d1 = Q::d1, dm = Q::dm;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  uint32_t *X = mem + Q::o_x + pitch, *Y = mem + Q::o_y + pitch, *M = mem + Q::o_m + pitch;   // row 0
  uint32_t *R = mem + Q::o_r;
  uint8_t *Rb = reinterpret_cast<uint8_t *>(R);
  const uint16_t *items = reinterpret_cast<const uint16_t *>(mem + Q::o_items);
  const int *slice = reinterpret_cast<const int *>(mem + Q::o_slice);   // items (and words of R) before slice u
  auto reversed = [&](int u, int s) { return Rb + 4 * (slice[u] + rows::words_below(s)); };
  steps = 0;
  // A1
  int bad = 0;
  if (tid < 35) {
    const int a = f35[tid];
    bad = a >= P;
    S.taps[tid] = a;
  }
  if (__syncthreads_or(bad)) return -1;
  for (int i = tid; i < Q::o_items; i += kRThreads) mem[i] = 0u;
  build_taps(S, S.taps);
  // f~ into Y; p - 2 (odd) products leave f~^(p-1) in X, one more f~^p in Y
  if (tid < 35) {
    int u, s, t;
    decode_packed(tid, u, s, t, 4);
    reinterpret_cast<uint8_t *>(Y + (tri(u) + s) * pitch + 1)[t] = (uint8_t)S.taps[tid];
    if (dm == 4) reinterpret_cast<uint8_t *>(M + (tri(u) + s) * pitch + 1)[t] = (uint8_t)S.taps[tid];   // p = 3
  }
  __syncthreads();
  uint32_t *cur = Y, *nxt = X;
#pragma unroll 1
  for (int m = 4; m < d1; m += 4) {
    const int n_items = slice[m + 5];
    for (int i = tid; i < n_items; i += kRThreads) {
      int u, s, w;
      rows::item_of(items, i, u, s, w);
      uint32_t g[4];
      rows::word_sums<pitch>(cur, m, S.T, u, s, w, g);
#pragma unroll
      for (int r = 0; r < 4; ++r) g[r] = mod_p2_mulhi<P>(g[r]);   // zero past the row's end
      const int o = (tri(u) + s) * pitch + 1 + w;
      nxt[o] = g[0] | g[1] << 8 | g[2] << 16 | g[3] << 24;
      if (m + 4 == dm) M[o] = g[0] % P | (g[1] % P) << 8 | (g[2] % P) << 16 | (g[3] % P) << 24;
      if (m + 4 == d) {   // g = f^(p-1) mod p, reversed
        uint8_t *row = reversed(u, s);
#pragma unroll
        for (int r = 0; r < 4; ++r)
          if (4 * w + r <= s) row[s - 4 * w - r] = (uint8_t)(g[r] % P);
      }
    }
    __syncthreads();
    if (m + 4 == d && reversed(Pr::wu, Pr::ws)[Pr::ws - Pr::wt] != 0) return 1;
    uint32_t *t = cur;
    cur = nxt;
    nxt = t;
  }
  // Delta_1(f) = (f~^p - sum a~_I^p x^(pI)) / p mod p into X's place, rows between guards
  uint32_t *D = mem + Q::o_x + Q::guard;   // row r at D + r dpitch
  for (int i = tid; i < Q::x_words; i += kRThreads) mem[Q::o_x + i] = 0u;
  __syncthreads();
  bool inexact = false;
  for (int i = tid; i < slice[d1 + 1]; i += kRThreads) {
    int u, s, w;
    rows::item_of(items, i, u, s, w);
    const uint32_t x = cur[(tri(u) + s) * pitch + 1 + w];
    uint32_t o = 0;
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int t = 4 * w + r;
      int G = (int)((x >> (8 * r)) & 0xFFu);
      if (u % P == 0 && s % P == 0 && t % P == 0 && t <= s) {
        G -= S.powp[S.taps[tet(u / P) + tri(s / P) + t / P]];
        if (G < 0) G += Pr::p2;
      }
      inexact |= G % P != 0;
      o |= (uint32_t)(G / P) << (8 * r);
    }
    D[(tri(u) + s) * Q::dpitch + w] = o;
  }
  if (inexact) atomicOr(status, kStatusInexactDivision);
  __syncthreads();
  for (int h = 2; h <= max_h; ++h) {
    for (int r = warp; r < 35; r += kRWarps) {
      int ur, sr, tr;
      decode_packed(r, ur, sr, tr, 4);
      const int eu0 = P * ur + 3 * (P - 1), es0 = P * sr + 2 * (P - 1), et0 = P * tr + (P - 1);
      unsigned a = 0;
      int uc = (isqrt(8 * lane + 1) - 1) >> 1, sc = lane - tri(uc);
      for (int col = lane; col < tri(d + 1); col += 32, sc += 32) {
        while (sc > uc) sc -= ++uc;
        const int eu = eu0 - uc, es = es0 - sc;
        if (eu < 0 || eu > d1 || es < 0 || es > eu) continue;
        // sum_j Delta_1(f)[eu, es, et0 - sc + j] F[uc, sc, sc - j]; bytes outside the row are zero
        const int byte = 4 * ((tri(eu) + es) * Q::dpitch) + et0 - sc;
        const uint32_t *dw = D + (byte >> 2);
        const unsigned sh = 8u * (unsigned)(byte & 3);
        const uint32_t *rw = reinterpret_cast<const uint32_t *>(reversed(uc, sc));
        uint32_t lo = dw[0];
        for (int k = 0; k <= sc >> 2; ++k) {
          const uint32_t hi = dw[k + 1];
          a = __dp4a(__funnelshift_r(lo, hi, sh), rw[k], a);
          lo = hi;
        }
      }
      a = __reduce_add_sync(0xffffffffu, a);
      if (lane == 0) {
        const int v = (int)(a % P);
        S.q[r] = v ? P - v : 0;   // the taps of - u(F Delta_1(f))
      }
    }
    build_taps(S, S.q);
    bool any = false;
    for (int i = tid; i < slice[d + 1]; i += kRThreads) {
      int u, s, w;
      rows::item_of(items, i, u, s, w);
      uint32_t acc[4];
      rows::word_sums<pitch>(M, dm, S.T, u, s, w, acc);
      uint8_t *row = reversed(u, s);
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        const uint32_t v = acc[r] % P;   // zero past the row's end
        if (4 * w + r <= s) row[s - 4 * w - r] = (uint8_t)v;
        any |= v != 0;
      }
    }
    const int nonzero = __syncthreads_or(any ? 1 : 0);
    steps = h - 1;
    if (reversed(Pr::wu, Pr::ws)[Pr::ws - Pr::wt] != 0) return h;
    if (!nonzero) return 0;
  }
  return 0;
}

// Persistent CTAs take the listed items; every group of the launch has prime P.
template <int P>
__global__ void __launch_bounds__(kRThreads) reduced_kernel(const __grid_constant__ FusedParams prm) {
  using Q = Red<P>;
  extern __shared__ __align__(16) uint32_t mem[];
  __shared__ RSmem S;
  {
    int *slice = reinterpret_cast<int *>(mem + Q::o_slice);
    rows::build_items(reinterpret_cast<uint16_t *>(mem + Q::o_items), Q::d1);
    for (int u = threadIdx.x; u <= Q::d1 + 1; u += kRThreads) {
      int n = 0;
      for (int v = 0; v < u; ++v) n += rows::words_below(v + 1);
      slice[u] = n;
    }
    if (threadIdx.x < P) {
      int v = 1;
      for (int e = 0; e < P; ++e) v = v * (int)threadIdx.x % Prime<P>::p2;
      S.powp[threadIdx.x] = v;
    }
  }
  const int64_t n_run = (int64_t)*prm.n_list;
  for (;;) {
    __syncthreads();
    if (threadIdx.x == 0) {
      const int64_t k = (int64_t)atomicAdd(prm.counter, 1ull);
      S.item = k < n_run ? prm.list[k] : -1;
    }
    __syncthreads();
    const int64_t item = S.item;
    if (item < 0) return;
    int gi = 0;
    while (gi + 1 < prm.n_groups && item >= prm.g[gi + 1].item_begin) ++gi;
    const FusedGroup &G = prm.g[gi];
    const int64_t row = item - G.item_begin;
    int steps;
    const int h = reduced_quartic<P>(G.coeffs + 35 * row, prm.max_h, S, mem, prm.status, steps);
    if (threadIdx.x == 0) {
      G.heights[row] = (int8_t)h;
      if (h != 1 && h != -1) {
        atomicAdd(prm.stats, 1ull);
        atomicAdd(prm.stats + 1, (unsigned long long)steps);
      }
    }
  }
}

template <int P>
cudaError_t launch(const FusedParams &prm, int sms, cudaStream_t st) {
  const size_t smem = sizeof(uint32_t) * Red<P>::words;
  cudaError_t e = cudaFuncSetAttribute(reduced_kernel<P>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, reduced_kernel<P>, kRThreads, smem);
  if (e != cudaSuccess) return e;
  const int64_t grid = (int64_t)sms * (per_sm > 0 ? per_sm : 1);
  reduced_kernel<P><<<(int)(grid < prm.n_items ? grid : prm.n_items), kRThreads, smem, st>>>(prm);
  return cudaGetLastError();
}

}  // namespace

cudaError_t reduced_launch(int p, const FusedParams &prm, int sms, cudaStream_t st) {
  switch (p) {
    case 3: return launch<3>(prm, sms, st);
    case 5: return launch<5>(prm, sms, st);
    default: return launch<7>(prm, sms, st);
  }
}

}  // namespace qfs
