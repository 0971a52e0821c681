// Theta by residue classes with the classes stored by rows (chain power mode, p <= 5).
//
// theta(g) = sum_sigma Delta_sigma * g_rho over the p^3 residue classes (qfs_engine.cuh, Poly): products of forms whose
// kernel g_rho has degree k <= 3.  Delta is split once per quartic into one array per class, all of one size, in global
// memory: rows (u, s) of bytes, each after a zero word (rows beyond the class's degree are zero), behind a zero row.  A
// step copies the classes through shared memory by cp.async, kGroup at a time (all of them at p = 3), one barrier per
// group, and multiplies them as they lie there: a thread takes one output word (four outputs) and every fourth class,
// reads two words of each input row and meets the taps by dp4a in the windows of qfs_block.cuh.  (The padded byte cube
// of theta_poly takes a scatter of every class into the cube, a barrier per class and a byte load per MAC.)
//
// Bound by instruction issue.  Whole calls, by cube and by rows: p = 5, 131,071 sparse quartics (4.4 steps each) 133.9 and
// 118.4 ms; p = 5, 65,536 dense 25.1 and 24.4 ms; 65 quartics at p = 3, where up to ten steps follow each other, 93 and 66 us.
#pragma once
#include <cstdint>
#include "qfs_common.cuh"
#include "qfs_rows.cuh"

namespace qfs {

template <int P>
struct RowClasses {
  static constexpr int d = 4 * (P - 1), ld = tet(d + 1), n_cls = P * P * P;
  static constexpr int zero = d / 4 + 2;                                         // words of the zero row
  static constexpr int n_items = rows::items_of(d), items = (n_items + 31) & ~31;   // output words; padded to warps
  static constexpr int words = (zero + n_items + tri(d + 1) + 3) & ~3;           // of a class
  static constexpr int kQuarters = 4;                                            // a thread takes every fourth class
  static constexpr int units = kQuarters * items / kThreads;                     // (output word, quarter) per thread
  static_assert(kQuarters * items % kThreads == 0, "whole rounds of units");
  static constexpr int group = P == 3 ? n_cls + 1 : 8;                           // classes staged at a time
  static constexpr int groups = (n_cls + group - 1) / group;
  static constexpr int slots = groups > 1 ? 2 : 1;
  // shared memory, word offsets
  static constexpr int o_taps = 0, o_acc = o_taps + 8 * n_cls, o_stage = (o_acc + 4 * items + 3) & ~3,
                       o_items = o_stage + slots * group * words, o_slice = o_items + (items + 1) / 2,
                       smem_words = o_slice + d + 2;
  static_assert(group % kQuarters == 0, "a group holds as many classes of every quarter");
};
__host__ __device__ constexpr int row_class_smem_words(int p) {
  return p == 3 ? RowClasses<3>::smem_words : p == 5 ? RowClasses<5>::smem_words : 0;
}
// words of device memory per CTA for the classes
__host__ __device__ constexpr size_t row_class_words(int p) {
  return p == 3 ? (size_t)RowClasses<3>::n_cls * RowClasses<3>::words
                : p == 5 ? (size_t)RowClasses<5>::n_cls * RowClasses<5>::words : 0;
}

// Word offset of row (u, s) in a class; slice[u]: words of the rows of the slices before u.
template <int P>
__device__ __forceinline__ int class_row(const int *slice, int u, int s) {
  return RowClasses<P>::zero + slice[u] + rows::words_below(s) + s;
}

// Padded Delta (degree D) -> the classes `rc`; class s2 + p s3 + p^2 s4 holds Delta[p e + sigma], sigma = (.., s2, s3, s4)
// per exponent.  Also builds the tables of theta_rows.  Ends with a barrier.
template <int P>
__device__ __noinline__ void delta_to_rows(const uint32_t *__restrict__ delta, uint32_t *__restrict__ rc, const Smem &sm,
                                           uint32_t *ring) {
  using Q = RowClasses<P>;
  constexpr int D = Prime<P>::D;
  int *slice = reinterpret_cast<int *>(ring + Q::o_slice);
  for (int i = threadIdx.x; i < Q::n_cls * Q::words / 4; i += blockDim.x)
    reinterpret_cast<uint4 *>(rc)[i] = make_uint4(0u, 0u, 0u, 0u);
  rows::build_items(reinterpret_cast<uint16_t *>(ring + Q::o_items), Q::d);
  for (int u = threadIdx.x; u <= Q::d + 1; u += blockDim.x) {
    int n = 0;
    for (int v = 0; v < u; ++v) n += rows::words_below(v + 1) + v + 1;
    slice[u] = n;
  }
  __syncthreads();
  uint8_t *rb = reinterpret_cast<uint8_t *>(rc);
  const int nchunks = sm.SW[D + 1] / 4;
  for (int k = threadIdx.x; k < nchunks; k += blockDim.x) {
    int U, S, c;
    decode_form_chunk(k, D, sm.SW, U, S, c);
    const uint4 v = __ldcg(reinterpret_cast<const uint4 *>(delta + 4 * k));   // a crew's write
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const int e2 = U - S, q2 = e2 / P, r2 = e2 - P * q2;
    const int T0 = 16 * c;
    int q4 = T0 / P, r4 = T0 - P * q4;                 // e4 = T
    int q3 = (S - T0) / P, r3 = (S - T0) - P * q3;     // e3 = S - T (>= 0 while T <= S)
#pragma unroll
    for (int b = 0; b < 16; ++b) {
      if (T0 + b <= S) {
        const int up = q2 + q3 + q4, sp = q3 + q4;
        rb[4 * ((r2 + P * r3 + P * P * r4) * Q::words + class_row<P>(slice, up, sp) + 1) + q4] =
            (uint8_t)(w[b >> 2] >> (8 * (b & 3)));
      }
      if (++r4 == P) { r4 = 0; ++q4; }
      if (--r3 < 0) { r3 = P - 1; --q3; }
    }
  }
  __syncthreads();
}

// Degree of class x's kernel, and rho's exponents of x2, x3, x4.
template <int P>
__device__ __forceinline__ int class_kernel(int x, int &r2, int &r3, int &r4) {
  r2 = P - 1 - x % P;
  r3 = P - 1 - (x / P) % P;
  r4 = P - 1 - x / (P * P);
  constexpr int d = 4 * (P - 1);
  const int rest = d - r2 - r3 - r4;   // = p k + r1
  return rest / P;
}

// One theta step: g (shared, packed) -> gn.  `rc`: the classes (delta_to_rows, which also left the tables in `ring`).
// Returns whether some output is nonzero (same value in every thread).
template <int P>
__device__ __noinline__ bool theta_rows(const uint32_t *__restrict__ rc, const uint8_t *__restrict__ g,
                                        uint8_t *__restrict__ gn, uint32_t *ring) {
  using Q = RowClasses<P>;
  const int tid = threadIdx.x;
  uint32_t *taps = ring + Q::o_taps;
  int *acc = reinterpret_cast<int *>(ring + Q::o_acc);
  uint32_t *stage = ring + Q::o_stage;
  const uint16_t *items = reinterpret_cast<const uint16_t *>(ring + Q::o_items);
  const int *slice = reinterpret_cast<const int *>(ring + Q::o_slice);
  auto fetch = [&](int gi) {
    if (gi < Q::groups) {
      const int n = min(Q::group, Q::n_cls - gi * Q::group) * Q::words / 4;
      uint32_t *dst = stage + (gi % Q::slots) * Q::group * Q::words;
      const uint32_t *src = rc + (size_t)gi * Q::group * Q::words;
      for (int i = tid; i < n; i += kThreads) cp_async16(dst + 4 * i, src + 4 * i, true);
    }
    cp_async_commit();
  };
  fetch(0);
  // tap words of every class: 0: a(0,0,0) in byte 3; uI = 1 .. 3: Y, byte 1: a(uI,0,0), 2: a(uI,1,1), 3: a(uI,1,0); 4, 5: the
  // pairs (2, 2), (3, 2), byte k: a(uI, sI, 3 - k); 6: (3, 3)
  for (int i = tid; i < 8 * Q::n_cls; i += kThreads) {
    int r2, r3, r4;
    const int k = class_kernel<P>(i >> 3, r2, r3, r4), j = i & 7;
    const int uI = j < 4 ? j : j == 4 ? 2 : 3;
    uint32_t w = 0;
    if (j < 7 && uI <= k) {
      const int sI = j == 0 ? 0 : j < 4 ? 1 : j < 6 ? 2 : 3;
      const uint8_t *gu = g + tet(P * uI + r2 + r3 + r4) + r4;
      const uint8_t *gr = gu + tri(P * sI + r3 + r4);
      for (int t = 0; t <= sI; ++t) w |= (uint32_t)gr[P * t] << (8 * (3 - t));
      if (j >= 1 && j < 4) w |= (uint32_t)gu[tri(r3 + r4)] << 8;
    }
    taps[i] = w;
  }
  for (int i = tid; i < 4 * Q::items; i += kThreads) acc[i] = 0;
  // this thread's units: row offsets A[uI] + B[sI] + w of the input rows (u - uI, s - sI), and which of them exist
  int A[Q::units][4], B[Q::units][4], quarter[Q::units];
  unsigned on[Q::units];
  int sum[Q::units][4];
#pragma unroll
  for (int n = 0; n < Q::units; ++n) {
    const int unit = tid + kThreads * n;
    quarter[n] = unit / Q::items;
    const int item = unit % Q::items;
    int u = 0, s = 0, w = 0;
    if (item < Q::n_items) rows::item_of(items, item, u, s, w);
    on[n] = 0;
#pragma unroll
    for (int I = 0; I < 4; ++I) {
      A[n][I] = u >= I ? Q::zero + slice[u - I] + w : 0;
      B[n][I] = s >= I ? rows::words_below(s - I) + s - I : 0;
    }
#pragma unroll
    for (int uI = 0; uI < 4; ++uI)
#pragma unroll
      for (int sI = 0; sI <= uI; ++sI)
        if (item < Q::n_items && s >= sI && s - sI <= u - uI) on[n] |= 1u << (tri(uI) + sI);
#pragma unroll
    for (int r = 0; r < 4; ++r) sum[n][r] = 0;
  }
  for (int gi = 0; gi < Q::groups; ++gi) {
    cp_async_wait_all();
    __syncthreads();   // group gi is staged for every thread, and nobody reads the slot of the group before
    fetch(gi + 1);
    const uint32_t *st = stage + (gi % Q::slots) * Q::group * Q::words;
    const int n_here = min(Q::group, Q::n_cls - gi * Q::group);
#pragma unroll
    for (int n = 0; n < Q::units; ++n)
      for (int c = quarter[n]; c < n_here; c += Q::kQuarters) {
        const int x = gi * Q::group + c;
        int r2, r3, r4;
        const int k = class_kernel<P>(x, r2, r3, r4);   // the same for the whole warp
        const uint32_t *cls = st + c * Q::words;
        const uint4 ta = *reinterpret_cast<const uint4 *>(taps + 8 * x);
        const uint32_t y[4] = {ta.x, ta.y, ta.z, ta.w};
        auto row = [&](int uI, int sI) { return cls + ((on[n] >> (tri(uI) + sI)) & 1u ? A[n][uI] + B[n][sI] : 0); };
        {
          const uint32_t x1 = row(0, 0)[1], a = y[0] >> 24;
#pragma unroll
          for (int r = 0; r < 4; ++r) sum[n][r] = (int)__dp4a(x1, a << (8 * r), (unsigned)sum[n][r]);
        }
#pragma unroll
        for (int uI = 1; uI < 4; ++uI) {
          if (uI > k) break;
          const uint32_t *q1 = row(uI, 1);
          const uint32_t z1 = row(uI, 0)[1], x0 = q1[0], x1 = q1[1];
          const uint32_t t1 = __byte_perm(x0, x1, 0x4300u);
          sum[n][0] = (int)__dp4a(__byte_perm(z1, t1, 0x7600u), y[uI], (unsigned)sum[n][0]);
          sum[n][1] = (int)__dp4a(__byte_perm(z1, x1, 0x5410u), y[uI], (unsigned)sum[n][1]);
          sum[n][2] = (int)__dp4a(__byte_perm(z1, x1, 0x6520u), y[uI], (unsigned)sum[n][2]);
          sum[n][3] = (int)__dp4a(__byte_perm(z1, x1, 0x7630u), y[uI], (unsigned)sum[n][3]);
#pragma unroll
          for (int sI = 2; sI <= uI; ++sI) {
            const uint32_t *q = row(uI, sI);
            const uint32_t v0 = q[0], v1 = q[1], tw = taps[8 * x + (sI == 3 ? 6 : uI + 2)];
            sum[n][0] = (int)__dp4a(__byte_perm(v0, v1, 0x4321u), tw, (unsigned)sum[n][0]);
            sum[n][1] = (int)__dp4a(__byte_perm(v0, v1, 0x5432u), tw, (unsigned)sum[n][1]);
            sum[n][2] = (int)__dp4a(__byte_perm(v0, v1, 0x6543u), tw, (unsigned)sum[n][2]);
            sum[n][3] = (int)__dp4a(v1, tw, (unsigned)sum[n][3]);
          }
        }
      }
    if (Q::slots == 1) __syncthreads();
  }
#pragma unroll
  for (int n = 0; n < Q::units; ++n)
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (on[n]) atomicAdd(acc + 4 * ((tid + kThreads * n) % Q::items) + r, sum[n][r]);
  __syncthreads();
  bool any = false;
  for (int i = tid; i < Q::n_items; i += kThreads) {
    int u, s, w;
    rows::item_of(items, i, u, s, w);
#pragma unroll
    for (int r = 0; r < 4; ++r)
      if (4 * w + r <= s) {
        const int v = acc[4 * i + r] % P;
        gn[tet(u) + tri(s) + 4 * w + r] = (uint8_t)v;
        any |= v != 0;
      }
  }
  return __syncthreads_or(any ? 1 : 0) != 0;
}

}  // namespace qfs
