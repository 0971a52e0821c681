// Theta by residue classes with the classes stored by rows (chain power mode at p <= 5, identity mode at p <= 7).
//
// theta(g) = sum_sigma Delta_sigma * g_rho over the p^3 residue classes (qfs_engine.cuh, Poly): products of forms whose
// kernel g_rho has degree k <= 3.  Delta is split once per quartic (the identity mode forms it class by class) into one array
// per class, all of one size, in global memory: rows (u, s) of bytes, each after a zero word (rows beyond the class's degree are zero), behind a zero row.  A
// step copies the classes through shared memory by cp.async, a group at a time (all of them at p = 3), one barrier per
// group, and multiplies them as they lie there: a thread takes one output word (four outputs) and every fourth class
// (p = 7: four output words and every class), reads two words of each input row and meets the taps by dp4a in the windows of qfs_block.cuh.  (The padded byte cube
// of theta_poly takes a scatter of every class into the cube, a barrier per class and a byte load per MAC.)
//
// Bound by latency and barriers at 16 warps per SM: the fused launch over sparse quartics at p = 5, where theta and the
// classes are two fifths of it, issues in 54 % of the cycles (per issue: fixed latency 1.6, barrier 1.5, shared memory 0.8), the
// identity mode's at p = 7 in 58 %; DRAM 3 and 15 %.  Whole calls, by cube and by rows: p = 5, 131,071 sparse quartics (4.4 steps each) 133.9 and
// 102.4 ms; p = 5, 65,536 dense 25.1 and 21.6 ms; 65 quartics at p = 3, where up to ten steps follow each other, 93 and 66 us.
// The identity mode at p = 7, 65,536 dense quartics (9,400 past height 1): 41.8 and 23.7 ms.
#pragma once
#include <cstdint>
#include "qfs_common.cuh"
#include "qfs_rows.cuh"

namespace qfs {

template <int P>
struct RowClasses {
  static constexpr int d = 4 * (P - 1), ld = tet(d + 1), dm = 4 * (P - 2), n_cls = P * P * P;
  static constexpr int zero = d / 4 + 2;                                         // words of the zero row
  static constexpr int kQuarters = P == 7 ? 1 : 4;                               // a thread takes every such class ...
  static constexpr int n_items = rows::items_of(d);                              // ... for some of the output words
  static constexpr int round = kThreads / kQuarters, items = (n_items + round - 1) / round * round;
  static constexpr int words = (zero + n_items + tri(d + 1) + 3) & ~3;           // of a class
  static constexpr int units = kQuarters * items / kThreads;                     // (output word, quarter) per thread
  static constexpr int group = P == 3 ? n_cls + 1 : P == 5 ? 12 : 4;             // classes staged at a time
  static constexpr int groups = (n_cls + group - 1) / group;
  static constexpr int slots = groups > 1 ? 2 : 1;
  // shared memory, word offsets
  static constexpr int o_taps = 0, o_acc = o_taps + 8 * n_cls, o_stage = (o_acc + 4 * items + 3) & ~3,
                       o_items = o_stage + slots * group * words, o_slice = o_items + (items + 1) / 2,
                       smem_words = o_slice + d + 2;
  static_assert(group % kQuarters == 0, "a group holds as many classes of every quarter");
  // the identity mode, before theta: f^(p-2) by rows (between two zero rows) and twelve tap words per class
  static constexpr int pitch = rows::pitch_of(dm), o_form = pitch, o_dtaps = (pitch * (tri(dm + 1) + 2) + 3) & ~3;
  static_assert(o_dtaps + 12 * n_cls <= o_items, "the identity mode's arrays fit before the tables");
};
__host__ __device__ constexpr int row_class_smem_words(int p) {
  return p == 3 ? RowClasses<3>::smem_words : p == 5 ? RowClasses<5>::smem_words : p == 7 ? RowClasses<7>::smem_words : 0;
}
// words of device memory per CTA for the classes
__host__ __device__ constexpr size_t row_class_words(int p) {
  return p == 3 ? (size_t)RowClasses<3>::n_cls * RowClasses<3>::words
                : p == 5 ? (size_t)RowClasses<5>::n_cls * RowClasses<5>::words
                         : p == 7 ? (size_t)RowClasses<7>::n_cls * RowClasses<7>::words : 0;
}
// Whether a fused launch takes theta by rows at prime p: where Delta comes from the chain only at p <= 5 (at p = 7
// theta_stream reads the padded Delta as the chain leaves it).
__host__ __device__ constexpr bool theta_by_rows(int p, int power_mode) {
  return (power_mode == 0 && p <= 5) || (power_mode == 1 && p <= 7);
}

// Word offset of row (u, s) in a class; slice[u]: words of the rows of the slices before u.
template <int P>
__device__ __forceinline__ int class_row(const int *slice, int u, int s) {
  return RowClasses<P>::zero + slice[u] + rows::words_below(s) + s;
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

// The tables of theta_rows: its items and slice offsets.  The caller synchronises.
template <int P>
__device__ __forceinline__ void row_class_tables(uint32_t *ring) {
  using Q = RowClasses<P>;
  int *slice = reinterpret_cast<int *>(ring + Q::o_slice);
  rows::build_items(reinterpret_cast<uint16_t *>(ring + Q::o_items), Q::d);
  for (int u = threadIdx.x; u <= Q::d + 1; u += blockDim.x) {
    int n = 0;
    for (int v = 0; v < u; ++v) n += rows::words_below(v + 1) + v + 1;
    slice[u] = n;
  }
}

// Padded Delta (degree D) -> the classes `rc`; class s2 + p s3 + p^2 s4 holds Delta[p e + sigma], sigma = (.., s2, s3, s4)
// per exponent.  A warp takes every eighth class and gathers it word by word, kAhead words per lane at a time to have as
// many loads in flight; the reads of a row's bytes meet in L1 and the stores are whole rows.  (A scatter of Delta's
// bytes, chunk by chunk, writes a sector per byte: at p = 5, 92,000 of them per quartic, 115.9 ms per 131,071 sparse
// quartics against 105.8, and 24.3 ms per 65,536 dense ones against 21.9.)  Also builds the tables of theta_rows.  Ends
// with a barrier.
template <int P>
__device__ __noinline__ void delta_to_rows(const uint32_t *delta, uint32_t *__restrict__ rc, const Smem &sm,
                                           uint32_t *ring) {
  using Q = RowClasses<P>;
  constexpr int kAhead = 5;
  row_class_tables<P>(ring);
  __syncthreads();
  const uint16_t *items = reinterpret_cast<const uint16_t *>(ring + Q::o_items);
  const int *slice = reinterpret_cast<const int *>(ring + Q::o_slice);
  const uint8_t *db = reinterpret_cast<const uint8_t *>(delta);
  const int lane = threadIdx.x & 31;
  for (int x = threadIdx.x >> 5; x < Q::n_cls; x += kThreads / 32) {
    int r2, r3, r4;
    const int k = class_kernel<P>(x, r2, r3, r4);
    const int s3 = P - 1 - r3, s4 = P - 1 - r4, su = 3 * (P - 1) - r2 - r3 - r4;   // sigma
    uint32_t *out = rc + (size_t)x * Q::words;
    for (int i = lane; i < Q::zero; i += 32) out[i] = 0;
    for (int i0 = 0; i0 < Q::n_items; i0 += 32 * kAhead) {
      uint32_t v[kAhead];
      int at[kAhead];
      bool first[kAhead];
#pragma unroll
      for (int j = 0; j < kAhead; ++j) {
        const int i = i0 + 32 * j + lane;
        int u = 0, s = 0, w = 0;
        if (i < Q::n_items) rows::item_of(items, i, u, s, w);
        at[j] = i < Q::n_items ? class_row<P>(slice, u, s) + w : -1;
        first[j] = w == 0;
        v[j] = 0;
        if (i < Q::n_items && u <= Q::d - k) {
          const uint8_t *q = db + 4 * (sm.SW[P * u + su] + colw(P * s + s3 + s4)) + 4 * P * w + s4;
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (4 * w + r <= s) v[j] |= (uint32_t)q[P * r] << (8 * r);
        }
      }
#pragma unroll
      for (int j = 0; j < kAhead; ++j)
        if (at[j] >= 0) {
          if (first[j]) out[at[j]] = 0;
          out[at[j] + 1] = v[j];
        }
    }
  }
  __syncthreads();
}

// The identity mode's Delta_1 array (identity_classes in qfs_engine.cuh states the classes' formula) in the order and
// layout of delta_to_rows.  f^(p-2) lies by rows in shared memory.  A thread takes one output word at a time, holds the
// forty byte windows that its products can need in registers, and goes through the classes: a class takes its tap words
// (the same address for the whole warp), 4, 12, 24 or 40 dp4a, four reductions and a store that a warp writes together.
// (A warp per class, which reads and aligns the rows anew for every class, took 15.1 ms for 9,400 quartics at p = 7, this takes 8.5.)
// Also builds the tables of theta_rows.  Ends with a barrier.
template <int P>
__device__ __noinline__ void identity_rows(const uint8_t *__restrict__ fpm2, const uint8_t *__restrict__ d1f,
                                           const uint8_t *__restrict__ E, uint32_t *__restrict__ rc, uint32_t *ring) {
  using Q = RowClasses<P>;
  const int tid = threadIdx.x;
  row_class_tables<P>(ring);
  uint8_t *fb = reinterpret_cast<uint8_t *>(ring);
  for (int i = tid; i < tri(Q::dm + 1) + 2; i += kThreads)   // the zero rows, every row's zero word and the rows' ends
    for (int w = 0; w < Q::pitch; ++w) ring[i * Q::pitch + w] = 0;
  // Twelve words per class: Y1, Y2, P22, K, Y3, P32, P33, Y4, P42, P43, P44, 0.  YuI holds a(uI,0,0) in byte 1, a(uI,1,1) in byte
  // 2, a(uI,1,0) in byte 3; PuIsI a(uI, sI, 3 - k) in byte k.  a(0,0,0) rides in byte 0 of Y1, a(4,4,4) in byte 0 of P22.
  for (int i = tid; i < 12 * Q::n_cls; i += kThreads) {
    const int x = i / 12, j = i % 12;
    int r2, r3, r4;
    const int K = 4 - class_kernel<P>(x, r2, r3, r4);
    const int s3 = P - 1 - r3, s4 = P - 1 - r4, su = 3 * (P - 1) - r2 - r3 - r4;   // sigma
    const int uI = j == 0 ? 1 : j < 3 ? 2 : j < 7 ? 3 : 4;
    const int sI = j == 2 || j == 5 || j == 8 ? 2 : j == 6 || j == 9 ? 3 : j == 10 ? 4 : 1;
    const int u = j == 7 ? 4 : uI;   // Y4
    auto tap = [&](int uu, int ss, int tt) {
      return (uint32_t)d1f[tet(P * uu + su) + tri(P * ss + s3 + s4) + P * tt + s4];
    };
    uint32_t w = 0;
    if (j == 3) w = (uint32_t)K;
    else if (j < 11 && u <= K) {
      for (int t = 0; t <= sI && t < 4; ++t) w |= tap(u, sI, t) << (8 * (3 - t));
      if (sI == 1) w |= tap(u, 0, 0) << 8;
      if (j == 0) w |= tap(0, 0, 0);
      if (j == 2 && K == 4) w |= tap(4, 4, 4);
    }
    ring[Q::o_dtaps + i] = w;
  }
  for (int i = tid; i < Q::n_cls * Q::zero; i += kThreads) rc[(size_t)(i / Q::zero) * Q::words + i % Q::zero] = 0;
  __syncthreads();
  for (int i = tid; i < tri(Q::dm + 1); i += kThreads) {
    int u = 0;
    while (tri(u + 1) <= i) ++u;
    const int s = i - tri(u);
    for (int t = 0; t <= s; ++t) fb[4 * (Q::o_form + i * Q::pitch + 1) + t] = fpm2[tet(u) + tri(s) + t];
  }
  __syncthreads();
  const uint16_t *items = reinterpret_cast<const uint16_t *>(ring + Q::o_items);
  const int *slice = reinterpret_cast<const int *>(ring + Q::o_slice);
  for (int i = tid; i < Q::n_items; i += kThreads) {
    int u, s, w;
    rows::item_of(items, i, u, s, w);
    auto row = [&](int uI, int sI) {
      const int u2 = u - uI, s2 = s - sI;
      const uint32_t *form = ring + Q::o_form;
      return form + (u2 >= s2 && s2 >= 0 && u2 <= Q::dm ? (tri(u2) + s2) * Q::pitch + w : -Q::pitch);
    };
    uint32_t Y[4][4], W[6][4];   // Y1 .. Y4; P22, P32, P33, P42, P43, P44
#pragma unroll
    for (int uI = 1; uI < 5; ++uI) {
      const uint32_t *q = row(uI, 1);
      const uint32_t z1 = row(uI, 0)[1], x0 = q[0], x1 = q[1];
      Y[uI - 1][0] = __byte_perm(z1, __byte_perm(x0, x1, 0x4300u), 0x7600u);
      Y[uI - 1][1] = __byte_perm(z1, x1, 0x5410u);
      Y[uI - 1][2] = __byte_perm(z1, x1, 0x6520u);
      Y[uI - 1][3] = __byte_perm(z1, x1, 0x7630u);
#pragma unroll
      for (int sI = 2; sI <= uI; ++sI) {
        const uint32_t *qq = row(uI, sI);
        const uint32_t v0 = qq[0], v1 = qq[1];
        uint32_t(&x)[4] = W[tri(uI - 2) + sI - 2];
        x[0] = __byte_perm(v0, v1, 0x4321u);
        x[1] = __byte_perm(v0, v1, 0x5432u);
        x[2] = __byte_perm(v0, v1, 0x6543u);
        x[3] = v1;
      }
    }
    {
      const uint32_t x00 = row(0, 0)[1], x44 = row(4, 4)[0];
#pragma unroll
      for (int r = 0; r < 4; ++r) {
        Y[0][r] = __byte_perm(Y[0][r], x00, 0x3214u + r);
        W[0][r] = __byte_perm(W[0][r], x44, 0x3214u + r);
      }
    }
    uint32_t *out = rc + class_row<P>(slice, u, s) + w;
    const uint4 *taps = reinterpret_cast<const uint4 *>(ring + Q::o_dtaps);
    for (int x = 0; x < Q::n_cls; ++x, out += Q::words, taps += 3) {
      const uint4 t = taps[0];
      const int K = (int)t.w;
      uint32_t v = 0;
      if (u <= Q::d - 4 + K) {
        uint32_t acc[4];
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = __dp4a(Y[0][r], t.x, 0u);
        if (K >= 2) {
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[r] = __dp4a(W[0][r], t.z, __dp4a(Y[1][r], t.y, acc[r]));
        }
        if (K >= 3) {
          const uint4 t3 = taps[1];
#pragma unroll
          for (int r = 0; r < 4; ++r)
            acc[r] = __dp4a(W[2][r], t3.z, __dp4a(W[1][r], t3.y, __dp4a(Y[2][r], t3.x, acc[r])));
          if (K >= 4) {
            const uint4 t4 = taps[2];
#pragma unroll
            for (int r = 0; r < 4; ++r)
              acc[r] = __dp4a(W[5][r], t4.z, __dp4a(W[4][r], t4.y, __dp4a(W[3][r], t4.x,
                              __dp4a(Y[3][r], t3.w, acc[r]))));
          }
        }
        if (x == 0) {   // class 0 also receives E
#pragma unroll
          for (int r = 0; r < 4; ++r)
            if (4 * w + r <= s) acc[r] += (uint32_t)(P - E[tet(u) + tri(s) + 4 * w + r]);
        }
#pragma unroll
        for (int r = 0; r < 4; ++r) {
          const uint32_t m = acc[r] % P;
          v |= (m ? P - m : 0u) << (8 * r);   // -(f^(p-2) D_sigma - E) mod p
        }
      }
      if (w == 0) out[0] = 0;
      out[1] = v;
    }
  }
  __syncthreads();
}

// One theta step: g (shared, packed) -> gn.  `rc`: the classes (delta_to_rows or identity_rows, which also left the tables in `ring`).
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
  // pairs (2, 2), (3, 2), byte k: a(uI, sI, 3 - k); 6: (3, 3); 7: the degree k
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
    taps[i] = j == 7 ? (uint32_t)k : w;
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
    for (int n = 0; n < Q::units; ++n) {
      int off[10];   // of the input rows, the zero row where there is none
#pragma unroll
      for (int uI = 0; uI < 4; ++uI)
#pragma unroll
        for (int sI = 0; sI <= uI; ++sI) off[tri(uI) + sI] = (on[n] >> (tri(uI) + sI)) & 1u ? A[n][uI] + B[n][sI] : 0;
      for (int c = quarter[n]; c < n_here; c += Q::kQuarters) {
        const uint32_t *cls = st + c * Q::words;
        const uint4 *tp = reinterpret_cast<const uint4 *>(taps + 8 * (gi * Q::group + c));
        const uint4 ta = tp[0], tb = tp[1];
        const uint32_t y[4] = {ta.x, ta.y, ta.z, ta.w};
        const int k = (int)tb.w;   // the same for the whole warp
        {
          const uint32_t x1 = cls[off[0] + 1], a = y[0] >> 24;
#pragma unroll
          for (int r = 0; r < 4; ++r) sum[n][r] = (int)__dp4a(x1, a << (8 * r), (unsigned)sum[n][r]);
        }
#pragma unroll
        for (int uI = 1; uI < 4; ++uI) {
          if (uI > k) break;
          const uint32_t *q1 = cls + off[tri(uI) + 1];
          const uint32_t z1 = cls[off[tri(uI)] + 1], x0 = q1[0], x1 = q1[1];
          const uint32_t t1 = __byte_perm(x0, x1, 0x4300u);
          sum[n][0] = (int)__dp4a(__byte_perm(z1, t1, 0x7600u), y[uI], (unsigned)sum[n][0]);
          sum[n][1] = (int)__dp4a(__byte_perm(z1, x1, 0x5410u), y[uI], (unsigned)sum[n][1]);
          sum[n][2] = (int)__dp4a(__byte_perm(z1, x1, 0x6520u), y[uI], (unsigned)sum[n][2]);
          sum[n][3] = (int)__dp4a(__byte_perm(z1, x1, 0x7630u), y[uI], (unsigned)sum[n][3]);
#pragma unroll
          for (int sI = 2; sI <= uI; ++sI) {
            const uint32_t *q = cls + off[tri(uI) + sI];
            const uint32_t v0 = q[0], v1 = q[1], tw = sI == 3 ? tb.z : uI == 2 ? tb.x : tb.y;
            sum[n][0] = (int)__dp4a(__byte_perm(v0, v1, 0x4321u), tw, (unsigned)sum[n][0]);
            sum[n][1] = (int)__dp4a(__byte_perm(v0, v1, 0x5432u), tw, (unsigned)sum[n][1]);
            sum[n][2] = (int)__dp4a(__byte_perm(v0, v1, 0x6543u), tw, (unsigned)sum[n][2]);
            sum[n][3] = (int)__dp4a(v1, tw, (unsigned)sum[n][3]);
          }
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
