// Small forms by rows, for kernels that keep every form of a quartic in shared memory (qfs_screen.cu, qfs_reduced.cu).
//
// A form of degree m is stored by rows (u, s) in the coordinates of qfs_layout.cuh, row tri(u) + s, one byte per
// coefficient t = 0 .. s, at a fixed pitch that starts with a zero word; row -1 is zero, and a row's bytes past its end
// are zero.  A product with a quartic takes one output word, four outputs, at a time: its 15 tap pairs (uI, sI) read two
// words of one row each, rows beyond the cone read row -1, and the bytes meet the taps by dp4a as in qfs_block.cuh.  An item is
// one output word (u, s, w), u | s << 5 | w << 10; the items in order of u serve every degree with a prefix.
#pragma once
#include <cstdint>
#include "qfs_layout.cuh"

namespace qfs {
namespace rows {

// words of a row of a form whose degree is at most m
__host__ __device__ constexpr int pitch_of(int m) { return m / 4 + 2; }
// output words of a form of degree m: sum over u <= m of E(u + 1), E(n) = sum_{s < n} (s/4 + 1) for n = 4a + b
__host__ __device__ constexpr int words_below(int n) { return ((n >> 2) + 1) * (2 * (n >> 2) + (n & 3)); }
__host__ __device__ constexpr int items_of(int m) {
  int n = 0;
  for (int u = 0; u <= m; ++u) n += words_below(u + 1);
  return n;
}

// The items of degree m into `items`, by the calling block; the caller synchronises.
__device__ __forceinline__ void build_items(uint16_t *items, int m) {
  for (int row = threadIdx.x; row < tri(m + 1); row += blockDim.x) {
    int u = (isqrt(8 * row + 1) - 1) >> 1;
    while (tri(u + 1) <= row) ++u;
    while (u > 0 && tri(u) > row) --u;
    const int s = row - tri(u);
    int at = words_below(s);
    for (int v = 0; v < u; ++v) at += words_below(v + 1);
    for (int w = 0; w <= s >> 2; ++w) items[at + w] = (uint16_t)(u | s << 5 | w << 10);
  }
}
__device__ __forceinline__ void item_of(const uint16_t *items, int i, int &u, int &s, int &w) {
  const int x = items[i];
  u = x & 31;
  s = (x >> 5) & 31;
  w = x >> 10;
}

// Taps of a quartic: tw at tri(uI) + sI, byte k: the tap (uI, sI, 3 - k); a44: the tap (4, 4, 4).
struct TapWords {
  uint32_t tw[15], a44;
};
// Tap word pi of the 35 taps `a` (packed order).
template <typename T>
__device__ __forceinline__ uint32_t tap_word(const T *a, int pi) {
  const int uI = pi >= 10 ? 4 : pi >= 6 ? 3 : pi >= 3 ? 2 : pi >= 1 ? 1 : 0, sI = pi - tri(uI);
  uint32_t w = 0;
  for (int t = 0; t <= sI && t < 4; ++t) w |= (uint32_t)a[tet(uI) + tri(sI) + t] << (8 * (3 - t));
  return w;
}

// The four sums of output word w of row (u, s) of the product of `in` (row 0; degree m) with the taps.
template <int PITCH>
__device__ __forceinline__ void word_sums(const uint32_t *in, int m, const TapWords &T, int u, int s, int w,
                                          uint32_t (&acc)[4]) {
#pragma unroll
  for (int r = 0; r < 4; ++r) acc[r] = 0;
#pragma unroll
  for (int uI = 0; uI < 5; ++uI) {
    const int u2 = u - uI;
    if (u2 < 0 || u2 > m) continue;
    const uint32_t *slice = in + (tri(u2) + s) * PITCH + w;
#pragma unroll
    for (int sI = 0; sI <= uI; ++sI) {
      const int s2 = s - sI;
      const uint32_t *q = s2 >= 0 && s2 <= u2 ? slice - sI * PITCH : in - PITCH;
      const uint32_t x1 = q[1], tw = T.tw[tri(uI) + sI];
      if (sI == 0) {
        const uint32_t a = tw >> 24;
#pragma unroll
        for (int r = 0; r < 4; ++r) acc[r] = __dp4a(x1, a << (8 * r), acc[r]);
      } else {
        const uint32_t x0 = q[0];
        acc[0] = __dp4a(__byte_perm(x0, x1, 0x4321u), tw, acc[0]);
        acc[1] = __dp4a(__byte_perm(x0, x1, 0x5432u), tw, acc[1]);
        acc[2] = __dp4a(__byte_perm(x0, x1, 0x6543u), tw, acc[2]);
        acc[3] = __dp4a(x1, tw, acc[3]);
        if (sI == 4)
#pragma unroll
          for (int r = 0; r < 4; ++r) acc[r] = __dp4a(x0, T.a44 << (8 * r), acc[r]);
      }
    }
  }
}

}  // namespace rows
}  // namespace qfs
