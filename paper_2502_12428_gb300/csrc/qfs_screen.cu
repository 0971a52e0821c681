// Height-1 screen of a batch (Algorithm 3, first test; Fedder's criterion, Sec. 3): h = 1 iff the coefficient of
// (x1 x2 x3 x4)^(p-1) in f^(p-1) is nonzero mod p.  Most quartics stop there (about 84 % of dense quartics at
// p = 7), so the batch is screened before the persistent launch, one warp per quartic, and only the survivors reach
// the CTA-wide pipeline (which repeats the test on its own f^(p-1) mod p^2, with the same outcome).
//
// With k = (p-1)/2, f^(p-1) = F * F for F = f^k, so the coefficient is sum_a F[a] F[(p-1)1 - a] over the
// monomials a of degree 2(p-1) whose four exponents are all <= p-1 (exactly the a for which (p-1)1 - a is a
// monomial).  F is formed mod p by k-1 products with f in the warp's shared memory, by rows (qfs_rows.cuh): one output
// word per lane, the taps by dp4a.  Bound by instruction issue.  262,144 quartics at p = 7 took 3.5 ms with
// one output and 35 byte loads at a time, 0.74 ms this way.
#include <cuda_runtime.h>

#include "qfs_layout.cuh"
#include "qfs_rows.cuh"
#include "qfs_screen.cuh"

namespace qfs {
namespace {

constexpr int kScreenWarps = kScreenThreads / 32;

// One warp's region for primes up to max_p, in words: the tap words, f (35 bytes), and two forms of degree 2(p-1) by rows.
constexpr int kTapWords = 16, kFWords = 12;
__host__ __device__ constexpr int screen_form_words(int p) {
  return (tri(2 * (p - 1) + 1) + 1) * rows::pitch_of(2 * (p - 1));
}
__host__ __device__ constexpr int screen_warp_words(int max_p) { return kTapWords + kFWords + 2 * screen_form_words(max_p); }
// words of the list of output words, shared by the CTA's warps
__host__ __device__ constexpr int screen_item_words(int max_p) { return (rows::items_of(2 * (max_p - 1)) + 1) / 2; }

// Screens one row with the calling warp; returns -1 (a coefficient >= p), 1 (height 1) or 0 (survivor), same in
// every lane.  fresh: the region last held forms of another prime (or nothing).
template <int P>
__device__ int screen_row(const uint8_t *__restrict__ f35, uint32_t *wsm, const uint16_t *items, bool fresh, int lane) {
  constexpr int k = (P - 1) / 2, m = 2 * (P - 1), pitch = rows::pitch_of(m), form = screen_form_words(P);
  rows::TapWords &T = *reinterpret_cast<rows::TapWords *>(wsm);
  uint8_t *f = reinterpret_cast<uint8_t *>(wsm + kTapWords);
  uint32_t *A = wsm + kTapWords + kFWords + pitch, *B = A + form;   // row 0; the words a row does not use stay zero
  if (fresh)
    for (int i = lane; i < 2 * form; i += 32) wsm[kTapWords + kFWords + i] = 0u;
  int bad = 0;
  for (int i = lane; i < 35; i += 32) {
    const int a = f35[i];
    bad |= a >= P;
    f[i] = (uint8_t)a;
  }
  if (__any_sync(0xffffffffu, bad)) return -1;
  __syncwarp();
  if (lane < 15) T.tw[lane] = rows::tap_word(f, lane);
  if (lane == 15) T.a44 = f[34];
  // F = f^k: the rows of f, then k - 1 products
  uint32_t *F = A, *next = B;
  for (int i = lane; i < 35; i += 32) {
    int u, s, t;
    decode_packed(i, u, s, t, 4);
    reinterpret_cast<uint8_t *>(F + (tri(u) + s) * pitch + 1)[t] = f[i];
  }
  __syncwarp();
  int n_items = rows::items_of(4);
#pragma unroll 1
  for (int j = 1; j < k; ++j) {
#pragma unroll
    for (int v = 1; v <= 4; ++v) n_items += rows::words_below(4 * j + v + 1);
    for (int i = lane; i < n_items; i += 32) {
      int u, s, w;
      rows::item_of(items, i, u, s, w);
      uint32_t g[4];
      rows::word_sums<pitch>(F, 4 * j, T, u, s, w, g);
      next[(tri(u) + s) * pitch + 1 + w] = g[0] % P | (g[1] % P) << 8 | (g[2] % P) << 16 | (g[3] % P) << 24;
    }
    __syncwarp();
    uint32_t *t = F;
    F = next;
    next = t;
  }
  // coefficient of (x1 x2 x3 x4)^(p-1) in F * F, one row (u, s) per lane
  int acc = 0;
  int u = (isqrt(8 * lane + 1) - 1) >> 1, s = lane - tri(u);
  for (int row = lane; row < tri(m + 1); row += 32, s += 32) {
    while (s > u) s -= ++u;
    if (m - u > P - 1 || u - s > P - 1) continue;
    const uint8_t *x = reinterpret_cast<const uint8_t *>(F + (tri(u) + s) * pitch + 1);
    const int ub = 3 * (P - 1) - u, sb = 2 * (P - 1) - s;
    const uint8_t *y = reinterpret_cast<const uint8_t *>(F + (tri(ub) + sb) * pitch + 1) + (P - 1);
    const int t_hi = min(s, P - 1);
    for (int t = max(0, s - (P - 1)); t <= t_hi; ++t) acc += (int)x[t] * (int)y[-t];
  }
  acc = __reduce_add_sync(0xffffffffu, acc);
  return (acc % P) != 0 ? 1 : 0;
}

// GROUPED: survivors are listed group by group (a kernel of its own: with both lists in one, a row at p = 11 takes 3 us
// more).
template <bool GROUPED>
__global__ void __launch_bounds__(kScreenThreads) screen_kernel(const __grid_constant__ FusedParams prm, int max_p,
                                                                int64_t *list, unsigned long long *n_list) {
  extern __shared__ __align__(16) uint32_t smem[];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint16_t *items = reinterpret_cast<uint16_t *>(smem);
  uint32_t *wsm = smem + screen_item_words(max_p) + (size_t)warp * screen_warp_words(max_p);
  rows::build_items(items, 2 * (max_p - 1));
  if (GROUPED && blockIdx.x == 0 && (int)threadIdx.x < prm.n_groups)
    n_list[kMaxGroups + threadIdx.x] = (unsigned long long)prm.g[threadIdx.x].item_begin;
  __syncthreads();
  const int64_t stride = (int64_t)gridDim.x * kScreenWarps;
  int last_p = 0;   // prime of the forms in the warp's region
  for (int64_t item = (int64_t)blockIdx.x * kScreenWarps + warp; item < prm.n_items; item += stride) {
    int gi = 0;
    while (gi + 1 < prm.n_groups && item >= prm.g[gi + 1].item_begin) ++gi;
    const FusedGroup &G = prm.g[gi];
    const int64_t row = item - G.item_begin;
    const uint8_t *f = G.coeffs + 35 * row;
    const bool fresh = G.p != last_p;
    last_p = G.p;
    int r;
    switch (G.p) {
      case 3: r = screen_row<3>(f, wsm, items, fresh, lane); break;
      case 5: r = screen_row<5>(f, wsm, items, fresh, lane); break;
      case 7: r = screen_row<7>(f, wsm, items, fresh, lane); break;
      case 11: r = screen_row<11>(f, wsm, items, fresh, lane); break;
      default: r = screen_row<13>(f, wsm, items, fresh, lane); break;
    }
    if (lane == 0) {
      if (r != 0) G.heights[row] = (int8_t)r;
      else if (GROUPED) list[G.item_begin + (int64_t)atomicAdd(n_list + gi, 1ull)] = item;
      else list[atomicAdd(n_list, 1ull)] = item;
    }
    __syncwarp();
  }
}

}  // namespace

size_t screen_smem_bytes(int max_p) {
  return sizeof(uint32_t) * ((size_t)screen_item_words(max_p) + (size_t)kScreenWarps * screen_warp_words(max_p));
}

cudaError_t screen_launch(const FusedParams &prm, int max_p, int64_t *list, unsigned long long *n_list,
                          int grid_ctas, cudaStream_t st) {
  const size_t smem = screen_smem_bytes(max_p);
  const auto kernel = prm.grouped ? screen_kernel<true> : screen_kernel<false>;
  cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  kernel<<<grid_ctas, kScreenThreads, smem, st>>>(prm, max_p, list, n_list);
  return cudaGetLastError();
}

}  // namespace qfs
