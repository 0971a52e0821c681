// Definitions shared by the per-quartic pipeline (qfs_engine.cuh) and the chain products (qfs_sweep.cuh, qfs_block.cuh):
// block size, device status bits, debug outputs and the static part of the shared memory.
#pragma once
#include <cstddef>
#include <cstdint>
#include "qfs_layout.cuh"

namespace qfs {

constexpr int kThreads = 256;
constexpr int kMaxUparDecl = 8;
constexpr int kMaxStrips = 100;   // strips of a block product (qfs_block.cuh)
constexpr int kMaxSmallStrips = 6;   // strips of one up to f~^p

// Workspace buffers.  Every buffer a chain product reads from is preceded by kGuardWords zero words (the swept
// product reads columns that do not exist from there).  A launch's workspace holds, per CTA, two buffers of
// workspace_stride_words(p) words each, and starts with one guard: buffer k of CTA b begins at word
// kGuardWords + (2b + k) * stride, and its guard is the last kGuardWords words of the stride before it, which
// nothing in the buffer reaches (its contents use at most stride - kGuardWords words).  Each CTA clears
// its two guards when it starts, since an earlier launch with another stride may have left data there.  A buffer
// holds either a padded form of degree up to 4p(p-1) or theta's guarded copy of Delta, which is larger.
constexpr int kGuardWords = 4;
size_t workspace_stride_words(int p);   // qfs_engine.cuh: the larger of a padded degree-D form and theta's copy
inline size_t workspace_words(int64_t ctas, size_t stride) { return kGuardWords + 2 * (size_t)ctas * stride; }

#if defined(__CUDACC__)
__device__ __forceinline__ void cta_buffers(uint32_t *ws, size_t stride, uint32_t *&bufA, uint32_t *&bufB) {
  bufA = ws + kGuardWords + (size_t)blockIdx.x * 2 * stride;
  bufB = bufA + stride;
  if (threadIdx.x < 2 * kGuardWords)
    (threadIdx.x < kGuardWords ? bufA : bufB)[(int)(threadIdx.x % kGuardWords) - kGuardWords] = 0u;
}
#endif

// Status bits (atomicOr into the device status word).
constexpr uint32_t kStatusInexactDivision = 1u;
constexpr uint32_t kStatusTheta = 2u;
constexpr uint32_t kStatusWait = 4u;   // a bounded wait inside a kernel ran out

struct DebugPtrs {
  uint32_t *G;        // padded, degree D: raw G (mod p^2) before the Delta_1 epilogue
  uint32_t *delta;    // padded, degree D: Delta (mod p)
  int32_t *g;         // packed, ld values
  int32_t *iters;     // packed, (max_h-1) x ld
};

// Crews.  A launch over few quartics runs as thread-block clusters: the CTAs of a cluster (a crew, 1, 2, 4 or 8 of them)
// work on one quartic together.  Each forms f^(p-1) for itself; the products of A4 and the theta steps are split, with
// the forms in the first CTA's buffers.  Every CTA of a crew takes the same decisions from the same data.  In a launch over
// several primes the crews take the heavy quartics, then each CTA the rest for itself (joint_items in qfs_engine.cuh).
#if defined(__CUDACC__)
__device__ __forceinline__ int crew_rank() {
  unsigned r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return (int)r;
}
__device__ __forceinline__ int crew_size() {
  unsigned n;
  asm("mov.u32 %0, %%cluster_nctaid.x;" : "=r"(n));
  return (int)n;
}
// Barrier over the crew; writes before it, to shared and global memory, are visible to the whole crew after it.
__device__ __forceinline__ void crew_sync(int crew) {
  if (crew > 1) {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  } else {
    __syncthreads();
  }
}
// The shared-memory address of a variable of this CTA in the CTA of the given rank.
__device__ __forceinline__ uint32_t crew_addr(const void *p, int rank) {
  uint32_t a;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return a;
}
#endif

struct Smem {
  int SW[kSWLen];
  int taps[35];           // coefficients of f, packed order (index tet(uI) + tri(sI) + tI)
  uint32_t tapword[15];   // tap words per (uI, sI) pair: byte k = a(uI, sI, 3-k)
  uint32_t pair_mask;     // bit tri(uI)+sI set iff that pair has a nonzero tap
  int dense_min;          // nonzero tap pairs from which the swept chain (int32 form) runs every pair
  int powp[kMaxP];        // c^p mod p^2
  int slot_tab[2][kMaxUparDecl + 4];  // ring word offsets of the slices a chain round reads (double buffered)
  union {                             // one product form per launch
    uint16_t chunk_tab[32 * 40];      // slice ring: flat chunk index -> (column - s0) << 8 | chunk
    struct {                          // block products
      uint32_t strip_tab[kMaxStrips]; // first item of every strip (block::build_strip_tab)
      uint32_t small_tab[kMaxSmallStrips];   // the same of the products up to f~^p, where they have strips of their own
      int unit_next[2];               // next unit of a product's queue, by the product's parity
      int unit_slot[4][2];            // a team's next unit
    };
  };
  int tile_round, tile_ring;          // chain tile configuration of the current quartic's prime
  int64_t item;
  int flag;
  int task_next;   // swept chain: next task of the current product (work queue shared by the CTA's warps)
  int crew, rank;  // CTAs working on this quartic's products together, and this one's place (1 and 0: alone)
  int task_done;   // swept chain: warps that found the queue empty; the last one resets both counters
  // followed in dynamic shared memory by two byte arrays of ld entries: g (current iterate) and g_next
};

// Dynamic shared memory layout: [Smem][g: ld][g_next: ld][pad to 16 B][chain ring].
__host__ __device__ constexpr size_t ring_offset_for(int max_ld) {
  return (sizeof(Smem) + 2 * (size_t)max_ld + 15) & ~(size_t)15;
}

}  // namespace qfs
