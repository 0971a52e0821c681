// Matrix multiplication mod p (the paper's Sec. 5 workload: square matrices mod 11 of size 5,000 .. 20,000).
// C = A B mod p for A (n x k), B (k x m), C (n x m), all uint8 row-major.
//
// The products run on the fifth-generation tensor cores (tcgen05.mma kind::f8f6f4, accumulators in TMEM), whose 8-bit
// floating-point operands hold small integers exactly: e4m3 has every integer up to 16 and every multiple of 16 up to
// 128.  A residue is taken in its symmetric range, |v| <= p/2, so for p <= 33 it is one e4m3 value; for larger p it is
// split as v = 16 h + l with |16 h| <= 128 and |l| <= 8, two e4m3 planes per operand and four plane products.  The
// float32 accumulator holds integers below 2^24 exactly, and the accumulators are drained, reduced mod p and added up
// as integers before a sum of absolute values could pass that, so the result is exact (the int8 kinds of tcgen05 do
// not exist on sm_103a, and mma.sync's int8 path runs at 1/28 of the rate).
//
// A pack kernel writes A and the transpose of B as K-major planes, K padded with zeros to a multiple of 128 bytes.
// The product kernel is persistent, one CTA per SM: tiles of 128 x 256 outputs, K steps of 128 bytes, brought in by
// TMA (128-byte swizzle) into a ring of stages; one thread issues the MMAs; four warps drain one accumulator of TMEM
// while the other is being filled.
//
// What bounds it: the copies from L2 into shared memory (48 KB per K step of a tile, 512 clocks of MMAs: 96 bytes per clock
// where about 60 arrive in the full waves), a last wave of tiles (800 on 152 SMs: 5.3), and about 20 us of packing at n =
// 5,000, where the tensor pipe is active in 58 % of the product's cycles and DRAM runs at 7 %.  n = m =
// k, mod 11: 132 us at 5,000 and 773 us at 10,000 (1.90 and 2.59 PFLOP/s with the pack), against 1,895 us and 13.9 ms
// by mma.sync m16n8k32 u8, which ran at 0.82 and 0.91 of its own peak; mod 101 and 251 at 5,000: 347 and 360 us.  Up
// to about 512 x 512 x 512 a call takes as long as the host needs to enqueue it (17 to 20 us).  The product kernel
// starts while the pack runs (programmatic dependent launch): 700 x 90 x 3,000 mod 31 took 32.9 us, takes 28.8.
#include <cuda.h>
#include <cuda_runtime.h>

#include <atomic>
#include <cstdint>

#include "qfs_common.cuh"
#include "qfs_matmul.cuh"

namespace qfs {
namespace {

constexpr int kBM = 128, kBN = 256, kBK = 128;   // output tile, and bytes of K per step
constexpr int kTileA = kBM * kBK, kTileB = kBN * kBK;
constexpr int kMMThreads = 192;                  // warps: TMA, MMA, four that drain
constexpr int kPackTile = 64;
constexpr int kRowWords = kBN / 4 + 1;           // a tile's row on its way to an unaligned C: an odd pitch, and a word more to read

__host__ __device__ constexpr int stages_of(int planes) { return 4 / planes; }
__host__ __device__ constexpr size_t ring_bytes(int planes) { return (size_t)stages_of(planes) * planes * (kTileA + kTileB); }
__host__ __device__ constexpr size_t mm_smem(int planes) { return ring_bytes(planes) + 1024 + 4 * kBM * kRowWords; }

// ------------------------------------------------------------------------------------------------ pack
// e4m3 code of an integer with at most four significant bits, |x| <= 128
__device__ __forceinline__ uint32_t e4m3_of(int x) {
  const uint32_t m = (uint32_t)(x < 0 ? -x : x);
  if (m == 0) return 0;
  const int e = 31 - __clz((int)m);
  return (x < 0 ? 0x80u : 0u) | (uint32_t)((e + 7) << 3) | (((m << 3) >> e) & 7u);
}

// Sixteen bytes from p (any alignment), of which the first `have` exist; `all` is the array's byte range.
__device__ __forceinline__ void load16(const uint8_t *p, int have, const uint8_t *lo, const uint8_t *hi,
                                       uint32_t (&w)[4]) {
  const uintptr_t a = reinterpret_cast<uintptr_t>(p) & ~(uintptr_t)3;
  const int sh = 8 * (int)(reinterpret_cast<uintptr_t>(p) & 3);
  if (have == 16 && a >= reinterpret_cast<uintptr_t>(lo) && a + 20 <= reinterpret_cast<uintptr_t>(hi)) {
    const uint32_t *q = reinterpret_cast<const uint32_t *>(a);
    uint32_t x[5];
#pragma unroll
    for (int i = 0; i < 5; ++i) x[i] = q[i];
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(x[i], x[i + 1], sh);
  } else {
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = 0;
#pragma unroll
    for (int i = 0; i < 16; ++i)
      if (i < have) w[i >> 2] |= (uint32_t)p[i] << (8 * (i & 3));
  }
}

// Planes of A (blockIdx.z = 0: rows as they are) and of B^T (blockIdx.z = 1) in 64 x 64 byte tiles; a byte goes through
// a table (its residue mod p, symmetric, as e4m3 codes).
template <int PLANES>
__global__ void __launch_bounds__(256) pack_kernel(const uint8_t *__restrict__ A, const uint8_t *__restrict__ B, int n,
                                                   int m, int k, int kp, int p, uint8_t *__restrict__ Ap,
                                                   uint8_t *__restrict__ Bp) {
  __shared__ uint8_t lut[PLANES][256];
  __shared__ __align__(16) uint32_t t[PLANES][kPackTile][kPackTile / 4 + 1];
  const int tid = threadIdx.x;
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");   // the product's CTAs set themselves up meanwhile
  {
    int v = tid % p;
    if (2 * v > p) v -= p;
    if constexpr (PLANES == 1) {
      lut[0][tid] = (uint8_t)e4m3_of(v);
    } else {
      const int h = (v + 8) >> 4;
      lut[0][tid] = (uint8_t)e4m3_of(16 * h);
      lut[1][tid] = (uint8_t)e4m3_of(v - 16 * h);
    }
  }
  __syncthreads();
  auto code = [&](int pl, uint32_t w) {
    return (uint32_t)lut[pl][w & 255u] | (uint32_t)lut[pl][(w >> 8) & 255u] << 8 |
           (uint32_t)lut[pl][(w >> 16) & 255u] << 16 | (uint32_t)lut[pl][w >> 24] << 24;
  };
  const int r = tid >> 2, seg = 16 * (tid & 3);
  const int kk0 = blockIdx.x * kPackTile;
  if (blockIdx.z == 0) {
    const int i = blockIdx.y * kPackTile + r, kk = kk0 + seg;
    if (i >= n) return;
    const int have = max(0, min(16, k - kk));
    uint32_t w[4];
    load16(A + (size_t)i * k + kk, have, A, A + (size_t)n * k, w);
#pragma unroll
    for (int pl = 0; pl < PLANES; ++pl)
      *reinterpret_cast<uint4 *>(Ap + ((size_t)pl * n + i) * kp + kk) =
          make_uint4(code(pl, w[0]), code(pl, w[1]), code(pl, w[2]), code(pl, w[3]));
  } else {
    const int j0 = blockIdx.y * kPackTile;
    if (j0 >= m) return;
    const int kk = kk0 + r;
    const int have = kk < k ? max(0, min(16, m - (j0 + seg))) : 0;
    uint32_t w[4] = {0, 0, 0, 0};
    if (have > 0) load16(B + (size_t)kk * m + j0 + seg, have, B, B + (size_t)k * m, w);
#pragma unroll
    for (int pl = 0; pl < PLANES; ++pl)
#pragma unroll
      for (int i = 0; i < 4; ++i) t[pl][r][(seg >> 2) + i] = code(pl, w[i]);
    __syncthreads();
    const int j = j0 + r;
    if (j >= m) return;
#pragma unroll
    for (int pl = 0; pl < PLANES; ++pl) {
      const uint8_t *tb = reinterpret_cast<const uint8_t *>(t[pl]);
      uint32_t o[4] = {0, 0, 0, 0};
#pragma unroll
      for (int i = 0; i < 16; ++i)
        o[i >> 2] |= (uint32_t)tb[(seg + i) * (kPackTile + 4) + r] << (8 * (i & 3));
      *reinterpret_cast<uint4 *>(Bp + ((size_t)pl * m + j) * kp + kk0 + seg) = make_uint4(o[0], o[1], o[2], o[3]);
    }
  }
}

// ------------------------------------------------------------------------------------------------ product
struct Maps {
  CUtensorMap a[2], b[2];   // planes of A (n x kp) and of B^T (m x kp)
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void mbar_init(uint64_t *b, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(b)), "r"(count));
}
__device__ __forceinline__ void mbar_expect(uint64_t *b, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(b)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t *b) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(b)) : "memory");
}
// Waits for the phase of the given parity; gives up after kSpins tries or when another warp has (returns false).
constexpr int kSpins = 1 << 22;
__device__ __forceinline__ bool mbar_wait(uint64_t *b, uint32_t parity, volatile int *abort_flag) {
  for (int i = 0; i < kSpins; ++i) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
        : "=r"(done)
        : "r"(smem_u32(b)), "r"(parity)
        : "memory");
    if (done) return true;
    if ((i & 63) == 63 && *abort_flag) return false;
  }
  *abort_flag = 1;
  return false;
}
__device__ __forceinline__ void tma_load(uint32_t dst, const CUtensorMap *map, int x, int y, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(
          dst),
      "l"(map), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}
// K-major operand tile with 128-byte rows and 128-byte swizzle: groups of eight rows are 1,024 bytes apart.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  return (uint64_t)((addr & 0x3FFFFu) >> 4) | (1ull << 16) | ((uint64_t)(1024 >> 4) << 32) | (1ull << 46) | (2ull << 61);
}
// f32 accumulator, e4m3 x e4m3, both K-major, M = kBM, N = kBN
constexpr uint32_t kIdesc = (1u << 4) | ((uint32_t)(kBN / 8) << 17) | ((uint32_t)(kBM / 16) << 24);
__device__ __forceinline__ void mma_f8(uint32_t d, uint64_t a, uint64_t b, uint32_t accumulate) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.b32 q, %4, 0;\n"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, q;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(kIdesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t addr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, "
      "%24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// C, n x m; ksteps: K steps of kBK bytes; chunk: K steps between drains; vec: bytes a store to C may take at once.
template <int PLANES>
__global__ void __launch_bounds__(kMMThreads, 1)
    product_kernel(const __grid_constant__ Maps maps, uint8_t *__restrict__ C, int n, int m, int ksteps, int chunk,
                   int p, uint32_t magic, uint32_t bias, int vec, uint32_t *status) {
  constexpr int kStages = stages_of(PLANES);
  constexpr uint32_t kStageBytes = PLANES * (kTileA + kTileB);
  extern __shared__ uint8_t smem_raw[];
  __shared__ uint64_t full[kStages], empty[kStages], tfull[2], tempty[2], mma_done;
  __shared__ uint32_t tmem_base;
  __shared__ int abort_flag;
  volatile int no_abort = 0;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t stage0 = (smem_u32(smem_raw) + 1023u) & ~1023u;   // swizzled tiles start on 1,024-byte boundaries
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 512;" ::"r"(smem_u32(&tmem_base)) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  } else if (threadIdx.x == 32) {
    for (int s = 0; s < kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int a = 0; a < 2; ++a) {
      mbar_init(&tfull[a], 1);
      mbar_init(&tempty[a], 4);
    }
    mbar_init(&mma_done, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base;
  asm volatile("griddepcontrol.wait;" ::: "memory");   // the planes are packed, and whatever read C is done
  const int tiles_n = (n + kBM - 1) / kBM, tiles = tiles_n * ((m + kBN - 1) / kBN);

  if (warp == 0) {
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
        const int i0 = (tile % tiles_n) * kBM, j0 = (tile / tiles_n) * kBN;
        for (int ks = 0; ks < ksteps; ++ks, ++it) {
          const uint32_t s = it % kStages;
          if (!(ok = mbar_wait(&empty[s], ((it / kStages) & 1u) ^ 1u, &abort_flag))) break;
          mbar_expect(&full[s], kStageBytes);
          const uint32_t st = stage0 + s * kStageBytes;
#pragma unroll
          for (int pl = 0; pl < PLANES; ++pl) {
            tma_load(st + pl * kTileA, &maps.a[pl], ks * kBK, i0, &full[s]);
            tma_load(st + PLANES * kTileA + pl * kTileB, &maps.b[pl], ks * kBK, j0, &full[s]);
          }
        }
      }
      // the copies in flight land before the CTA's shared memory is given up, also after a wait that ran out
      for (uint32_t k = it > (uint32_t)kStages ? it - kStages : 0; !ok && k < it; ++k)
        for (int i = 0; i < kSpins; ++i) {
          uint32_t done;
          asm volatile(
              "{\n.reg .pred q;\nmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\nselp.u32 %0, 1, 0, q;\n}\n"
              : "=r"(done)
              : "r"(smem_u32(&full[k % kStages])), "r"((k / kStages) & 1u)
              : "memory");
          if (done) break;
        }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      uint32_t it = 0, cc = 0;
      bool ok = true;
      for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x)
        for (int k0 = 0; k0 < ksteps && ok; k0 += chunk, ++cc) {
          const uint32_t a = cc & 1u;
          if (!(ok = mbar_wait(&tempty[a], ((cc >> 1) & 1u) ^ 1u, &abort_flag))) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const int k1 = min(ksteps, k0 + chunk);
          for (int ks = k0; ks < k1; ++ks, ++it) {
            const uint32_t s = it % kStages;
            if (!(ok = mbar_wait(&full[s], (it / kStages) & 1u, &abort_flag))) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t st = stage0 + s * kStageBytes;
#pragma unroll
            for (int pa = 0; pa < PLANES; ++pa)
#pragma unroll
              for (int pb = 0; pb < PLANES; ++pb) {
                const uint64_t da = smem_desc(st + pa * kTileA), db = smem_desc(st + PLANES * kTileA + pb * kTileB);
#pragma unroll
                for (int kk = 0; kk < kBK / 32; ++kk)   // 32 bytes of K per MMA
                  mma_f8(tmem + a * kBN, da + 2 * kk, db + 2 * kk, !(ks == k0 && pa == 0 && pb == 0 && kk == 0));
              }
            mma_commit(&empty[s]);
          }
          mma_commit(&tfull[a]);
        }
      mma_commit(&mma_done);   // no MMA is left when the CTA gives up its memory, also after a wait that ran out
      mbar_wait(&mma_done, 0, &no_abort);
    }
  } else {
    const int quad = warp & 3;   // the 32 lanes of TMEM this warp may read
    uint32_t cc = 0;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += gridDim.x) {
      const int i = (tile % tiles_n) * kBM + 32 * quad + lane, j0 = (tile / tiles_n) * kBN;
      const int len = min(kBN, m - j0);
      uint32_t res[kBN / 4];   // residues of the chunks so far, four to a word
#pragma unroll
      for (int w = 0; w < kBN / 4; ++w) res[w] = 0;
      for (int k0 = 0; k0 < ksteps; k0 += chunk, ++cc) {
        const uint32_t a = cc & 1u;
        ok = mbar_wait(&tfull[a], (cc >> 1) & 1u, &abort_flag);
        if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int c = 0; c < kBN; c += 32) {
          if (c >= len) continue;   // columns past the end of C
          uint32_t v[32];
          tmem_ld32(tmem + ((uint32_t)(32 * quad) << 16) + a * kBN + c, v);
#pragma unroll
          for (int e = 0; e < 32; ++e) {
            const int w = (c + e) >> 2, sh = 8 * (e & 3);
            // x + bias >= 0 (bias: the multiple of p from 2^24 on); the quotient estimate is at most one too large
            const uint32_t x = (uint32_t)__float2int_rn(__uint_as_float(v[e])) + bias + ((res[w] >> sh) & 255u);
            const uint32_t rr = x - __umulhi(x, magic) * (uint32_t)p;
            const uint32_t y = min(rr, rr + (uint32_t)p);
            res[w] = (res[w] & ~(255u << sh)) | (y << sh);
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&tempty[a]);
      }
      if (!ok) break;
      if (vec >= 4) {
        if (i < n) {
          uint8_t *row = C + (size_t)i * m + j0;
#pragma unroll
          for (int w = 0; w < kBN / 4; w += 4) {
            if (vec >= 16 && 4 * w + 16 <= len) {
              *reinterpret_cast<uint4 *>(row + 4 * w) = make_uint4(res[w], res[w + 1], res[w + 2], res[w + 3]);
              continue;
            }
#pragma unroll
            for (int x = w; x < w + 4; x += 2) {
              if (vec >= 8 && 4 * x + 8 <= len) {
                *reinterpret_cast<uint2 *>(row + 4 * x) = make_uint2(res[x], res[x + 1]);
                continue;
              }
#pragma unroll
              for (int y = x; y < x + 2; ++y)
                if (4 * y < len) *reinterpret_cast<uint32_t *>(row + 4 * y) = res[y];   // (len: a multiple of four)
            }
          }
        }
        continue;
      }
      // Rows of C at odd addresses: the warp's 32 rows go through shared memory and out as aligned words, a row (several
      // rows, where they are short) at a time, instead of as single bytes of 32 rows at a time.  mod 31, n = m = 4,097,
      // k = 129: 169 us by bytes, 43 so (rows of 4,096: 29).
      uint32_t *rows = reinterpret_cast<uint32_t *>(smem_raw + (stage0 - smem_u32(smem_raw)) + ring_bytes(PLANES)) +
                       32 * quad * kRowWords;
#pragma unroll
      for (int w = 0; w < kBN / 4; ++w)
        if (4 * w < len) rows[lane * kRowWords + w] = res[w];
      __syncwarp();
      int per_row = 32;   // lanes of a row
      while (per_row > 1 && 4 * (per_row / 2) >= len + 3) per_row /= 2;
      const int sub = lane & (per_row - 1), step = 32 / per_row, n_rows = min(32, n - (i - lane));
#pragma unroll 4
      for (int r = lane / per_row; r < n_rows; r += step) {
        const uint32_t *src = rows + r * kRowWords;
        const uint8_t *bytes = reinterpret_cast<const uint8_t *>(src);
        uint8_t *dst = C + (size_t)(i - lane + r) * m + j0;
        const int head = min(len, (int)(-reinterpret_cast<uintptr_t>(dst) & 3)), words = (len - head) >> 2;
        const int edges = len - 4 * words;   // bytes before the first aligned word and after the last
        for (int w = sub; w < words; w += per_row)   // bytes head + 4w .. head + 4w + 3
          *reinterpret_cast<uint32_t *>(dst + head + 4 * w) = __funnelshift_r(src[w], src[w + 1], 8 * head);
        for (int e = sub; e < edges; e += per_row) {
          const int at = e < head ? e : e + 4 * words;
          dst[at] = bytes[at];
        }
      }
      __syncwarp();   // the next tile overwrites the rows
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) {
    if (abort_flag && lane == 0) atomicOr(status, kStatusWait);
    __syncwarp();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 512;" ::"r"(tmem));
  }
}

using EncodeTiled = CUresult (*)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                 const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                 CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

// The driver's tensor-map encoder, looked up once.
EncodeTiled encoder() {
  static EncodeTiled fn = [] {
    void *f = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      f = nullptr;
    return reinterpret_cast<EncodeTiled>(f);
  }();
  return fn;
}

// Tensor map of a plane of `rows` rows of kp bytes, in boxes of box_rows x kBK; rows past the end read as zeros.
bool plane_map(CUtensorMap *map, const uint8_t *base, int rows, int kp, int box_rows) {
  const cuuint64_t dims[2] = {(cuuint64_t)kp, (cuuint64_t)rows}, strides[1] = {(cuuint64_t)kp};
  const cuuint32_t box[2] = {kBK, (cuuint32_t)box_rows}, step[2] = {1, 1};
  return encoder()(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<uint8_t *>(base), dims, strides, box, step,
                   CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                   CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

constexpr int kMaxOnePlane = 33;   // |v| <= 16: one e4m3 value
int planes_of(int p) { return p <= kMaxOnePlane ? 1 : 2; }
size_t plane_stride(size_t rows, size_t kp, int planes) { return (rows * kp * planes + 1023) & ~(size_t)1023; }

template <int PLANES>
cudaError_t launch(int p, int n, int m, int k, const uint8_t *A, const uint8_t *B, uint8_t *C, uint8_t *scratch, int sms,
                   uint32_t *status, cudaStream_t st) {
  const int kp = (k + kBK - 1) / kBK * kBK;
  uint8_t *Ap = scratch, *Bp = scratch + plane_stride(n, kp, PLANES);
  Maps maps;
  if (!encoder()) return cudaErrorNotSupported;
  for (int pl = 0; pl < PLANES; ++pl)
    if (!plane_map(&maps.a[pl], Ap + (size_t)pl * n * kp, n, kp, kBM) ||
        !plane_map(&maps.b[pl], Bp + (size_t)pl * m * kp, m, kp, kBN))
      return cudaErrorInvalidValue;
  if (PLANES == 1) {   // (not read)
    maps.a[1] = maps.a[0];
    maps.b[1] = maps.b[0];
  }
  const dim3 pgrid(kp / kPackTile, (unsigned)((n > m ? n : m) + kPackTile - 1) / kPackTile, 2);
  pack_kernel<PLANES><<<pgrid, 256, 0, st>>>(A, B, n, m, k, kp, p, Ap, Bp);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  // K steps between drains: sums of absolute values of the plane products stay at most 2^24
  const long long mag = PLANES == 1 ? p / 2 : p / 2 + 16;
  long long chunk = (1ll << 24) / (mag * mag * kBK);
  if (chunk > kp / kBK) chunk = kp / kBK;
  const uint32_t magic = (uint32_t)((0x100000000ull + (uint64_t)p - 1) / (uint64_t)p);
  const uint32_t bias = (uint32_t)(((1 << 24) + p - 1) / p * p);
  const uintptr_t al = reinterpret_cast<uintptr_t>(C) | (uintptr_t)m;
  const int vec = (al & 15) == 0 ? 16 : (al & 7) == 0 ? 8 : (al & 3) == 0 ? 4 : 1;
  // the attribute is set once per device: a small product takes as long as the host needs to enqueue it (17 us)
  static std::atomic<uint64_t> attribute_set{0};
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  const uint64_t bit = 1ull << (dev & 63);
  if (!(attribute_set.load() & bit)) {
    e = cudaFuncSetAttribute(product_kernel<PLANES>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mm_smem(PLANES));
    if (e != cudaSuccess) return e;
    attribute_set.fetch_or(bit);
  }
  const long long tiles = (long long)((n + kBM - 1) / kBM) * ((m + kBN - 1) / kBN);
  const int grid = (int)(tiles < sms ? tiles : sms);
  // The product may start while the pack runs; it waits for it after setting up its barriers and TMEM.
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kMMThreads);
  cfg.dynamicSmemBytes = mm_smem(PLANES);
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, product_kernel<PLANES>, maps, C, n, m, kp / kBK, (int)chunk, p, magic, bias, vec, status);
}

}  // namespace

size_t matmul_scratch_bytes(int p, int n, int m, int k) {
  const size_t kp = ((size_t)k + kBK - 1) / kBK * kBK;
  return plane_stride(n, kp, planes_of(p)) + plane_stride(m, kp, planes_of(p)) + 1024;
}

cudaError_t matmul_mod_launch(int p, int n, int m, int k, const uint8_t *A, const uint8_t *B, uint8_t *C,
                              uint8_t *scratch, int sms, uint32_t *status, cudaStream_t st) {
  return planes_of(p) == 1 ? launch<1>(p, n, m, k, A, B, C, scratch, sms, status, st)
                           : launch<2>(p, n, m, k, A, B, C, scratch, sms, status, st);
}

}  // namespace qfs
