// One product of the chain, out = in * f~ (mod p^2), by strips of output columns and blocks of four output slices
// (dp4a form).  Algorithm 1 needs lift(g)^p mod p^2; the chain forms it as f~^(p(p-1)) one multiplication by f~ at a
// time (see qfs_engine.cuh), and this file is that multiplication.
//
// Work item = one half-chunk of an output column: column s, outputs t = 8h .. 8h+7 (column s has s/8 + 1 of them).
// A strip is as many consecutive items as a team has threads, one per thread; the team takes it through output
// slices in blocks of four, u0 .. u0+3.  A block's 32 sums per thread are fed by the input slices u0-4 .. u0+3 (tap
// pair uI = u - v), each of which contributes its columns s - sI, sI <= uI.  Nothing is carried from block to block,
// so a block is straight-line code with every register index fixed, and a strip can be cut anywhere: a unit of work
// is a segment of a strip, and the teams of a CTA take the units of a product from a queue.
//
// The strip's columns of the input slices are staged in shared memory by 16-byte cp.async, four slices (a group) at
// a time: block b of a unit reads groups b and b + 1, and the group after them (or the next unit's first one) is in
// flight meanwhile, so that a whole block's arithmetic covers its latency.  Columns beyond the input's cone, slices
// before the first and the chunk before the strip's first column hold zeros, so that no read of a block needs a
// bounds check.  One barrier of the team per block.
//
// Eleven dp4a per output for its 35 taps.  A window is four bytes of input for the output (u, s, t):
//   Y   in_4(t-4), in_0(t), in_1(t-1), in_1(t)    the taps of (uI, 0) and (uI, 1), and tap (4, 4, 4)
//   Wc  in_c(t-3) .. in_c(t), c = 2, 3, 4         the taps of (uI, c)
// (in_c: column s - c of the input slice), so uI = 1 .. 4 take 1, 2, 3 and 4 products; uI = 0 has the one tap
// in_0(t), a product of the loaded word with the tap shifted to byte r.  The windows of a slice serve every output
// slice of the block it feeds: 5.5 byte permutes per output.
//
// What bounds it: instruction issue.  About 30 instructions per output, issued 63 % of the time with the 16 warps
// that 128 registers allow; dp4a runs at half the issue rate, so the eleven products alone are 22 cycles.  Measured on
// one GB300, every product up to f~^(p(p-1)): 12.5 us per quartic at p = 7 and 1.20 at p = 5, against 16.3 and 1.50
// by sweeps of single lanes over global memory with five live accumulator sets (37 instructions per output, issued
// 53 % of the time).  Tried on the way, at p = 7: the same blocks with loads from global memory (19 us, each slice
// waits for its first touch), whole strips by teams of 256, 128 and 64 threads (14.8, 13.8 and 13.0 us: a small
// team's short strips leave fewer threads waiting for their first slice), the products of zero taps left out behind
// warp-uniform branches (13.2 us on quartics of eight terms: the branches cost more than the products), and three
// CTAs per SM (15 us: 80 registers spill).
#pragma once
#include <cstdint>
#include "qfs_common.cuh"
#include "qfs_sweep.cuh"

namespace qfs {

__device__ __forceinline__ void cp_async16(uint32_t *smem, const uint32_t *gmem, bool valid) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(valid ? 16 : 0));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_group 0;\n" ::); }

namespace block {

constexpr int kSlices = 4;   // output slices of a block, input slices of a group
constexpr int kGroups = 3;   // staged groups of a team: two being read, one in flight
// Threads of a team: the strips of a small team are short, which leaves fewer threads waiting for the strip's later
// columns; at p >= 11 the rings of several teams would not fit in shared memory.  The products up to f~^p (SMALL, degree
// 4p at most) fit four teams at every prime, and one team of 256 has a single strip of them to do: f^(p-1) takes
// 133 us by four teams at p = 11 and 233 by one.
constexpr int kSmallTeam = 64;
__host__ __device__ constexpr int team_threads(int p) { return p <= 7 ? kSmallTeam : kThreads; }
// whether a prime's small products run by other teams than its long ones
__host__ __device__ constexpr bool small_apart(int p) { return team_threads(p) != kSmallTeam; }

// First item of every strip of the longest product, and of the strip after it: column | half-chunk << 16.
__device__ __forceinline__ void build_strip_tab(int p, Smem &sm) {
  static_assert(half_prefix(kMaxD + 1) / team_threads(kMaxP) + 2 <= kMaxStrips, "strips of the largest prime");
  static_assert(half_prefix(4 * kMaxP + 1) / kSmallTeam + 2 <= kMaxSmallStrips, "strips of its small products");
  auto build = [](uint32_t *tab, int team, int degree) {
    const int n = half_prefix(degree + 1) / team + 2;
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
      int s, h;
      decode_half(k * team, s, h);
      tab[k] = (uint32_t)s | ((uint32_t)h << 16);
    }
  };
  build(sm.strip_tab, team_threads(p), 4 * p * (p - 1));
  if (small_apart(p)) build(sm.small_tab, kSmallTeam, 4 * p);
}

// Columns s_lo .. s_hi of strip k of a product of degree m_out, staged from column c_lo; h_lo: its first half-chunk.
struct Strip {
  int s_lo, h_lo, s_hi, c_lo;
};
__device__ __forceinline__ Strip strip_at(const uint32_t *tab, int k, int m_out) {
  const uint32_t a = tab[k], b = tab[k + 1];
  Strip S;
  S.s_lo = (int)(a & 0xFFFFu);
  S.h_lo = (int)(a >> 16);
  S.s_hi = min((int)(b & 0xFFFFu) - ((b >> 16) == 0), m_out);
  S.c_lo = max(S.s_lo - 4, 0);
  return S;
}

// Words of one staged slice (a zero chunk, then the strip's columns) that every strip of every product up to degree D
// fits in: strips start at multiples of a team's items and a longer product only adds columns at the end, so the
// strips of the longest form cover all.
__host__ __device__ constexpr int slice_stride(int D, int team) {
  int best = 0, s_lo = 0, first = 0;   // first: items before column s_lo
  for (int i0 = 0; i0 < half_prefix(D + 1); i0 += team) {
    while (first + half_chunks_of(s_lo) <= i0) first += half_chunks_of(s_lo++);
    int s_hi = s_lo;
    while (s_hi < D && half_prefix(s_hi + 1) < i0 + team) ++s_hi;
    const int words = 4 + colw(s_hi + 1) - colw(s_lo < 4 ? 0 : s_lo - 4);
    best = words > best ? words : best;
  }
  return best;
}
template <int P, bool SMALL>
struct Ring {
  static constexpr int team = SMALL ? kSmallTeam : team_threads(P);
  static constexpr int stride = slice_stride(SMALL ? 4 * P : 4 * P * (P - 1), team);   // words between the slices of a group
  static constexpr int group = kSlices * stride;             // words of a group
  static constexpr int words = kGroups * group;              // words of a team's ring
};

// Per-thread state of one strip.
struct Lane {
  int s, h;
  uint32_t off[5];   // byte offset of input column s - sI, half-chunk h, in a staged slice
  uint32_t *out;     // output half-chunk, less the slice's offset
  int s_min;         // first output slice of this thread (past every slice if the item does not exist)
  int s_pad1, s_pad2;   // first slice whose padding half-chunks after the item (one, two) this thread clears
};

// Words 2h-1, 2h, 2h+1 of one input column.
struct Col {
  uint32_t w[3];
};
__device__ __forceinline__ Col load_col(const char *q) {
  const uint2 x = *reinterpret_cast<const uint2 *>(q);
  return Col{{*reinterpret_cast<const uint32_t *>(q - 4), x.x, x.y}};
}

struct Taps {
  uint32_t y[5];           // byte 0: a(4,4,4) (uI = 4 only), 1: a(uI,0,0), 2: a(uI,1,1), 3: a(uI,1,0); uI = 1 .. 4
  uint32_t w[3][5];        // w[c-2][uI], byte k: a(uI, c, 3-k); uI = c .. 4
  uint32_t a00[4];         // a(0,0,0) in byte r
};

// Windows Wc of word q: out[r], r = 0 .. 3.
__device__ __forceinline__ void windows(const Col &x, int q, uint32_t *out) {
  out[0] = __byte_perm(x.w[q], x.w[q + 1], 0x4321u);
  out[1] = __byte_perm(x.w[q], x.w[q + 1], 0x5432u);
  out[2] = __byte_perm(x.w[q], x.w[q + 1], 0x6543u);
  out[3] = x.w[q + 1];
}

// The columns of input slice v = u0 - 4 + K that a block needs: sI <= the largest uI it takes part in.
template <int STRIDE, int K>
__device__ __forceinline__ void load_slice(const char *group, const Lane &L, Col (&x)[5]) {
  constexpr int u_hi = K < 3 ? 4 : 7 - K;
#pragma unroll
  for (int c = 0; c <= u_hi; ++c) x[c] = load_col(group + L.off[c] + (K & 3) * 4 * STRIDE);
}

// Input slice v = u0 - 4 + K of a block into the sums of the output slices it feeds (j with uI = j + 4 - K in 0..4).
template <int K>
__device__ __forceinline__ void slice_macs(const Col (&x)[5], const Taps &T, uint32_t (&acc)[kSlices][8]) {
  constexpr int j_lo = K > 4 ? K - 4 : 0, j_hi = K < 3 ? K : 3;
  constexpr int u_hi = j_hi + 4 - K;   // largest uI (and largest column) this slice takes part in
  if constexpr (K >= 4) {   // uI = 0 for j = K - 4
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[K - 4][e] = __dp4a(x[0].w[(e >> 2) + 1], T.a00[e & 3], acc[K - 4][e]);
  }
  if constexpr (u_hi >= 1) {
    uint32_t Y[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const uint32_t x0 = x[0].w[q + 1], x1 = x[1].w[q + 1], x4 = x[4].w[q];
      const uint32_t t1 = __byte_perm(x[1].w[q], x1, 0x4300u);
      if constexpr (u_hi == 4) {
        const uint32_t c01 = __byte_perm(x4, x0, 0x5140u), c23 = __byte_perm(x4, x0, 0x7362u);
        Y[4 * q + 0] = __byte_perm(c01, t1, 0x7610u);
        Y[4 * q + 1] = __byte_perm(c01, x1, 0x5432u);
        Y[4 * q + 2] = __byte_perm(c23, x1, 0x6510u);
        Y[4 * q + 3] = __byte_perm(c23, x1, 0x7632u);
      } else {   // byte 0 meets a zero tap
        Y[4 * q + 0] = __byte_perm(x0, t1, 0x7600u);
        Y[4 * q + 1] = __byte_perm(x0, x1, 0x5410u);
        Y[4 * q + 2] = __byte_perm(x0, x1, 0x6520u);
        Y[4 * q + 3] = __byte_perm(x0, x1, 0x7630u);
      }
    }
#pragma unroll
    for (int j = j_lo; j <= j_hi; ++j) {
      const int uI = j + 4 - K;
      if (uI >= 1)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[j][e] = __dp4a(Y[e], T.y[uI], acc[j][e]);
    }
  }
#pragma unroll
  for (int c = 2; c <= u_hi; ++c) {
    uint32_t W[8];
#pragma unroll
    for (int q = 0; q < 2; ++q) windows(x[c], q, W + 4 * q);
#pragma unroll
    for (int j = j_lo; j <= j_hi; ++j) {
      const int uI = j + 4 - K;
      if (uI >= c)
#pragma unroll
        for (int e = 0; e < 8; ++e) acc[j][e] = __dp4a(W[e], T.w[c - 2][uI], acc[j][e]);
    }
  }
}

// Output slice u of this thread: reduce mod p^2 and store; in the last product apply the Delta_1 epilogue first.
template <int P, bool LAST, bool DEBUG>
__device__ __forceinline__ void store_slice(uint32_t *__restrict__ out, const Smem &sm, const Lane &L, int u,
                                            const uint8_t *gs, uint32_t (&acc)[8], uint32_t &bad, DebugPtrs dbg) {
  using Pr = Prime<P>;
  uint32_t G[8];
  uint32_t *o = L.out + sm.SW[max(u, 0)];
  if (LAST) {
    if (u < L.s_min) return;
    if (DEBUG) {
      uint32_t *g = dbg.G + (o - out);
      g[0] = g[1] = 0u;
      for (int j = 0; j < 8; ++j) g[j >> 2] |= mod_p2_mulhi<P>(acc[j]) << (8 * (j & 3));
      for (int k = 2; k < (u >= L.s_pad2 ? 6 : u >= L.s_pad1 ? 4 : 2); ++k) g[k] = 0u;
    }
    if (u % P == 0 && L.s % P == 0) {   // lattice points pJ: subtract S[pJ] = c_J^p mod p^2
      const uint8_t *gc = gs + tet(u / P) + tri(L.s / P);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int t = 8 * L.h + j;
        if (t % P == 0 && t <= L.s) acc[j] += (uint32_t)(Pr::p2 - sm.powp[gc[t / P]]);
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      // acc = p (p k + d): d by two multiply-highs (exact for every value here, as mod_p2_mulhi's)
      constexpr uint32_t M = (uint32_t)((0x100000000ull + P - 1) / P);
      static_assert((uint64_t)(Pr::chain_max + Pr::p2) * ((uint64_t)M * P - 0x100000000ull) < 0x100000000ull,
                    "division by p exact over the chain's range");
      const uint32_t q = __umulhi(acc[j], M);
      bad |= acc[j] - (uint32_t)P * q;
      G[j] = q - (uint32_t)P * __umulhi(q, M);
    }
  } else {
#pragma unroll
    for (int j = 0; j < 8; ++j) G[j] = mod_p2_mulhi<P>(acc[j]);   // outputs past the column's end are zero
  }
  uint32_t w[2];
#pragma unroll
  for (int q = 0; q < 2; ++q)
    w[q] = __byte_perm(__byte_perm(G[4 * q], G[4 * q + 1], 0x0040u), __byte_perm(G[4 * q + 2], G[4 * q + 3], 0x0040u),
                       0x5410u);
  if (u >= L.s_min) *reinterpret_cast<uint2 *>(o) = make_uint2(w[0], w[1]);
  if (u >= L.s_pad1) *reinterpret_cast<uint2 *>(o + 2) = make_uint2(0u, 0u);
  if (u >= L.s_pad2) *reinterpret_cast<uint2 *>(o + 4) = make_uint2(0u, 0u);
}

// The block u0 .. u0+3 over every tap pair: groups ga (slices u0-4 .. u0-1) and gb (u0 .. u0+3; absent in the block
// of the last four output slices, whose inputs end at u0 - 1).  The columns of a slice are loaded while the slice
// before is multiplied.
template <int STRIDE>
__device__ __forceinline__ void dense_block(const char *ga, const char *gb, bool last, const Lane &L, const Taps &T,
                                            uint32_t (&acc)[kSlices][8]) {
  Col xa[5], xb[5];
  load_slice<STRIDE, 0>(ga, L, xa);
  load_slice<STRIDE, 1>(ga, L, xb);
  slice_macs<0>(xa, T, acc);
  load_slice<STRIDE, 2>(ga, L, xa);
  slice_macs<1>(xb, T, acc);
  load_slice<STRIDE, 3>(ga, L, xb);
  slice_macs<2>(xa, T, acc);
  if (last) {
    slice_macs<3>(xb, T, acc);
    return;
  }
  load_slice<STRIDE, 4>(gb, L, xa);
  slice_macs<3>(xb, T, acc);
  load_slice<STRIDE, 5>(gb, L, xb);
  slice_macs<4>(xa, T, acc);
  load_slice<STRIDE, 6>(gb, L, xa);
  slice_macs<5>(xb, T, acc);
  load_slice<STRIDE, 7>(gb, L, xb);
  slice_macs<6>(xa, T, acc);
  slice_macs<7>(xb, T, acc);
}

// A unit of work: the blocks of one segment of a strip, segments counted back from the strip's last block.  It reads
// ng groups of input slices from slice v0 on: one per block, and one more unless the unit ends with the product's
// last slices.
struct Unit {
  int v0, nb, ng;
};
__device__ __forceinline__ Unit unit_at(const Strip &S, int j, int seg, int m_out) {
  Unit U;
  const int hi = m_out - 4 * seg * j;
  U.nb = min(seg, ((m_out - S.s_lo + 4) >> 2) - seg * j);
  U.ng = U.nb + (j > 0);
  U.v0 = hi - 3 - 4 * U.nb;
  return U;
}

// Blocks of a unit (log2).  Short units keep the teams level in a small product, but each reads one group more and
// ends with one more barrier: 16 / 8 / 4 blocks took 1.203 us per quartic at p = 5 (16 / 16 / 8: 1.386, 8 / 4 / 2:
// 1.300) and 12.5 at p = 7 (32 / 16 / 4: level, 8 / 4 / 2: 13.0).
__device__ __forceinline__ int unit_log2(int m_out) { return m_out >= 120 ? 4 : m_out >= 72 ? 3 : 2; }

template <int n>
__device__ __forceinline__ void team_sync(int team) {
  if constexpr (n == kThreads) __syncthreads();
  else asm volatile("bar.sync %0, %1;" ::"r"(1 + team), "n"(n) : "memory");
}

template <int P, bool SMALL, bool LAST, bool DEBUG>
__device__ __noinline__ void run_strips(const uint32_t *__restrict__ in, uint32_t *__restrict__ out, int m_in,
                                        Smem &sm, uint32_t *ring, const uint8_t *gs, uint32_t *status,
                                        DebugPtrs dbg) {
  using R = Ring<P, SMALL>;
  constexpr int kTeam = R::team, kOwn = kThreads / kTeam, kPerSlice = kTeam / kSlices;
  constexpr int kCopies = (R::stride / 4 - 1 + kPerSlice - 1) / kPerSlice;   // 16-byte copies per thread and group
  const uint32_t *tab = SMALL && small_apart(P) ? sm.small_tab : sm.strip_tab;
  const int m_out = m_in + 4;
  const int n_items = half_prefix(m_out + 1), n_strips = (n_items + kTeam - 1) / kTeam;
  const int team = (int)threadIdx.x / kTeam, tt = (int)threadIdx.x % kTeam;
  const int fs = tt / kPerSlice, fk = tt % kPerSlice;   // slice of a group and first chunk this thread copies
  ring += team * R::words;
  // teams of the crew; a crew's units are shorter, so that there are enough of them
  const int kTeams = kOwn * sm.crew, me = kOwn * sm.rank + team;
  const int lg = max(1, unit_log2(m_out) - (sm.crew > 1 ? high_bit((unsigned)sm.crew) : 0)), seg = 1 << lg;   // blocks of a unit
  Taps T;
#pragma unroll
  for (int uI = 1; uI < 5; ++uI) {
    T.y[uI] = (sm.tapword[tri(uI)] >> 24 << 8) | (sm.tapword[tri(uI) + 1] & 0xFFFF0000u);
    if (uI == 4) T.y[uI] |= (uint32_t)sm.taps[34];
#pragma unroll
    for (int c = 2; c <= uI; ++c) T.w[c - 2][uI] = sm.tapword[tri(uI) + c];
  }
#pragma unroll
  for (int r = 0; r < 4; ++r) T.a00[r] = (uint32_t)sm.taps[0] << (8 * r);
  // the zero chunk before each staged slice
  if (tt < kGroups * kSlices) *reinterpret_cast<uint4 *>(ring + tt * R::stride) = make_uint4(0u, 0u, 0u, 0u);

  // Unit queue of the product (counter (m_in / 4) mod 2 of the crew's first CTA; the other one is cleared for the next
  // product).  Units are numbered strip after strip; a team's first two are fixed, the others come from the counter.
  const int par = (m_in >> 2) & 1;
  if (threadIdx.x == 0) sm.unit_next[par ^ 1] = 0;
  auto claim = [&]() {
    if (sm.crew == 1) return atomicAdd(&sm.unit_next[par], 1);
    int n;
    asm volatile("atom.relaxed.cluster.shared::cluster.add.s32 %0, [%1], 1;"
                 : "=r"(n)
                 : "r"(crew_addr(&sm.unit_next[par], 0))
                 : "memory");
    return n;
  };
  int cur_k = 0, cur_base = 0;   // cursor: strip and the number of units before it
  auto find = [&](int u) {       // unit u >= the last one -> strip | segment << 16, or -1 past the end
    while (cur_k < n_strips) {
      const int nb = (m_out - (int)(tab[cur_k] & 0xFFFFu) + 4) >> 2;
      const int n = (nb + seg - 1) >> lg;
      if (u < cur_base + n) return cur_k | ((u - cur_base) << 16);
      cur_base += n;
      ++cur_k;
    }
    return -1;
  };
  // the unit being staged
  int fid = find(me), f_g = 0, f_ng = 0, f_v = 0, f_hi = 0, f_base = 0, f_n = 0;
  auto stage_unit = [&]() {
    if (fid < 0) { f_ng = 0; return; }
    const Strip S = strip_at(tab, fid & 0xFFFF, m_out);
    const Unit U = unit_at(S, fid >> 16, seg, m_out);
    f_g = 0;
    f_ng = U.ng;
    f_v = U.v0;
    f_hi = S.s_hi;
    f_base = colw(S.c_lo);                          // word offset of column c_lo in a slice
    f_n = (colw(S.s_hi + 1) - f_base) >> 2;         // chunks of the strip's columns
  };
  stage_unit();
  int uid = fid;                     // the unit being multiplied
  int q0 = -1, q1 = -1;              // units staged after it
  int nxt = me + kTeams;             // the unit to stage after fid
  int qp = 0;
  bool want = false;
  // next group -> ring slot `slot`
  auto fetch = [&](int slot) {
    if (f_ng > 0 && f_g == f_ng) {   // on to the next unit
      if (want) {   // the leader took it from the counter before the last barrier
        nxt = sm.unit_slot[team][qp];
        qp ^= 1;
      }
      fid = find(nxt);
      stage_unit();
      if (q0 < 0) q0 = fid; else q1 = fid;
      want = fid >= 0;
      if (want && tt == 0) sm.unit_slot[team][qp] = 2 * kTeams + claim();
    }
    if (f_ng > 0) {
      const int v = f_v + fs;
      uint32_t *dst = ring + slot * R::group + fs * R::stride + 4 + 4 * fk;
      const uint32_t *src = in + sm.SW[max(v, 0)] + f_base + 4 * fk;
      int have = f_n;
      if (f_v < f_hi) {   // a slice of this group lacks some of the strip's columns: zeros there
        have = v >= 0 ? min(f_n, max(0, (colw(v + 1) - f_base) >> 2)) : 0;
        for (int k = fk; k < f_n; k += kPerSlice)
          if (k >= have) *reinterpret_cast<uint4 *>(dst + 4 * (k - fk)) = make_uint4(0u, 0u, 0u, 0u);
      }
#pragma unroll
      for (int c = 0; c < kCopies; ++c)
        if (fk + c * kPerSlice < have) cp_async16(dst + 4 * c * kPerSlice, src + 4 * c * kPerSlice, true);
      f_v += 4;
      ++f_g;
    }
    cp_async_commit();
  };
  int slot = 0;   // ring slot of the current block's first group
  uint32_t bad = 0;
  fetch(0);
  fetch(1);
  while (uid >= 0) {
    const Strip S = strip_at(tab, uid & 0xFFFF, m_out);
    const Unit U = unit_at(S, uid >> 16, seg, m_out);
    const bool top = (uid >> 16) == 0;
    Lane L;
    // item tt of the strip; past s_hi there is none
    L.s = S.s_lo;
    L.h = S.h_lo + tt;
    while (L.s < S.s_hi && L.h >= half_chunks_of(L.s)) L.h -= half_chunks_of(L.s++);
    const bool valid = L.h < half_chunks_of(L.s);
    if (!valid) L.h = 0;
    const int s_first = __shfl_sync(0xffffffffu, valid ? L.s : 1 << 30, 0);
#pragma unroll
    for (int sI = 0; sI < 5; ++sI) {
      const int sc = L.s - sI;   // a column before the first reads the zero chunk
      L.off[sI] = 4u * (uint32_t)(sc >= 0 ? 4 + colw(sc) - colw(S.c_lo) + 2 * L.h : 2);
    }
    L.out = out + colw(L.s) + 2 * L.h;
    // the last item of column s also clears the padding half-chunks after it (2 chunks_of(s) - (s/8 + 1) of them)
    const int pad = L.h == half_chunks_of(L.s) - 1 ? 2 * chunks_of(L.s) - half_chunks_of(L.s) : 0;
    L.s_min = valid ? L.s : 1 << 30;
    L.s_pad1 = pad >= 1 ? L.s_min : 1 << 30;
    L.s_pad2 = pad >= 2 ? L.s_min : 1 << 30;
    int u0 = U.v0 + 4;
    for (int b = 0; b < U.ng; ++b, u0 += 4) {
      // this block's groups have arrived for every thread, and nobody reads the slot of the block before any more
      cp_async_wait_all();
      team_sync<kTeam>(team);
      const int slot_b = slot == kGroups - 1 ? 0 : slot + 1, slot_f = slot_b == kGroups - 1 ? 0 : slot_b + 1;
      fetch(slot_f);
      if (b < U.nb && u0 + 3 >= s_first) {
        const char *ga = reinterpret_cast<const char *>(ring + slot * R::group);
        const char *gb = reinterpret_cast<const char *>(ring + slot_b * R::group);
        uint32_t acc[kSlices][8];
#pragma unroll
        for (int j = 0; j < kSlices; ++j)
#pragma unroll
          for (int e = 0; e < 8; ++e) acc[j][e] = 0;
        dense_block<R::stride>(ga, gb, top && b == U.nb - 1, L, T, acc);
#pragma unroll
        for (int j = 0; j < kSlices; ++j)
          store_slice<P, LAST, DEBUG>(out, sm, L, u0 + j, gs, acc[j], bad, dbg);
      }
      slot = slot_b;
    }
    uid = q0;
    q0 = q1;
    q1 = -1;
  }
  if (LAST && bad) atomicOr(status, kStatusInexactDivision);
}

}  // namespace block

// Words of shared memory a dp4a product of prime p stages its input in.
__host__ __device__ constexpr int block_ring_words(int p) {
  return kThreads / block::team_threads(p) * block::kGroups * block::kSlices *
         block::slice_stride(4 * p * (p - 1), block::team_threads(p));
}

// The dp4a product (every tap pair, whatever sm.dense_min).  The caller runs it with every thread of the crew, between
// two barriers of the crew, after setup_quartic; consecutive products have degrees four apart or start again at degree 4 (their
// unit counters alternate); ring: block_ring_words words, 16-byte aligned.  SMALL: the product's degree is 4P at most.
template <int P, bool SMALL, bool LAST, bool DEBUG>
__device__ __forceinline__ void block_chain_step(const uint32_t *__restrict__ in, uint32_t *__restrict__ out,
                                                 int m_in, Smem &sm, uint32_t *ring, const uint8_t *gs,
                                                 uint32_t *status, DebugPtrs dbg) {
  constexpr bool kApart = SMALL && block::small_apart(P);
  static_assert(kThreads / block::Ring<P, kApart>::team * block::Ring<P, kApart>::words <= block_ring_words(P),
                "the small products' rings fit in the long ones'");
  block::run_strips<P, kApart, LAST, DEBUG>(in, out, m_in, sm, ring, gs, status, dbg);
}

}  // namespace qfs
