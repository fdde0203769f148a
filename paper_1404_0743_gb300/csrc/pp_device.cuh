// pp_device.cuh -- device code shared by the kernel files.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

#include "pp_internal.h"

namespace pp {

// Index of the last descriptor whose first block (or first warp) is <= x, by
// whole warps: 32 probes at a time, so that a thousand descriptors take two
// dependent loads instead of ten.  x and the arguments are the same in every
// lane; descriptor 0 starts at 0.
template <typename T, typename First>
__device__ __forceinline__ int find_owner(const T* __restrict__ d, int n, uint32_t x, First first) {
  const int lane = threadIdx.x & 31;
  int lo = 0;
  while (n > 1) {  // the owner is one of d[lo .. lo + n)
    const int step = (n + 31) / 32, at = lo + lane * step;
    const bool below = lane * step < n && first(d[at]) <= x;
    const int last = 31 - __clz(__ballot_sync(0xFFFFFFFFu, below));  // probe 0 always holds
    n = min(step, n - last * step);
    lo += last * step;
  }
  return lo;
}
template <typename T>
__device__ __forceinline__ int find_block_owner(const T* __restrict__ d, int n, uint32_t b) {
  return find_owner(d, n, b, [](const T& t) { return t.block0; });
}

// 256-bit accesses (sm_100 and later): one load or store instruction per 32
// bytes, half the instructions and L1 sector lookups of 128-bit accesses to
// the same scattered addresses.  The address must be 32-byte aligned.
// Read-only data (written by an earlier launch): the compiler may schedule
// the load freely.
__device__ __forceinline__ void ld256_nc(const void* p, uint32_t r[8]) {
  asm("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}
// The same, kept in program order with the stores and other such loads: for
// loads meant to be in flight during the work written after them.
__device__ __forceinline__ void ld256_nc_early(const void* p, uint32_t r[8]) {
  asm volatile("ld.global.nc.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p));
}
// Data other blocks of the same launch wrote before a grid barrier: read
// through L2, ordered with the barrier.
__device__ __forceinline__ void ld256_cg(const void* p, uint32_t r[8]) {
  asm volatile("ld.global.cg.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "l"(p)
               : "memory");
}
__device__ __forceinline__ void st256(void* p, const uint32_t r[8]) {
  asm volatile("st.global.v8.u32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// Data this launch wrote before a grid barrier the caller has passed, read
// through L1 (no line of it was read before).  The compiler may schedule the
// load freely after its address is known, so the address must come from a
// load made after the barrier (the callers keep it in shared memory).
__device__ __forceinline__ void ld256(const void* p, uint32_t r[8]) {
  asm("ld.global.v8.u32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "l"(p));
}

// Eight words of eight bits per byte -> bit t of byte s of word i becomes bit
// i of byte s of word t (an 8 x 8 transpose in every byte).
__device__ __forceinline__ void transpose8(uint32_t w[8]) {
#pragma unroll
  for (int d = 4; d > 0; d >>= 1) {
    const uint32_t m = d == 4 ? 0x0F0F0F0Fu : d == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int i = 0; i < 8; i++) {
      if (i & d) continue;
      const uint32_t t = ((w[i] >> d) ^ w[i + d]) & m;
      w[i + d] ^= t;
      w[i] ^= t << d;
    }
  }
}

// rmax(x)(g) = OR over the 8 single-quadrant quarter turns r of x(g + r)
// (paper, "Abstracting over rotations").  For one axis, x(g+1) | x(g-1) =
// y(g+1) with y(g) = x(g) | x(g+2), and y has period 2 along that axis.
__device__ __forceinline__ void rmax(const uint32_t x[8], uint32_t r[8]) {
  uint32_t a2[4], v[4];
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const uint32_t u = x[2 * j] | x[2 * j + 1];  // axis 2: fold g2 with g2 + 2
    a2[j] = __funnelshift_l(u, u, 16);           // then step g2 by one
    v[j] = x[j] | x[j + 4];                      // axis 3: fold g3 with g3 + 2
  }
#pragma unroll
  for (int w = 0; w < 8; w++) {
    const uint32_t y0 = x[w] | ((x[w] >> 2) & 0x33333333u) | ((x[w] << 2) & 0xCCCCCCCCu);
    const uint32_t a0 = ((y0 >> 1) & 0x55555555u) | ((y0 << 1) & 0xAAAAAAAAu);
    const uint32_t y1 = x[w] | __byte_perm(x[w], 0, 0x2301);
    const uint32_t a1 = ((y1 >> 4) & 0x0F0F0F0Fu) | ((y1 << 4) & 0xF0F0F0F0u);
    r[w] = a0 | a1 | a2[w >> 1] | v[(w + 2) & 3];
  }
}

__device__ __forceinline__ void load_super(const pp_super* p, uint32_t W[8], uint32_t N[8]) {
  const uint4* v = reinterpret_cast<const uint4*>(p);
  const uint4 a = __ldg(v), b = __ldg(v + 1), c = __ldg(v + 2), d = __ldg(v + 3);
  W[0] = a.x, W[1] = a.y, W[2] = a.z, W[3] = a.w, W[4] = b.x, W[5] = b.y, W[6] = b.z, W[7] = b.w;
  N[0] = c.x, N[1] = c.y, N[2] = c.z, N[3] = c.w, N[4] = d.x, N[5] = d.y, N[6] = d.z, N[7] = d.w;
}

__device__ __forceinline__ void store_super(pp_super* p, const uint32_t W[8], const uint32_t N[8]) {
  uint4* v = reinterpret_cast<uint4*>(p);
  v[0] = make_uint4(W[0], W[1], W[2], W[3]);
  v[1] = make_uint4(W[4], W[5], W[6], W[7]);
  v[2] = make_uint4(N[0], N[1], N[2], N[3]);
  v[3] = make_uint4(N[4], N[5], N[6], N[7]);
}

__device__ __forceinline__ void load_mask(const uint4* p, uint32_t F[8]) { ld256_nc(p, F); }

// ---------------------------------------------------------------------------
// Half tables (paper, "Open source and data": rmax flips the parity of
// g0 + g1 + g2 + g3, so a solve that wants one parity class at the root
// needs only one class at every level, alternating, and stores 32 bytes per
// position instead of 64).  Parity of beta(g) = b0 ^ b2 ^ b4 ^ b6: inside a
// word, neighbouring bits (b0 = 0, 1) belong to opposite classes, and b6 is
// word bit 1.  A class's 16 bits of a word are gathered to the even bit
// positions; words 2j and 2j + 1 (same class pattern) then share one word,
// 2j at even and 2j + 1 at odd positions.  Bits of the other class are not
// stored and unpack as zero: rmax, the combine and the five masks never let
// them reach the wanted class.
// ---------------------------------------------------------------------------
constexpr uint32_t kClass0 = 0x5A5AA5A5u;  // in-word positions t with t0 ^ t2 ^ t4 = 0

__device__ __forceinline__ uint32_t class_bits(uint32_t p, int w) {
  return ((p ^ (uint32_t)(w >> 1)) & 1u) ? ~kClass0 : kClass0;
}

// 8 words (class p valid) -> 4 words
__device__ __forceinline__ void half_pack(const uint32_t x[8], uint32_t p, uint32_t h[4]) {
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const uint32_t K = class_bits(p, 2 * j), E = K & 0x55555555u, O = (K >> 1) & 0x55555555u;
    const uint32_t a = (x[2 * j] & E) | ((x[2 * j] >> 1) & O);
    const uint32_t b = (x[2 * j + 1] & E) | ((x[2 * j + 1] >> 1) & O);
    h[j] = a | (b << 1);
  }
}

// 4 words -> 8 words, the other class zero
__device__ __forceinline__ void half_unpack(const uint32_t h[4], uint32_t p, uint32_t x[8]) {
#pragma unroll
  for (int j = 0; j < 4; j++) {
    const uint32_t K = class_bits(p, 2 * j), E = K & 0x55555555u, O = (K >> 1) & 0x55555555u;
    const uint32_t a = h[j] & 0x55555555u, b = (h[j] >> 1) & 0x55555555u;
    x[2 * j] = (a & E) | ((a & O) << 1);
    x[2 * j + 1] = (b & E) | ((b & O) << 1);
  }
}

// Out of line for whole tables with a lane to a fill: beside the fold it made
// the persistent kernel spill (one board with 16 empty cells 615 us, 584 so).
static __device__ __noinline__ int find_segment(const MidSeg* segs, int n, uint32_t b) {
  return find_block_owner(segs, n, b);
}

// One thread block's worth (kBlock fills) of one midgame level: block vb of
// the level's segments (paper, "Open source and data").
//
// A fill's value folds its children: on rotations where the fill has no
// five, win = OR_e (I_e | rmax(~notlose_e)) and notlose = OR_e (I_e |
// rmax(~win_e)), where I_e, the mover's five after the move e, is the
// child's five-in-a-row set of the colour that is not to move there (rmax
// distributes over OR; paper, "Abstracting over rotations").  So every fill
// below the root stores, instead of its value, the two tables its parents
// OR: (F_o | rmax(~notlose), F_o | rmax(~win)), F_o its own five-in-a-row
// set of the colour not to move.  A parent then reads one 64-byte record
// per move and takes no rmax; each fill still takes two.  The root stores
// its value.  A fill's own masks come from the board's colour-subset five
// tables (five_table_kernel); its children from the level below.
//
// Whole tables: a pair of lanes shares a fill, the even one folding the
// children's win slots and making the fill's not-lose slot, the odd one the
// other way round, four loads in flight each.  A warp's load of children then
// takes 64 bytes of each line it touches (a lane to a record took 32 at a
// time, two L1 wavefronts a record).  Still bound by the latency and the L1
// wavefronts of scattered records: one board with 16 empty cells, graph, 562
// us with a lane to a fill, 495 so.  Fills h0 to h1 of the block, in halves of
// kBlock / 2.
template <bool L2ONLY>
__device__ __forceinline__ void midgame_fill_pairs(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                                                  int nsegs, uint32_t vb, pp_super* __restrict__ table,
                                                  pp_super* __restrict__ out, int final_level,
                                                  const uint4* __restrict__ masks, uint32_t seg_blocks,
                                                  uint32_t h0, uint32_t h1) {
  const uint32_t per = seg_blocks & ~kSharedSegs;
  const int owner = per ? (int)(vb / per) : find_block_owner(segs, nsegs, vb);
  MidSeg sg = segs[(seg_blocks & kSharedSegs) ? 0 : owner];
  if (seg_blocks & kSharedSegs) sg.board += (uint32_t)owner, sg.block0 = (uint32_t)owner * per;
  const MidBoard& B = boards[sg.board];
  const int k = (int)B.k, level = (int)sg.level;
  const uint32_t c = (level & 1) ? 3u - B.mover : B.mover;  // colour to move
  const uint4* mt = masks + 2 * B.masks;
  const uint32_t kk = 1u << k, moves = (uint32_t)(k - level), slot = threadIdx.x & 1;
  const char* kids = reinterpret_cast<const char*>(table + B.table + sg.coff) + 32 * slot;
  pp_super* own = table + B.table + sg.loff;
  auto load = [&](uint32_t child, uint32_t r[8]) {
    if (L2ONLY)
      ld256_cg(kids + (uint64_t)child * sizeof(pp_super), r);
    else
      ld256_nc(kids + (uint64_t)child * sizeof(pp_super), r);
  };
#pragma unroll 1
  for (uint32_t half = h0; half < h1; half++) {
    const uint32_t e = (vb - sg.block0) * kBlock + half * (kBlock / 2) + (threadIdx.x >> 1);
    if (e >= sg.count) return;
    const uint64_t entry = __ldg(sg.list + e);
    const uint32_t* __restrict__ rk = sg.ranks + (uint64_t)e * moves;
    uint32_t A[8];
    const uint32_t full = slot && !moves ? 0xFFFFFFFFu : 0u;
#pragma unroll
    for (int w = 0; w < 8; w++) A[w] = full;
    uint32_t m = 0;
    for (; m + 3 < moves; m += 4) {
      const uint32_t r0 = __ldg(rk + m), r1 = __ldg(rk + m + 1), r2 = __ldg(rk + m + 2), r3 = __ldg(rk + m + 3);
      uint32_t a[8], b[8], x[8], y[8];
      load(r0, a);
      load(r1, b);
      load(r2, x);
      load(r3, y);
#pragma unroll
      for (int w = 0; w < 8; w++) A[w] |= a[w] | b[w], A[w] |= x[w] | y[w];
    }
    for (; m < moves; m++) {
      uint32_t a[8];
      load(__ldg(rk + m), a);
#pragma unroll
      for (int w = 0; w < 8; w++) A[w] |= a[w];
    }
    const uint32_t bm = (uint32_t)(entry >> 32) & 0xFFFFu, wm = (uint32_t)(entry >> 48);
    uint32_t Fc[8], Fo[8], R[8];
    load_mask(mt + 2 * ((c - 1) * kk + (c == 1 ? bm : wm)), Fc);
    load_mask(mt + 2 * ((2 - c) * kk + (c == 1 ? wm : bm)), Fo);
    const uint32_t nl = slot ? 0xFFFFFFFFu : 0u;
#pragma unroll
    for (int w = 0; w < 8; w++) {
      const uint32_t mine = Fc[w] & (nl | ~Fo[w]);
      A[w] = mine | (~Fo[w] & A[w]);
    }
    if (final_level || sg.final) {
      uint4* v = reinterpret_cast<uint4*>(slot ? out[B.out].notlose : out[B.out].win);
      v[0] = make_uint4(A[0], A[1], A[2], A[3]);
      v[1] = make_uint4(A[4], A[5], A[6], A[7]);
      continue;
    }
#pragma unroll
    for (int w = 0; w < 8; w++) A[w] = ~A[w];
    rmax(A, R);
#pragma unroll
    for (int w = 0; w < 8; w++) R[w] |= Fo[w];
    st256(slot ? own[e].win : own[e].notlose, R);
  }
}

// One lane to a fill: half tables (32-byte records), and whole ones of large
// batches in the persistent kernel (see kPairFills).
template <bool L2ONLY, bool HALF>
__device__ __forceinline__ void midgame_fill_lane(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                                             int nsegs, uint32_t vb, pp_super* __restrict__ table,
                                             pp_super* __restrict__ out, int final_level,
                                             const uint4* __restrict__ masks, uint32_t seg_blocks, uint32_t parity) {
  // segments of equal size (boards sharing k and mover): the owner is a division;
  // shared segments: one stored descriptor, the board follows from the owner
  const uint32_t per = seg_blocks & ~kSharedSegs;
  const int owner = per                ? (int)(vb / per)
                    : L2ONLY && !HALF ? find_segment(segs, nsegs, vb)
                                      : find_block_owner(segs, nsegs, vb);
  MidSeg sg = segs[(seg_blocks & kSharedSegs) ? 0 : owner];
  if (seg_blocks & kSharedSegs) sg.board += (uint32_t)owner, sg.block0 = (uint32_t)owner * per;
  const uint32_t e = (vb - sg.block0) * kBlock + threadIdx.x;
  if (e >= sg.count) return;
  const uint64_t entry = __ldg(sg.list + e);
  const uint32_t bm = (uint32_t)(entry >> 32) & 0xFFFFu, wm = (uint32_t)(entry >> 48);
  const MidBoard& B = boards[sg.board];
  const int k = (int)B.k, level = (int)sg.level;
  const uint32_t c = (level & 1) ? 3u - B.mover : B.mover;  // colour to move
  const uint4* mt = masks + 2 * B.masks;
  const uint32_t kk = 1u << k, mc = c == 1 ? bm : wm, mo = c == 1 ? wm : bm;
  const uint4* mtc = mt + 2 * ((c - 1) * kk);  // the mover's table
  const uint32_t own = (parity ^ (uint32_t)level) & 1u;  // half: this level's class (its children store it)
  uint32_t Fc[8], Fo[8], W[8], N[8];
  if (level == k) {  // full board
    load_mask(mtc + 2 * mc, Fc);
    load_mask(mt + 2 * ((2 - c) * kk + mo), Fo);
#pragma unroll
    for (int w = 0; w < 8; w++) W[w] = Fc[w] & ~Fo[w], N[w] = Fc[w] | ~Fo[w];
  } else {
    uint32_t AW[8] = {0}, AN[8] = {0};
    // compact table: level + 1 starts at coff; the fill's children's
    // positions there are listed in slot order
    const pp_super* tab = table + B.table + sg.coff;
    const uint32_t* htab = reinterpret_cast<const uint32_t*>(table) + 8 * ((uint64_t)B.table + sg.coff);  // half
    const uint32_t moves = (uint32_t)(k - level);
    const uint32_t* __restrict__ rk = sg.ranks + (uint64_t)e * moves;
    auto fold = [&](uint32_t child) {
      uint32_t cW[8], cN[8];
      auto load = [](const void* p, uint32_t r[8]) {
        if (L2ONLY)
          ld256_cg(p, r);
        else
          ld256_nc(p, r);
      };
      if (HALF) {
        uint32_t h[8];
        load(htab + 8 * (uint64_t)child, h);
        half_unpack(h, own, cW);
        half_unpack(h + 4, own, cN);
      } else {
        load(tab[child].win, cW);
        load(tab[child].notlose, cN);
      }
#pragma unroll
      for (int w = 0; w < 8; w++) AW[w] |= cW[w], AN[w] |= cN[w];
    };
    if constexpr (L2ONLY) {
      // persistent kernel: two moves per round, both children's loads in
      // flight together, the next round's positions read while they are
      uint32_t r0 = __ldg(rk), r1 = moves > 1 ? __ldg(rk + 1) : 0u;  // level < k: at least one move
      uint32_t m = 0;
      for (; m + 1 < moves; m += 2) {
        const uint32_t a = r0, b = r1;
        if (m + 2 < moves) r0 = __ldg(rk + m + 2);
        if (m + 3 < moves) r1 = __ldg(rk + m + 3);
        fold(a);
        fold(b);
      }
      if (m < moves) fold(r0);
    } else {
      // level kernel (40 registers): one move at a time, the next move's
      // position in flight with this child
      uint32_t next = __ldg(rk);
      for (uint32_t m = 0; m < moves; m++) {
        const uint32_t child = next;
        if (m + 1 < moves) next = __ldg(rk + m + 1);
        fold(child);
      }
    }
    // the position's own masks, loaded last to keep the loop's registers free
    load_mask(mtc + 2 * mc, Fc);
    load_mask(mt + 2 * ((2 - c) * kk + mo), Fo);
#pragma unroll
    for (int w = 0; w < 8; w++) {
      const uint32_t T = Fc[w] | Fo[w];
      W[w] = (Fc[w] & ~Fo[w]) | (~T & AW[w]);
      N[w] = Fc[w] | (~T & AN[w]);
    }
  }
  if (final_level || sg.final) {
    if (HALF) {  // the root: the wanted class, the other zero
#pragma unroll
      for (int w = 0; w < 8; w++) {
        const uint32_t K = class_bits(parity, w);
        W[w] &= K, N[w] &= K;
      }
    }
    store_super(out + B.out, W, N);
    return;
  }
  // the tables the parents OR
  uint32_t P[8], R[8];
#pragma unroll
  for (int w = 0; w < 8; w++) N[w] = ~N[w], W[w] = ~W[w];
  rmax(N, P);
  rmax(W, R);
#pragma unroll
  for (int w = 0; w < 8; w++) P[w] |= Fo[w], R[w] |= Fo[w];
  if (HALF) {  // on the parents' class
    uint32_t h[8];
    half_pack(P, own ^ 1u, h);
    half_pack(R, own ^ 1u, h + 4);
    st256(reinterpret_cast<uint32_t*>(table) + 8 * ((uint64_t)B.table + sg.loff + e), h);
  } else {
    pp_super* r = table + B.table + sg.loff + e;
    st256(r->win, P);
    st256(r->notlose, R);
  }
}

template <bool L2ONLY, bool HALF>
__device__ __forceinline__ void midgame_fill(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                                             int nsegs, uint32_t vb, pp_super* __restrict__ table,
                                             pp_super* __restrict__ out, int final_level,
                                             const uint4* __restrict__ masks, uint32_t seg_blocks, uint32_t parity) {
  if constexpr (HALF)
    midgame_fill_lane<L2ONLY, true>(boards, segs, nsegs, vb, table, out, final_level, masks, seg_blocks, parity);
  else
    midgame_fill_pairs<L2ONLY>(boards, segs, nsegs, vb, table, out, final_level, masks, seg_blocks, 0, 2);
}

// Grid-wide barrier for a cooperative launch (every block resident).  The
// wait is bounded: after `limit` polls it records PP_ETIMEOUT in
// *status and lets the block go; the kernel then stops at its next level and
// the host reports the error.  bar[0] counts arrivals, bar[1] is the
// generation.
__device__ __forceinline__ bool grid_barrier(uint32_t* bar, uint32_t* status, uint32_t limit) {
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    volatile uint32_t* vgen = bar + 1;
    const uint32_t gen = *vgen;
    if (atomicAdd(bar, 1u) + 1 == gridDim.x) {
      atomicExch(bar, 0u);
      __threadfence();
      atomicAdd(bar + 1, 1u);
    } else {
      uint32_t spins = 0;
      while (*vgen == gen) {
        if (++spins > limit) {
          atomicExch(status, (uint32_t)PP_ETIMEOUT);
          break;
        }
        __nanosleep(64);
      }
    }
    __threadfence();
  }
  __syncthreads();
  return *(volatile uint32_t*)status == 0;
}

}  // namespace pp
