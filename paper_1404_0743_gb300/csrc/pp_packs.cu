// pp_packs.cu -- midgame solves of many boards at once, sixteen boards of the
// same shape to a pack (paper, "Open source and data").
//
// Boards with the same number of empty cells and the same mover have the same
// fills, so a pack computes one fill of sixteen boards together with their
// tables sliced across boards: a 32-bit word holds, for one (g0, g1, g2), the
// four turns g3 (a byte each) of eight boards (a bit each), and a table of
// eight boards is 64 words, word g0 + 4 g1 + 16 g2.  A step along axis 0, 1 or
// 2 is then another word and a step along axis 3 a byte rotation, so rmax
// takes six operations a word, 48 a board where the one-board layout takes
// about 125.  The other reason is the loads: a record is read by eight
// neighbouring lanes as whole 128-byte lines, where 64-byte records gathered
// one to a lane use one sector of each line and keep the L1 data pipe the
// bound.
//
// What bounds it is the latency of the children's records at 16 warps per SM:
// 18.8 GB of records for 1024 boards with 12 empty cells (each written and read
// once) would take 2.8 ms at the copy rate, the whole step takes 3.54 (5.5
// before), of which the masks 0.19; DRAM is two thirds busy, the integer pipe a
// third, and without rmax the step takes as long.
//
// Eight lanes take one fill: two slots, two groups of eight boards, and the
// turns g2 even and odd.  A lane holds 32 words, g0 + 4 g1 + 16 (g2 >> 1); the
// neighbours along axis 2 are the other lane's, folded before they are
// exchanged (16 shuffles).  A lane per whole table needs 64 words, which left
// 16 warps per SM waiting on the children's loads.
//
// Record of a fill (1 KB): four rows of 256 bytes; row o holds words
// 8 o .. 8 o + 7 of each lane, 32 bytes, lane = slot + 2 (g2 & 1) + 4 group.
// Mask of a colour subset (512 bytes): four rows of 128 bytes, 32 bytes for
// each (g2 & 1) + 2 group.  Both take exactly the room the sixteen boards' own
// tables would.
//
// Half tables (one parity class, see half_pack): of each word only the bytes
// g3 = s, s + 2 belong to the class, s = class + g0 + g1 + g2 (mod 2), the same
// for g2 and g2 + 2.  A lane's word g0 + 4 g1 of 16 holds the two bytes of
// g2 = (g2 & 1) in its low half and those of g2 + 2 in its high half; records
// are two rows.  Masks stay whole.
#include <cuda_runtime.h>

#include "pp_device.cuh"
#include "pp_internal.h"

// Resident blocks of kPackThreads per SM: 16 warps at 128 registers for whole
// tables (24 at 80 spill: 4.9 ms against 3.6 for 1024 boards with 12 empty
// cells), 24 warps at 80 for half tables (2.4 ms, 16 warps 2.6).
#ifndef PP_PACK_MINB
#define PP_PACK_MINB 2
#endif
#ifndef PP_PACK_HALF_MINB
#define PP_PACK_HALF_MINB 3
#endif

namespace pp {

// This lane's 8 words of row o of a mask: whole words, or the bytes of class
// `cls` of rows o and o + 2 (odd: the lane's g2 & 1).
template <bool HALF>
__device__ __forceinline__ void load_mask_row(const char* mask, int o, uint32_t cls, uint32_t odd, uint32_t r[8]) {
  ld256_nc(mask + o * 128, r);
  if (HALF) {
    uint32_t hi[8];
    ld256_nc(mask + (o + 2) * 128, hi);
    const uint32_t even = (cls ^ odd) & 1u ? 0x7531u : 0x6420u;  // g0 + g1 even
#pragma unroll
    for (int i = 0; i < 8; i++)
      r[i] = __byte_perm(r[i], hi[i], ((i ^ i >> 2) & 1) ? even ^ 0x1111u : even);
  }
}

// OR of word w's neighbours along axes 0, 1 and 3 (paper, "Abstracting over
// rotations": rmax), the result on the other class for half tables.
template <bool HALF>
__device__ __forceinline__ uint32_t pack_rmax3(const uint32_t* x, int w) {
  const int g0 = w & 3, g1 = w >> 2 & 3;
  const uint32_t s0 = x[(w & ~3) | ((g0 + 1) & 3)] | x[(w & ~3) | ((g0 + 3) & 3)];
  const uint32_t s1 = x[(w & ~12) | (((g1 + 1) & 3) << 2)] | x[(w & ~12) | (((g1 + 3) & 3) << 2)];
  if (HALF) return s0 | s1 | x[w] | __byte_perm(x[w], 0, 0x2301);
  return s0 | s1 | __byte_perm(x[w], 0, 0x0321) | __byte_perm(x[w], 0, 0x2103);
}

// A pack's piece of a level, in shared memory while a block works on it.
struct PackSeg {
  const uint64_t* list;
  const uint32_t* ranks;
  char* rec;          // the pack's records
  const char* masks;  // its masks
  uint32_t count, level, k, mover, loff, coff;
};

// What a visit needs first: the fill's list entry and, spread over its eight
// lanes, its children's positions (lane s: children s and s + 8).
struct PackWork {
  uint64_t entry;
  uint32_t ranks[2];
  bool live;
};

__device__ __forceinline__ PackWork pack_fetch(const PackSeg& sg, uint32_t block) {
  const uint32_t e = block * kPackFills + (threadIdx.x >> 3), moves = sg.k - sg.level, sub = threadIdx.x & 7;
  PackWork w{0, {0, 0}, e < sg.count};
  if (w.live) {
    const uint32_t* __restrict__ rk = sg.ranks + (uint64_t)e * moves;
    w.entry = __ldg(sg.list + e);
    if (sub < moves) w.ranks[0] = __ldg(rk + sub);
    if (sub + 8 < moves) w.ranks[1] = __ldg(rk + sub + 8);
  }
  return w;
}

// One visit: eight lanes' fill.  A lane folds one slot of the children and so
// computes the other slot of the record the fill's parents read (the win slot
// is made from not-lose values and the other way round).
template <bool SAME_LAUNCH, bool HALF>
__device__ __forceinline__ void pack_fill(const PackSeg& sg, const PackWork& work, uint32_t parity) {
  constexpr int kRows = HALF ? 2 : 4, kEntry = HALF ? 32 : 64;
  constexpr uint32_t kRecord = kEntry * kPackBoards;
  const uint32_t sub = threadIdx.x & 7;
  const unsigned lanes = __ballot_sync(0xFFFFFFFFu, work.live);
  if (!work.live) return;
  const uint64_t entry = work.entry;
  const uint32_t pos = (uint32_t)entry, bm = (uint32_t)(entry >> 32) & 0xFFFFu, wm = (uint32_t)(entry >> 48);
  const int k = (int)sg.k, level = (int)sg.level;
  const uint32_t c = (level & 1) ? 3u - sg.mover : sg.mover;  // colour to move
  const uint32_t own = (parity ^ (uint32_t)level) & 1u;       // half: this level's class
  const uint32_t odd = sub >> 1 & 1u;                         // this lane's g2 & 1
  const uint32_t kk = 1u << k, mc = c == 1 ? bm : wm, mo = c == 1 ? wm : bm;
  const char* mk = sg.masks + (sub >> 1) * 32;
  const char* Fc = mk + (uint64_t)((c - 1) * kk + mc) * (kPackBoards * 32);
  const char* Fo = mk + (uint64_t)((2 - c) * kk + mo) * (kPackBoards * 32);
  char* rec = sg.rec;
  if (!HALF)  // both masks' lines on their way to L1 (4 rows of 128 bytes each) before the children
    asm volatile("prefetch.global.L1 [%0];" ::"l"((sub < 4 ? Fc : Fo) - (sub >> 1) * 32 + (sub & 3) * 128));
  const uint32_t notlose = (sub & 1) ? 0xFFFFFFFFu : 0u;  // the slot folded: win tables or not-lose tables
  uint32_t x[8 * kRows];
  const int moves = k - level;
  if (moves == 0) {  // full board: win = F_c & ~F_o, notlose = F_c | ~F_o
#pragma unroll
    for (int i = 0; i < 8 * kRows; i++) x[i] = notlose;
  } else {
    const char* kids = rec + (uint64_t)sg.coff * kRecord + sub * 32;
    auto child = [&](int m) {
      return kids + (uint64_t)__shfl_sync(lanes, m < 8 ? work.ranks[0] : work.ranks[1], m & 7, 8) * kRecord;
    };
    auto load = [&](const char* p, int o, uint32_t r[8]) {
      if (SAME_LAUNCH)
        ld256(p + o * 256, r);
      else
        ld256_nc(p + o * 256, r);
    };
    // an odd first child alone, then two at a time (one three-input
    // operation folds both)
    const char* a = child(0);
    int m = 1;
#pragma unroll
    for (int o = 0; o < kRows; o++) load(a, o, x + 8 * o);
    if (!(moves & 1)) {
      a = child(1);
      m = 2;
#pragma unroll
      for (int o = 0; o < kRows; o++) {
        uint32_t u[8];
        load(a, o, u);
#pragma unroll
        for (int i = 0; i < 8; i++) x[8 * o + i] |= u[i];
      }
    }
    for (; m < moves; m += 2) {
      a = child(m);
      const char* b = child(m + 1);
#pragma unroll
      for (int o = 0; o < kRows; o++) {
        uint32_t u[8], v[8];
        load(a, o, u);
        load(b, o, v);
#pragma unroll
        for (int i = 0; i < 8; i++) x[8 * o + i] |= u[i] | v[i];
      }
    }
  }
  // the fill's own table, complemented: win = ~F_o & (F_c | x), notlose =
  // F_c | (~F_o & x)
#pragma unroll
  for (int o = 0; o < kRows; o++) {
    uint32_t fc[8], fo[8];
    load_mask_row<HALF>(Fc, o, own, odd, fc);
    load_mask_row<HALF>(Fo, o, own, odd, fo);
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const uint32_t mine = fc[i] & (notlose | ~fo[i]);
      x[8 * o + i] = ~(mine | (~fo[i] & x[8 * o + i]));
    }
  }
  if (level == 0) {  // the roots' values themselves, for pack_root
    char* dst = rec + (uint64_t)sg.loff * kRecord + sub * 32;
#pragma unroll
    for (int o = 0; o < kRows; o++) {
      uint32_t r[8];
#pragma unroll
      for (int i = 0; i < 8; i++) r[i] = ~x[8 * o + i];
      st256(dst + o * 256, r);
    }
    return;
  }
  // the table the parents OR: F_o | rmax
  char* dst = rec + ((uint64_t)sg.loff + pos) * kRecord + (sub ^ 1) * 32;
#pragma unroll
  for (int q = 0; q < 2; q++) {  // words 8 q .. 8 q + 7, and those + 16
    // axis 2: both neighbours of g2 have the other lane's g2 & 1, and are the
    // same for g2 and g2 + 2
    uint32_t n[8];
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const int w = 8 * q + i;
      const uint32_t mine = HALF ? x[w] | __byte_perm(x[w], 0, 0x1032) : x[w] | x[(w + 16) % (8 * kRows)];
      n[i] = __shfl_xor_sync(lanes, mine, 2);
    }
#pragma unroll
    for (int o = q; o < kRows; o += 2) {
      uint32_t r[8];
      load_mask_row<HALF>(Fo, o, own ^ 1u, odd, r);
#pragma unroll
      for (int i = 0; i < 8; i++) r[i] |= n[i] | pack_rmax3<HALF>(x, 8 * o + i);
      st256(dst + o * 256, r);
    }
  }
}

// The roots' values, from the sliced records into the output; where the same
// launch wrote them, `table` was read after its last barrier.  Item (pack,
// group, slot, row): byte 8 g3 + row of that table of each of eight boards,
// row = (g1 >> 1) + 2 g2.
template <bool HALF>
__device__ __forceinline__ void pack_root(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                                          uint32_t seg_blocks, uint32_t item, const char* __restrict__ table,
                                          pp_super* __restrict__ out, uint32_t parity) {
  constexpr int kEntry = HALF ? 32 : 64;
  const uint32_t pack = item >> 5, row = item & 7, slot = item >> 3 & 1, group = item >> 4 & 1;
  const MidSeg& sg = segs[(seg_blocks & kSharedSegs) ? 0 : pack];
  const uint32_t first = (seg_blocks & kSharedSegs) ? sg.board + pack * kPackBoards : sg.board;
  const uint32_t g1hi = row & 1, odd = row >> 1 & 1, g2hi = row >> 2;
  uint32_t w[8];
  ld256(table + boards[first].table * kEntry + (uint64_t)sg.loff * (kEntry * kPackBoards) +
            (HALF ? g1hi : g1hi + 2 * g2hi) * 256 + (slot + 2 * odd + 4 * group) * 32,
        w);
  if (HALF) {
#pragma unroll
    for (int i = 0; i < 8; i++) {
      const uint32_t s = (parity ^ odd ^ (uint32_t)(i ^ i >> 2)) & 1u;
      const uint32_t h = g2hi ? w[i] >> 16 : w[i] & 0xFFFFu;  // bytes g3 = s, s + 2
      w[i] = __byte_perm(h, 0, s ? 0x1404 : 0x4140);
    }
  }
  transpose8(w);
#pragma unroll
  for (int b = 0; b < 8; b++) {
    unsigned char* o = reinterpret_cast<unsigned char*>(out + boards[first + 8 * group + b].out) + 32 * slot + row;
#pragma unroll
    for (int g3 = 0; g3 < 4; g3++) o[8 * g3] = (unsigned char)(w[b] >> (8 * g3));
  }
}

// One block's share of a level: a contiguous run of its blocks of kPackFills
// fills, pack after pack.  The fills of a level are listed by the stones of
// the colour not to move, and all children of the fills of one such set lie
// within C(n, a + 1) records (n cells left, a of them the mover's), so a
// share reads each of them about four times, the repeats from L1.  A pack's
// descriptor stays in shared memory (read from global memory at every visit
// it was mostly missing in L1, two round trips before the first child), and
// the next visit's list entries and child positions are loaded during this
// one.
template <bool SAME_LAUNCH, bool HALF>
__device__ __forceinline__ void pack_level(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                                           int nsegs, uint32_t blocks, uint32_t seg_blocks, char* __restrict__ table,
                                           const char* __restrict__ masks, uint32_t parity, PackSeg& sg) {
  const bool shared = seg_blocks & kSharedSegs;
  const uint32_t per = seg_blocks & ~kSharedSegs;
  const uint32_t v1 = (uint32_t)((uint64_t)blocks * (blockIdx.x + 1) / gridDim.x);
  for (uint32_t v = (uint32_t)((uint64_t)blocks * blockIdx.x / gridDim.x); v < v1;) {
    const uint32_t owner = per ? v / per : (uint32_t)find_block_owner(segs, nsegs, v);
    const uint32_t first = per ? owner * per : segs[owner].block0;
    uint32_t end = per ? first + per : owner + 1 < (uint32_t)nsegs ? segs[owner + 1].block0 : blocks;
    end = min(end, v1);
    __syncthreads();  // every warp is done with the piece before
    if (threadIdx.x == 0) {
      const MidSeg& m = segs[shared ? 0 : owner];
      const MidBoard& B = boards[m.board + (shared ? owner * kPackBoards : 0)];
      sg.list = m.list, sg.ranks = m.ranks;
      sg.rec = table + B.table * (HALF ? 32 : 64);
      sg.masks = masks + B.masks * 32;
      sg.count = m.count, sg.level = m.level, sg.k = B.k, sg.mover = B.mover, sg.loff = m.loff, sg.coff = m.coff;
    }
    __syncthreads();
    PackWork next = pack_fetch(sg, v - first);
    for (; v < end; v++) {
      const PackWork work = next;
      if (v + 1 < end) next = pack_fetch(sg, v + 1 - first);
      pack_fill<SAME_LAUNCH, HALF>(sg, work, parity);
    }
  }
}

template <bool HALF>
__global__ void __launch_bounds__(kPackThreads, HALF ? PP_PACK_HALF_MINB : PP_PACK_MINB)
    pack_level_kernel(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs, int nsegs, uint32_t blocks,
                      char* __restrict__ table, const char* __restrict__ masks, uint32_t seg_blocks, uint32_t parity) {
  __shared__ PackSeg sg;
  pack_level<false, HALF>(boards, segs, nsegs, blocks, seg_blocks, table, masks, parity, sg);
}

template <bool HALF>
__global__ void pack_root_kernel(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs, int npacks,
                                 const char* __restrict__ table, pp_super* __restrict__ out, uint32_t seg_blocks,
                                 uint32_t parity) {
  const uint32_t item = blockIdx.x * blockDim.x + threadIdx.x;
  if (item < (uint32_t)npacks * 32) pack_root<HALF>(boards, segs, seg_blocks, item, table, out, parity);
}

// A level of the boards left over, the last blocks first (the packs' shares
// of a short level fall to the first ones).  Not inlined: beside the packs'
// code it cost the packs 7%.
template <bool HALF>
__device__ __noinline__ void singles_level(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                                           const MidLevel lv, pp_super* __restrict__ table,
                                           pp_super* __restrict__ out, int final_level,
                                           const char* __restrict__ masks, uint32_t parity) {
  for (uint32_t vb = gridDim.x - 1 - blockIdx.x; vb < lv.blocks; vb += gridDim.x)
    midgame_fill<true, HALF>(boards, segs + lv.seg0, lv.nsegs, vb, table, out, final_level,
                             reinterpret_cast<const uint4*>(masks), lv.seg_blocks, parity);
}

// All levels of a plan's packs in one cooperative launch, then the roots; the
// boards left over one by one (singles) take their levels in the same steps.
// Children are read through L1: each is written once per launch, before the
// grid barrier that precedes its first read, and the barrier's fence drops
// what L1 held.
template <bool HALF, bool SINGLES>
__global__ void __launch_bounds__(kPackThreads, HALF ? PP_PACK_HALF_MINB : PP_PACK_MINB)
    pack_persistent_kernel(const MidBoard* __restrict__ boards, const MidSeg* __restrict__ segs,
                           const MidLevel* __restrict__ levels, int nlevels, const MidLevel* __restrict__ singles,
                           int nsingles, pp_super* __restrict__ table, pp_super* __restrict__ out, uint32_t* bar,
                           uint32_t* status, const char* __restrict__ masks, uint32_t parity, uint32_t spins) {
  static_assert(kPackThreads == kBlock, "singles run blocks of kBlock fills");
  __shared__ PackSeg sg;
  for (int L = 0; L < nlevels || (SINGLES && L < nsingles); L++) {
    if (L < nlevels) {
      const MidLevel lv = levels[L];
      pack_level<true, HALF>(boards, segs + lv.seg0, lv.nsegs, lv.blocks, lv.seg_blocks,
                             reinterpret_cast<char*>(table), masks, parity, sg);
    }
    if (SINGLES && L < nsingles)
      singles_level<HALF>(boards, segs, singles[L], table, out, L + 1 == nsingles, masks, parity);
    if (!grid_barrier(bar, status, spins)) return;
  }
  // the roots' addresses, too, from a load made after the last barrier (an
  // ordered load in pack_root instead cost packs beside single boards 5%)
  if (threadIdx.x == 0) sg.rec = reinterpret_cast<char*>(table);
  __syncthreads();
  const MidLevel lv = levels[nlevels - 1];
  for (uint32_t item = blockIdx.x * kPackThreads + threadIdx.x; item < (uint32_t)lv.nsegs * 32;
       item += gridDim.x * kPackThreads)
    pack_root<HALF>(boards, segs + lv.seg0, lv.seg_blocks, item, sg.rec, out, parity);
}

int launch_pack_level(const MidBoard* d_boards, const MidSeg* d_segs, int nsegs, uint32_t blocks, pp_super* d_table,
                      pp_super* d_out, int final_level, pp_stream s, const void* d_masks, uint32_t seg_blocks,
                      int parity) {
  if (!blocks) return 0;
  if (!d_masks) return (int)cudaErrorInvalidValue;
  char* table = reinterpret_cast<char*>(d_table);
  const char* masks = static_cast<const char*>(d_masks);
  const uint32_t p = parity >= 0 ? (uint32_t)parity : 0u;
  const uint32_t resident = (uint32_t)persistent_pack_blocks(0, parity >= 0, false);
  const uint32_t launched = resident && resident < blocks ? resident : blocks;
  if (parity >= 0)
    pack_level_kernel<true><<<launched, kPackThreads, 0, s>>>(d_boards, d_segs, nsegs, blocks, table, masks, seg_blocks, p);
  else
    pack_level_kernel<false><<<launched, kPackThreads, 0, s>>>(d_boards, d_segs, nsegs, blocks, table, masks, seg_blocks, p);
  count_launch();
  if (final_level) {
    const unsigned grid = ((unsigned)nsegs * 32 + 127) / 128;
    if (parity >= 0)
      pack_root_kernel<true><<<grid, 128, 0, s>>>(d_boards, d_segs, nsegs, table, d_out, seg_blocks, p);
    else
      pack_root_kernel<false><<<grid, 128, 0, s>>>(d_boards, d_segs, nsegs, table, d_out, seg_blocks, p);
    count_launch();
  }
  return (int)cudaGetLastError();
}

namespace {
const void* persistent_kernel(bool half, bool singles) {
  return half ? (singles ? (const void*)pack_persistent_kernel<true, true> : (const void*)pack_persistent_kernel<true, false>)
              : (singles ? (const void*)pack_persistent_kernel<false, true>
                         : (const void*)pack_persistent_kernel<false, false>);
}
}  // namespace

int persistent_pack_blocks(int ctas_per_sm, bool half, bool singles) {
  int dev = 0, sms = 0, per_sm = 0;
  if (cudaGetDevice(&dev) || cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) return 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, persistent_kernel(half, singles), kPackThreads, 0)) return 0;
  if (ctas_per_sm > 0 && ctas_per_sm < per_sm) per_sm = ctas_per_sm;
  return sms * per_sm;
}

int launch_pack_persistent(const MidBoard* d_boards, const MidSeg* d_segs, const MidLevel* d_levels, int nlevels,
                           const MidLevel* d_singles, int nsingles, pp_super* d_table, pp_super* d_out,
                           uint32_t* d_sync, int grid, pp_stream s, const void* d_masks, int parity) {
  if (grid <= 0 || nlevels <= 0 || !d_masks) return (int)cudaErrorInvalidValue;
  uint32_t* bar = d_sync;
  uint32_t* status = d_sync + 2;
  uint32_t p = parity >= 0 ? (uint32_t)parity : 0u;
  uint32_t spins = barrier_spins();
  void* args[] = {(void*)&d_boards, (void*)&d_segs,  (void*)&d_levels, (void*)&nlevels, (void*)&d_singles,
                  (void*)&nsingles, (void*)&d_table, (void*)&d_out,    (void*)&bar,     (void*)&status,
                  (void*)&d_masks,  (void*)&p,       (void*)&spins};
  cudaError_t e = cudaLaunchCooperativeKernel(persistent_kernel(parity >= 0, nsingles > 0), dim3(grid), dim3(kPackThreads), args, 0, s);
  count_launch();
  return (int)e;
}

}  // namespace pp
