// One warp's walk of one program piece over its tile of translations (the
// body shared by the single-image and the batched walk kernels).
//
// The program is a depth-first walk of the prefix tree of the canonical
// segments, baked into 16-byte groups (see lpf_paths.hpp): a record is a
// header group, then groups of four pixels (two pairs of pixels that read the
// same staged word window, or four single pixels), then at most one group
// with two single pixels.  Every pixel ANDs one funnel-shifted image word
// into the phase-1 mask and its complement into the phase-0 mask; emitting
// records count both masks (popc, warp sum, one atomic per phase);
// push/restore records keep branch masks on a small per-thread stack.  After
// every 8 pixels inside a record and at the end of an emitting or branching
// record the warp votes: once no translation of its tile is left in either
// phase, every count of the subtree below is zero there too, and the warp
// jumps to the record's skip target (the zero-count skip of Sec. 3.2,
// applied to whole subtrees).
//
// Masks only shrink down the tree, so most of the walk runs over tiles in
// which few words hold anything (512x512 ellipses, window 256, T = 4: 68 % of
// the pixels walked have at most 32 live (word, phase) masks of 256).  At a
// vote that finds at most 32 of them the warp therefore re-deals them, one
// per lane, and walks the subtree below on one mask per lane (the gathered
// walk): a pixel then costs one funnel shift and 3/4 of a three-input
// operation instead of T shifts and 2 T operations.  Every lane reads at its
// own word of the staged rows, so its loads meet in a bank now and then (45e6
// of 271e6 wavefronts), which the ALU time saved pays for (1.08e9 -> 0.70e9
// ALU instructions).  Restoring a mask that was pushed before the re-deal ends
// the gathered walk.  Measured, kernel alone: 512x512 ellipses, window 256: 2.46 -> 2.08 ms
// (issue slots 72 % busy: the decoding of records, 18 pixels each, is what is
// left); 175x201 squares, whole domain: 239 -> 191 us.
#pragma once
#include <cstdint>

#include "lpf_device.cuh"
#include "lpf_paths.hpp"

namespace lpf {

constexpr int kWalkStack = 24;

// A lane's T words: T / R words of each of R rows 32 rows apart (R > 1 folds
// the bands of narrow images into one tile, see layout_side); word t of the
// window is w[win<T, R>(t)] and its successor.
template <int T, int R>
__device__ __forceinline__ constexpr int win(int t) { return t + t / (T / R); }

// The R (T / R + 1) staged words of a pixel word's window; band: bytes from
// one of the lane's rows to the next.
template <int T, int R>
__device__ __forceinline__ void load_window(const uint32_t* lane_base, uint32_t pix, uint32_t band,
                                            uint32_t (&w)[T + R]) {
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const uint32_t* s = reinterpret_cast<const uint32_t*>(reinterpret_cast<const char*>(lane_word(lane_base, pix)) + r * band);
#pragma unroll
    for (int t = 0; t <= T / R; ++t) w[r * (T / R + 1) + t] = s[t];
  }
}

// Four single pixels (one group).
template <int T, int R>
__device__ __forceinline__ void walk_singles4(const uint32_t* lane_base, uint32_t band, uint4 P, uint32_t (&m1)[T],
                                              uint32_t (&m0)[T]) {
  if (T <= 4) {
    uint32_t wa[T + R], wb[T + R], wc[T + R], wd[T + R];
    load_window<T, R>(lane_base, P.x, band, wa);
    load_window<T, R>(lane_base, P.y, band, wb);
    load_window<T, R>(lane_base, P.z, band, wc);
    load_window<T, R>(lane_base, P.w, band, wd);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const uint32_t a = __funnelshift_r(wa[win<T, R>(t)], wa[win<T, R>(t) + 1], P.x);
      const uint32_t b = __funnelshift_r(wb[win<T, R>(t)], wb[win<T, R>(t) + 1], P.y);
      const uint32_t c = __funnelshift_r(wc[win<T, R>(t)], wc[win<T, R>(t) + 1], P.z);
      const uint32_t d = __funnelshift_r(wd[win<T, R>(t)], wd[win<T, R>(t) + 1], P.w);
      m1[t] = (m1[t] & a & b) & c & d;
      m0[t] = (m0[t] & ~a & ~b) & ~c & ~d;
    }
  } else {  // two pixels at a time (registers)
    uint32_t wa[T + R], wb[T + R];
    load_window<T, R>(lane_base, P.x, band, wa);
    load_window<T, R>(lane_base, P.y, band, wb);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const uint32_t a = __funnelshift_r(wa[win<T, R>(t)], wa[win<T, R>(t) + 1], P.x);
      const uint32_t b = __funnelshift_r(wb[win<T, R>(t)], wb[win<T, R>(t) + 1], P.y);
      m1[t] = m1[t] & a & b;
      m0[t] = m0[t] & ~a & ~b;
    }
    load_window<T, R>(lane_base, P.z, band, wa);
    load_window<T, R>(lane_base, P.w, band, wb);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const uint32_t a = __funnelshift_r(wa[win<T, R>(t)], wa[win<T, R>(t) + 1], P.z);
      const uint32_t b = __funnelshift_r(wb[win<T, R>(t)], wb[win<T, R>(t) + 1], P.w);
      m1[t] = m1[t] & a & b;
      m0[t] = m0[t] & ~a & ~b;
    }
  }
}

// Two single pixels.
template <int T, int R>
__device__ __forceinline__ void walk_singles2(const uint32_t* lane_base, uint32_t band, uint32_t p, uint32_t q, uint32_t (&m1)[T],
                                              uint32_t (&m0)[T]) {
  uint32_t wa[T + R], wb[T + R];
  load_window<T, R>(lane_base, p, band, wa);
  load_window<T, R>(lane_base, q, band, wb);
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const uint32_t a = __funnelshift_r(wa[win<T, R>(t)], wa[win<T, R>(t) + 1], p);
    const uint32_t b = __funnelshift_r(wb[win<T, R>(t)], wb[win<T, R>(t) + 1], q);
    m1[t] = m1[t] & a & b;
    m0[t] = m0[t] & ~a & ~b;
  }
}

// Two pairs {window|shift1, shift2} (one group): one window per pair.
template <int T, int R>
__device__ __forceinline__ void walk_pairs2(const uint32_t* lane_base, uint32_t band, uint4 P, uint32_t (&m1)[T], uint32_t (&m0)[T]) {
  uint32_t wa[T + R], wb[T + R];
  load_window<T, R>(lane_base, P.x, band, wa);
  load_window<T, R>(lane_base, P.z, band, wb);
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const uint32_t a1 = __funnelshift_r(wa[win<T, R>(t)], wa[win<T, R>(t) + 1], P.x), a2 = __funnelshift_r(wa[win<T, R>(t)], wa[win<T, R>(t) + 1], P.y);
    const uint32_t b1 = __funnelshift_r(wb[win<T, R>(t)], wb[win<T, R>(t) + 1], P.z), b2 = __funnelshift_r(wb[win<T, R>(t)], wb[win<T, R>(t) + 1], P.w);
    m1[t] = (m1[t] & a1 & a2) & b1 & b2;
    m0[t] = (m0[t] & ~a1 & ~a2) & ~b1 & ~b2;
  }
}

// Lanes that hold a translation of either phase (one vote); 0: none is left.
// (LANES = false: only whether there are any.)
template <int T, bool LANES>
__device__ __forceinline__ uint32_t live_lanes(const uint32_t (&m1)[T], const uint32_t (&m0)[T]) {
  uint32_t any = 0;
#pragma unroll
  for (int t = 0; t < T; ++t) any |= m1[t] | m0[t];
  return LANES ? __ballot_sync(0xffffffffu, any != 0) : (uint32_t)__any_sync(0xffffffffu, any != 0);
}

// Gathered walk: one mask m per lane, of phase 0 where f = ~0 and of phase 1
// where f = 0; word = shared address of its word in the staged rows (lanes
// whose mask is empty read the word of lane 0's, so that only live lanes meet
// in banks).

__device__ __forceinline__ uint32_t shared_word(uint32_t addr) {
  uint32_t r;
  asm("ld.shared.u32 %0, [%1];" : "=r"(r) : "r"(addr));
  return r;
}

// a & b for phase 1 (f = 0), ~a & ~b for phase 0 (f = ~0): one operation.
__device__ __forceinline__ uint32_t both_phase(uint32_t a, uint32_t b, uint32_t f) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0x42;" : "=r"(r) : "r"(a), "r"(b), "r"(f));
  return r;
}

__device__ __forceinline__ uint32_t gathered_pairs2(uint32_t word, uint4 P, uint32_t f, uint32_t m) {
  const uint32_t s = word + (P.x >> 5), r = word + (P.z >> 5);
  const uint32_t s0 = shared_word(s), s1 = shared_word(s + 4u), r0 = shared_word(r), r1 = shared_word(r + 4u);
  const uint32_t a = both_phase(__funnelshift_r(s0, s1, P.x), __funnelshift_r(s0, s1, P.y), f);
  const uint32_t b = both_phase(__funnelshift_r(r0, r1, P.z), __funnelshift_r(r0, r1, P.w), f);
  return m & a & b;
}

__device__ __forceinline__ uint32_t gathered_singles2(uint32_t word, uint32_t p, uint32_t q, uint32_t f, uint32_t m) {
  const uint32_t s = word + (p >> 5), r = word + (q >> 5);
  return m & both_phase(__funnelshift_r(shared_word(s), shared_word(s + 4u), p),
                        __funnelshift_r(shared_word(r), shared_word(r + 4u), q), f);
}

// The subtree below a re-deal: walks from group q of record rec on (q past
// the record's groups: its pixels are done) until a record that resets or
// restores a mask pushed before, which the caller goes on with.  Same groups
// and votes as walk_unit on one mask per lane.  Returns that record and the
// pixels walked, counted as walk_unit does (rec's own are counted by the
// caller).  counts: of the canonical vectors, phase 0.  A function of its own:
// inlined, it costs the walk of the full masks registers and 20 % of its time
// (128^3, window 16).
static __device__ __noinline__ uint2 gathered_walk(const uint4* __restrict__ prog, uint32_t rec, uint32_t end,
                                                   uint32_t q, uint32_t own, uint32_t f, uint32_t m,
                                                   unsigned long long* __restrict__ counts, int64_t n_full) {
  uint32_t stack[kWalkStack];
  const uint32_t idle = __shfl_sync(0xffffffffu, own, 0);
  uint32_t word = m ? own : idle;
  uint32_t levels = 0;  // stack levels pushed here
  uint32_t walked = 0;
  uint4 hd = __ldg(prog + rec);
  for (;;) {
    const uint32_t hdr = hd.x, skip = hd.z, cnt = hd.w;
    const uint32_t n_pg = cnt & kCntMask, n_sg = (cnt >> kCntBits) & kCntMask, half = cnt >> (2 * kCntBits);
    const uint32_t next = rec + 1u + n_pg + n_sg + half;
    const uint32_t vec = hd.y, n = hdr & kNpixMask;
    hd = next < end ? __ldg(prog + next) : make_uint4(0u, 0u, 0u, 0u);  // fetched while this record runs
    const uint4* g = prog + rec + 1u;
    bool dead = false;
    for (; q + 2u <= n_pg; q += 2u) {
      const uint4 P0 = __ldg(g + q), P1 = __ldg(g + q + 1u);
      m = gathered_pairs2(word, P0, f, m);
      m = gathered_pairs2(word, P1, f, m);
      if (skip != 0u && !__any_sync(0xffffffffu, m != 0u)) {
        dead = true;
        walked -= n - 4u * (q + 2u);
        break;
      }
      word = m ? word : idle;
    }
    if (!dead) {
      if (q < n_pg) { m = gathered_pairs2(word, __ldg(g + q), f, m); q = n_pg; }
      for (; q + 2u <= n_pg + n_sg; q += 2u) {
        const uint4 P0 = __ldg(g + q), P1 = __ldg(g + q + 1u);
        m = gathered_singles2(word, P0.x, P0.y, f, m);
        m = gathered_singles2(word, P0.z, P0.w, f, m);
        m = gathered_singles2(word, P1.x, P1.y, f, m);
        m = gathered_singles2(word, P1.z, P1.w, f, m);
        if (skip != 0u && !__any_sync(0xffffffffu, m != 0u)) {
          dead = true;
          const uint32_t done = 4u * (q + 2u);
          walked -= n > done ? n - done : 0u;
          break;
        }
      }
    }
    if (!dead) {
      if (q < n_pg + n_sg) {
        const uint4 P = __ldg(g + q);
        m = gathered_singles2(word, P.x, P.y, f, m);
        m = gathered_singles2(word, P.z, P.w, f, m);
        q = n_pg + n_sg;
      }
      if (half && q == n_pg + n_sg) {
        const uint4 P = __ldg(g + n_pg + n_sg);
        m = gathered_singles2(word, P.x, P.y, f, m);
      }
      if ((hdr & (kEmit | kPush)) && skip != 0u && !__any_sync(0xffffffffu, m != 0u)) dead = true;
    }
    if (dead) {
      rec += skip;
      hd = rec < end ? __ldg(prog + rec) : make_uint4(0u, 0u, 0u, 0u);
    } else {
      if (hdr & kEmit) {
        const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)__popc(m) << (f & 16u));
        if ((threadIdx.x & 31u) == 0u) {
          const uint32_t c1 = c & 0xffffu, c0 = c >> 16;
          if (c0) atomicAdd(counts + vec, (unsigned long long)c0);
          if (c1) atomicAdd(counts + n_full + vec, (unsigned long long)c1);
        }
      }
      if (hdr & kPush) {
        const int l = (hdr >> kPlevelShift) & kLevelMask;
        stack[l] = m;
        levels |= 1u << l;
      }
      rec = next;
    }
    if (rec >= end || (hd.x & kReset)) break;
    if (hd.x & kRestore) {
      const int l = (hd.x >> kRlevelShift) & kLevelMask;
      if (!((levels >> l) & 1u)) break;
      m = stack[l];
    }
    word = m ? own : idle;
    q = 0u;
    walked += hd.x & kNpixMask;
  }
  return make_uint2(rec, walked);
}

// Groups of program below which a re-deal does not pay (it costs about 100
// instructions, a group saves about 30; 6, 12 and 24 measured the same).
constexpr uint32_t kGatherGroups = 12;
constexpr int kMaxLive = 32;  // one mask per lane (16: 11 % slower at 512x512, window 256)
// Windows from which tiles empty out enough to re-deal (kernels of their own:
// their code costs a launch 4 us and a walk that never re-deals 3 to 6 %); at
// window 128 a third of the walk is gathered.  Images walked one at a time
// also need four words per thread or more (with two, 334x50, window 25x167,
// took 88 instead of 73 us) and two units per warp slot (112x93, whole
// domain: 93 instead of 87 us); at window 119 (239x230) it is a loss of 2 %,
// at 143 (210x286) a gain of a third; batches, whose images share a kernel, pay
// from windows of 120 (96 and less: 3 to 5 % slower).  Volumes do not re-deal.
constexpr int kGatherWindow = 128;
constexpr int kGatherWindowBatch = 120;

// Valid translations of a tile: word t of the lane (row y + 32 (t / (T / R)))
// holds translations x = 32 (j0 + t mod T / R) + bit; those with x < W in a
// row < H exist (and, with a selection, only the selected ones).
template <int T, int R>
__device__ __forceinline__ void tile_valid(int y0, int H, int W, int nw, int j0, const uint32_t* __restrict__ sel,
                                           uint32_t (&v)[T]) {
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int j = j0 + t % (T / R), y = y0 + 32 * (t / (T / R));
    uint32_t m = 0;
    if (y < H && j < nw) {
      const int rem = W - 32 * j;
      m = rem >= 32 ? 0xffffffffu : ((1u << rem) - 1u);
      if (sel) m &= sel[(size_t)y * nw + j];
    }
    v[t] = m;
  }
}

// Walk program groups [pc, end) for this warp's tile.  lane_base: the lane's
// first staged word (shared memory; row = the lane's first translation row),
// band: bytes to its next row (R > 1); deal:
// 32 entries of the warp's own for re-dealing its masks (GATHER), or null
// (never re-deals).  Counts go to counts[base + vec] (phase 0) and counts[n_full +
// base + vec] (phase 1).  Returns the pixels this warp walked (for the work
// statistics).
// UNROLL4: pair groups four per loop iteration (less loop control, more
// code: the batched kernel keeps two).
template <int T, int R, bool GATHER, bool UNROLL4 = true>
__device__ __forceinline__ uint32_t walk_unit(const uint4* __restrict__ prog, uint32_t pc, uint32_t end,
                                              const uint32_t* lane_base, uint32_t band, uint2* deal, int y, int H, int W, int nw,
                                              int j0, const uint32_t* __restrict__ sel, int lane,
                                              unsigned long long* __restrict__ counts, int64_t n_full,
                                              int64_t base) {
  constexpr bool kGather = GATHER && T >= 2;  // (one word per lane already: nothing to win)
  uint32_t m1[T], m0[T];
  uint32_t st1[kWalkStack][T], st0[kWalkStack][T];
  tile_valid<T, R>(y, H, W, nw, j0, sel, m1);
#pragma unroll
  for (int t = 0; t < T; ++t) m0[t] = m1[t];
  uint32_t walked = 0;
  // If at most 32 masks are live: re-deal them and walk on from group q of
  // record rec; the record to go on with, else 0 (no record follows a
  // subtree at 0).
  auto gather = [&](uint32_t rec, uint32_t q) -> uint32_t {
    int c = 0;
#pragma unroll
    for (int t = 0; t < T; ++t) c += (m1[t] != 0) + (m0[t] != 0);
    const int n = __reduce_add_sync(0xffffffffu, c);
    if (n > kMaxLive) return 0u;
    int at = c;  // exclusive sum over the lanes
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, at, o);
      if (lane >= o) at += v;
    }
    at -= c;
    const uint32_t word = smem_u32(lane_base);
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const uint32_t at_t = word + band * (t / (T / R)) + 4u * (t % (T / R));
      if (m1[t]) deal[at++] = make_uint2(at_t, m1[t]);
      if (m0[t]) deal[at++] = make_uint2(at_t | 1u, m0[t]);
    }
    __syncwarp();
    const uint2 d = lane < n ? deal[lane] : make_uint2(word, 0u);
    __syncwarp();
    const uint2 r = gathered_walk(prog, rec, end, q, d.x & ~1u, (d.x & 1u) ? 0xffffffffu : 0u, d.y, counts + base,
                                  n_full);
    walked += r.y;
    return r.x;
  };
  uint4 hd = pc < end ? __ldg(prog + pc) : make_uint4(0u, 0u, 0u, 0u);
  while (pc < end) {
    const uint32_t rec = pc;
    const uint32_t hdr = hd.x, skip = hd.z, cnt = hd.w;
    const uint32_t n_pg = cnt & kCntMask, n_sg = (cnt >> kCntBits) & kCntMask, half = cnt >> (2 * kCntBits);
    const uint32_t next = rec + 1u + n_pg + n_sg + half;
    const int vec = (int)hd.y;
    hd = next < end ? __ldg(prog + next) : make_uint4(0u, 0u, 0u, 0u);  // fetched while this record runs
    if (hdr & kReset) {
      tile_valid<T, R>(y, H, W, nw, j0, sel, m1);
#pragma unroll
      for (int t = 0; t < T; ++t) m0[t] = m1[t];
    }
    if (hdr & kRestore) {
      const int l = (hdr >> kRlevelShift) & kLevelMask;
#pragma unroll
      for (int t = 0; t < T; ++t) { m1[t] = st1[l][t]; m0[t] = st0[l][t]; }
    }
    const uint32_t n = hdr & kNpixMask;
    walked += n;
    bool dead = false;
    uint32_t to = 0;  // where a gathered walk of the subtree ended
    const uint4* g = prog + rec + 1u;
    // four groups (16 pixels) per iteration, their program loads issued
    // together, a vote after every two (8 pixels); then pairs of groups
    uint32_t q = 0;
    for (; UNROLL4 && q + 4u <= n_pg; q += 4u) {
      const uint4 P0 = __ldg(g + q), P1 = __ldg(g + q + 1u), P2 = __ldg(g + q + 2u), P3 = __ldg(g + q + 3u);
      walk_pairs2<T, R>(lane_base, band, P0, m1, m0);
      walk_pairs2<T, R>(lane_base, band, P1, m1, m0);
      if (skip != 0u && !live_lanes<T, false>(m1, m0)) {
        dead = true;
        walked -= n - 4u * (q + 2u);  // pixels not walked (pair groups hold four pixels of the record)
        break;
      }
      walk_pairs2<T, R>(lane_base, band, P2, m1, m0);
      walk_pairs2<T, R>(lane_base, band, P3, m1, m0);
      if (skip != 0u) {
        const uint32_t lanes = live_lanes<T, kGather>(m1, m0);
        if (!lanes) {
          dead = true;
          walked -= n - 4u * (q + 4u);
          break;
        }
        if (kGather && deal && skip >= q + kGatherGroups && __popc(lanes) <= kMaxLive - 4) {
          to = gather(rec, q + 4u);
          if (to) break;
        }
      }
    }
    for (; !dead && !to && q + 2u <= n_pg; q += 2u) {
      const uint4 P0 = __ldg(g + q), P1 = __ldg(g + q + 1u);
      walk_pairs2<T, R>(lane_base, band, P0, m1, m0);
      walk_pairs2<T, R>(lane_base, band, P1, m1, m0);
      if (skip != 0u && !live_lanes<T, false>(m1, m0)) {
        dead = true;
        walked -= n - 4u * (q + 2u);
        break;
      }
    }
    if (!dead && !to && q < n_pg) walk_pairs2<T, R>(lane_base, band, __ldg(g + q), m1, m0);
    if (!dead && !to) {
      g += n_pg;
      for (q = 0; q + 2u <= n_sg; q += 2u) {
        const uint4 P0 = __ldg(g + q), P1 = __ldg(g + q + 1u);
        walk_singles4<T, R>(lane_base, band, P0, m1, m0);
        walk_singles4<T, R>(lane_base, band, P1, m1, m0);
        if (skip != 0u && !live_lanes<T, false>(m1, m0)) {
          dead = true;
          const uint32_t done = 4u * (n_pg + q + 2u);
          walked -= n > done ? n - done : 0u;
          break;
        }
      }
      if (!dead) {
        if (q < n_sg) walk_singles4<T, R>(lane_base, band, __ldg(g + q), m1, m0);
        if (half) {
          const uint4 P = __ldg(g + n_sg);
          walk_singles2<T, R>(lane_base, band, P.x, P.y, m1, m0);
        }
      }
    }
    if (dead || to) {
      pc = dead ? rec + skip : to;
      hd = pc < end ? __ldg(prog + pc) : make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    if (hdr & (kEmit | kPush)) {
      if (skip != 0u) {
        // Empty for the whole warp (one vote): so is every count below this node.
        const uint32_t lanes = live_lanes<T, kGather>(m1, m0);
        if (!lanes) to = rec + skip;
        else if (kGather && deal && next + kGatherGroups <= rec + skip && __popc(lanes) <= kMaxLive - 4)
          to = gather(rec, n_pg + n_sg + 1u);
        if (to) {
          pc = to;
          hd = pc < end ? __ldg(prog + pc) : make_uint4(0u, 0u, 0u, 0u);
          continue;
        }
      }
      if (hdr & kEmit) {
        uint32_t c = 0;
#pragma unroll
        for (int t = 0; t < T; ++t) c += (uint32_t)__popc(m1[t]) + ((uint32_t)__popc(m0[t]) << 16);
        c = __reduce_add_sync(0xffffffffu, c);  // one warp-reduce instruction
        if (lane == 0) {
          const uint32_t c1 = c & 0xffffu, c0 = c >> 16;
          if (c0) atomicAdd(counts + base + vec, (unsigned long long)c0);
          if (c1) atomicAdd(counts + n_full + base + vec, (unsigned long long)c1);
        }
      }
    }
    if (hdr & kPush) {
      const int l = (hdr >> kPlevelShift) & kLevelMask;
#pragma unroll
      for (int t = 0; t < T; ++t) { st1[l][t] = m1[t]; st0[l][t] = m0[t]; }
    }
    pc = next;
  }
  return walked;
}

}  // namespace lpf
