// Count and error changes of candidate exchanges from bit planes (the
// annealer's modification operator, Sec. 4; the definition is in
// lpf_delta.cu).
//
// For one vector v with n = |S(v)| pixels let z(x) be the number of phase-0
// pixels of S(v) + x.  Exchanging a (phase 1) and b (phase 0) changes counts
// only on translations through one of them:
//   through a, z = 0       was all phase 1:              d1 -= 1
//   through a, z = n - 1   is all phase 0 after, unless it contains b: d0 += 1
//   through b, z = n       was all phase 0:              d0 -= 1
//   through b, z = 1       is all phase 1 after, unless it contains a: d1 += 1
// So all that is needed of v are three bits per translation: U (uniform: z =
// 0 or n), X1 (one phase-1 pixel: z = n - 1) and X0 (one phase-0 pixel: z =
// 1).  A block walks v over the bit-packed cell, 32 translations per word,
// with four masks (all phase 1, all phase 0, one phase-1 pixel so far, one
// phase-0 pixel so far: one funnel shift and four three-input operations per
// pixel and word), and then either
//   many candidates: adds the planes along S(v) for every pixel q at once --
//     u(q) = sum_i U(q - s_i) and m(q) = sum_i X_phase(q)(q - s_i), 32 pixels
//     per word in bit-sliced carry-save counters, turned into a byte per
//     pixel by 8x8 bit transposes -- and a candidate costs four byte reads,
//     plus, where a and b may share a segment of v, one pass over its pixels;
//   few candidates: looks the bits of the 2n translations up directly, a warp
//     per candidate.
//
// What bounds it: issue (logic and shared-memory loads) of the walk and the
// sums, sum_v n(v) H W / 32 word steps of about 9 and 22 instructions, with
// everything in shared memory; candidates add about 40 instructions per
// vector.  HBM holds no tables: the phase-0 counts that this replaces were
// one byte per vector and translation (136 MB at 128x128, window 64), filled
// and read by 2n scattered lookups per candidate and vector.
// Measured (error changes, a call): 4096 candidates on a 128x128 clustered
// cell, window 64: 15.66 -> 0.52 ms; 64 candidates on a 50x50 cell, full
// domain, with count changes: 0.300 -> 0.075 ms.
//
// Error changes are summed per (part of a chunk, candidate) in vector order
// and then over the parts in a fixed order that depends on the cell and window
// alone: bitwise reproducible, whatever the number of candidates.
#include <algorithm>

#include "lpf_delta.cuh"
#include "lpf_state.hpp"
#include "lpf_swap.hpp"

namespace lpf {

constexpr int kSwapThreads = 256;  // 2 words per thread at 128x128; 3 blocks (62 KB, 85 registers) per SM
constexpr int kSwapWarps = kSwapThreads / 32;
constexpr int kSwapMaxPixels = 255;  // pixels of a segment (the sums are bytes)

// Candidates, a holding phase 1 (both pixels 0: identity), as two arrays of K:
// the byte offsets of a and b in the sum tables, which every vector reads, and
// a and b as y << 16 | x, which few (vector, candidate) pairs need.
struct SwapCands {
  uint2 *table, *pixel;
};
constexpr int kSwapUnroll = 4;  // candidates a thread has in flight where it has several

struct SwapArgs {
  int H, W, nw, S, rx, ry, r32;
  int split;               // parts of a vector chunk, a block each
  int words;               // H * nw; word (y, j) of a plane is y + H j
  int tg, G;               // threads per vector, vectors side by side in a block
  int nmax;                // longest segment, rounded up to 8
  uint32_t inv_H, inv_S;   // ceil(2^32 / H), ceil(2^32 / S): i / H = umulhi(i, inv_H) while i H < 2^32
  const uint32_t* img;     // packed rows: (H + ry) rows of S words, bit e = column (e - r32) mod W
  const uint32_t* sel;     // selected start translations by word, or null
  const int32_t* dptr;
  const int16_t* off16;
  const int16_t* vec16;
  const int32_t* chunk;
  int64_t n_canon;
  const float* target;     // of the canonical vectors, phase 0 (phase 1 n_full later), or null
  const int64_t* counts;
  int64_t n_full;
  int phase_mask;
  float inv_norm;
};

// i / n by the reciprocal inv = ceil(2^32 / n) (n > 1; n = 1 has inv = 0).
__device__ __forceinline__ int fast_div(int i, uint32_t inv) { return inv ? (int)__umulhi((uint32_t)i, inv) : i; }

static int swap_img_words(int H, int ry, int S) { return ((H + ry) * S + 3) & ~3; }

// Bytes of dynamic shared memory.
static size_t swap_smem(const SwapArgs& g, bool many) {
  const size_t img = (size_t)swap_img_words(g.H, g.ry, g.S) * 4;
  const size_t group = many ? (size_t)g.words * 64 + 4 * img : (size_t)((g.words * 3 + 3) & ~3) * 4;
  return img + (size_t)((g.S + 3) & ~3) * 4 + (size_t)g.G * (group + (size_t)3 * g.nmax * 4) + 64;
}

// Packed rows of the cell (img), selection words and candidates; flags as
// build_ext_kernel and delta_kernel set them.
__global__ void swap_prep_kernel(const uint8_t* __restrict__ cell, SwapArgs g, uint32_t* __restrict__ img,
                                 const uint8_t* __restrict__ sel_ext, int We, uint32_t* __restrict__ sel,
                                 const int32_t* __restrict__ pairs, int K, SwapCands cand,
                                 int* __restrict__ status, int checked) {
  const int stride = gridDim.x * blockDim.x, i0 = blockIdx.x * blockDim.x + threadIdx.x;
  uint32_t high = 0;
  for (int i = i0; i < (g.H + g.ry) * g.S; i += stride) {
    const int r = i / g.S, k = i - r * g.S;
    const uint8_t* row = cell + (size_t)(r < g.H ? r : r - g.H) * g.W;
    int x = (32 * k - g.r32) % g.W;
    if (x < 0) x += g.W;
    uint32_t bits = 0;
    for (int b = 0; b < 32; ++b) {
      const uint32_t v = row[x];
      bits |= (uint32_t)(v != 0) << b;
      high |= v >> 1;
      if (++x == g.W) x = 0;
    }
    img[i] = bits;
  }
  if (checked && high) atomicOr(status, 8);
  if (sel)
    for (int i = i0; i < g.words; i += stride) {
      const int j = i / g.H, y = i - j * g.H;
      uint32_t bits = 0;
      for (int b = 0; b < 32 && 32 * j + b < g.W; ++b)
        bits |= (uint32_t)(sel_ext[(size_t)(y + g.ry) * We + 32 * j + b + g.rx] != 0) << b;
      sel[i] = bits;
    }
  const int npix = g.H * g.W;
  for (int k = i0; k < K; k += stride) {
    int a = pairs[2 * k], b = pairs[2 * k + 1];
    uint2 t = make_uint2(0u, 0u), c = make_uint2(0u, 0u);
    if (a < 0 || b < 0 || a >= npix || b >= npix) {
      atomicOr(status, 2);                                    // identity
    } else if ((cell[a] != 0) != (cell[b] != 0)) {
      if (cell[a] == 0) { const int t = a; a = b; b = t; }
      const int ay = a / g.W, ax = a - ay * g.W, by = b / g.W, bx = b - by * g.W;
      t.x = (uint32_t)(((ay + g.H * (ax >> 5)) * 8 + (ax & 7)) * 4 + ((ax >> 3) & 3));
      t.y = (uint32_t)(((by + g.H * (bx >> 5)) * 8 + (bx & 7)) * 4 + ((bx >> 3) & 3));
      c.x = (uint32_t)ay << 16 | (uint32_t)ax;
      c.y = (uint32_t)by << 16 | (uint32_t)bx;
    }
    cand.table[k] = t;
    cand.pixel[k] = c;
  }
}

// Carry-save counter of 32 pixels: bit p of every pixel's sum in c[p].
struct BitCounter {
  uint32_t c[8];
};

__device__ __forceinline__ uint32_t csa(uint32_t& s, uint32_t a, uint32_t b) {
  const uint32_t carry = (s & a) | (s & b) | (a & b);
  s ^= a ^ b;
  return carry;
}

__device__ __forceinline__ void add8(BitCounter& q, const uint32_t (&d)[8]) {
  const uint32_t ta = csa(q.c[0], d[0], d[1]), tb = csa(q.c[0], d[2], d[3]);
  const uint32_t fa = csa(q.c[1], ta, tb);
  const uint32_t tc = csa(q.c[0], d[4], d[5]), td = csa(q.c[0], d[6], d[7]);
  const uint32_t fb = csa(q.c[1], tc, td);
  uint32_t e = csa(q.c[2], fa, fb);
#pragma unroll
  for (int p = 3; p < 8; ++p) {
    const uint32_t t = q.c[p] & e;
    q.c[p] ^= e;
    e = t;
  }
}

// The bit planes of 32 pixels as bytes: byte k of c[j] becomes the sum of
// pixel 8 k + j (an 8x8 bit transpose of every byte column).
__device__ __forceinline__ void to_bytes(BitCounter& q) {
#pragma unroll
  for (int s = 0; s < 3; ++s) {
    const int d = 1 << s;
    const uint32_t m = s == 0 ? 0x55555555u : s == 1 ? 0x33333333u : 0x0f0f0f0fu;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
      if (a & d) continue;
      const uint32_t t = ((q.c[a] >> d) ^ q.c[a + d]) & m;
      q.c[a + d] ^= t;
      q.c[a] ^= t << d;
    }
  }
}

// Columns p0 .. p0 + 31 (periodic) of row y of the three planes without
// halo (plane_words apart).
__device__ __forceinline__ uint4 plane_columns(const uint32_t* planes, int plane_words, int y, int p0, int H, int W,
                                               int nw) {
  uint32_t w[3];
  if (W >= 32) {
    const int j = p0 >> 5, have = W - p0;
    const uint32_t* at = planes + y + H * j;
    const bool more = j + 1 < nw;
#pragma unroll
    for (int q = 0; q < 3; ++q) w[q] = __funnelshift_r(at[q * plane_words], more ? at[q * plane_words + H] : 0u, p0 & 31);
    if (have < 32) {
#pragma unroll
      for (int q = 0; q < 3; ++q) w[q] = (w[q] & ((1u << have) - 1u)) | planes[q * plane_words + y] << have;
    }
  } else {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const uint32_t row = planes[q * plane_words + y];  // W bits
      w[q] = row >> p0;
      for (int have = W - p0; have < 32; have += W) w[q] |= row << have;
    }
  }
  return make_uint4(w[0], w[1], w[2], 0u);
}

// Eight segment pixels (entries s[0..7], the last 8 - live of them absent)
// added to the counters of 32 pixels; p: the word's planes with halo.
template <bool FULL>
__device__ __forceinline__ void add_pixels(BitCounter& cu, BitCounter& cn, const uint4* p, const uint32_t* s,
                                           uint32_t chi, int live) {
  uint32_t du[8], dn[8];
  const uint4 s0 = *reinterpret_cast<const uint4*>(s), s1 = *reinterpret_cast<const uint4*>(s + 4);
  const uint32_t e[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
#pragma unroll
  for (int t = 0; t < 8; ++t) {
    du[t] = dn[t] = 0u;
    if (FULL || t < live) {
      const uint4* q = p + (e[t] >> 5);
      const uint4 lo = q[0], hi = q[1];
      du[t] = __funnelshift_r(lo.x, hi.x, e[t]);
      const uint32_t x1 = __funnelshift_r(lo.y, hi.y, e[t]), x0 = __funnelshift_r(lo.z, hi.z, e[t]);
      dn[t] = (chi & x1) | (~chi & x0);
    }
  }
  add8(cu, du);
  add8(cn, dn);
}

// One segment pixel of the walk: c = the image under 32 translations.
__device__ __forceinline__ void walk_masks(uint32_t c, uint32_t& all1, uint32_t& all0, uint32_t& one1, uint32_t& one0) {
  one1 = (all0 & c) | (one1 & ~c);
  one0 = (all1 & ~c) | (one0 & c);
  all0 &= ~c;
  all1 &= c;
}

// Whether a segment of vector (dx, dy) can hold two pixels q and q + (ddx,
// ddy) of the torus (ddx in (-W, W), ddy in (-H, H)): some representative of
// the displacement lies in the segment's box and within a = max(|dx|, dy) of
// the line along v (every pixel of S(v) lies within a / 2 of it).
__device__ __forceinline__ bool swap_maybe_both(int dx, int dy, int ddx, int ddy, int H, int W) {
  const int adx = dx < 0 ? -dx : dx, a = adx > dy ? adx : dy;
  bool any = false;
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int ex = (r & 1) ? (ddx > 0 ? ddx - W : ddx + W) : ddx;
    const int ey = (r & 2) ? (ddy > 0 ? ddy - H : ddy + H) : ddy;
    const int cross = ey * dx - ex * dy;
    any |= (ex < 0 ? -ex : ex) <= adx && (ey < 0 ? -ey : ey) <= dy && (cross < 0 ? -cross : cross) <= a;
  }
  return any;
}

// True when pixel (qx, qy) lies on S(v) placed at translation (x, y) (torus;
// the segment spans fewer than W columns and H rows); seg in shared memory.
__device__ __forceinline__ bool swap_on_segment(const short2* seg, int dx, int dy, int x, int y, int qx, int qy,
                                                int H, int W) {
  int uy = qy - y;
  if (uy < 0) uy += H;
  if (uy > dy) return false;
  const int xlo = dx < 0 ? dx : 0, xhi = dx < 0 ? 0 : dx;
  int ux = qx - x - xlo;
  if (ux < 0) ux += W;
  else if (ux >= W) ux -= W;
  ux += xlo;
  if (ux > xhi) return false;
  const int adx = dx < 0 ? -dx : dx;
  if (adx >= dy) return seg[dx < 0 ? -ux : ux].y == uy;  // x-major: pixel k at sx = sign(dx) k
  return seg[uy].x == ux;                                  // y-major: pixel k at sy = k
}

// Translation of the segment whose pixel (sx, sy) is (qx, qy).
__device__ __forceinline__ void swap_start(int qx, int qy, short2 s, int H, int W, int& x, int& y) {
  x = qx - s.x;
  y = qy - s.y;
  x = x < 0 ? x + W : (x >= W ? x - W : x);
  y = y < 0 ? y + H : y;  // 0 <= sy
}

// The float32 error change of one vector added to acc: for a phase with
// count change d and dd = target - count / N, (dd - x)^2 - dd^2 with x = d / N.
__device__ __forceinline__ float swap_add_error(float acc, int d0, int d1, float dd0, float dd1, const SwapArgs& g) {
  if (d0 && (g.phase_mask & 1)) {
    const float x = (float)d0 * g.inv_norm;
    acc += x * (x - 2.0f * dd0);
  }
  if (d1 && (g.phase_mask & 2)) {
    const float x = (float)d1 * g.inv_norm;
    acc += x * (x - 2.0f * dd1);
  }
  return acc;
}

// Block = one part of a vector chunk (x) and one share of the candidates (y);
// its threads form G groups of tg, which take the part's vectors G at a time.
// U: candidates that a thread takes at a time, 0: the way of few candidates.
// partial[part][K] (or null), dcounts [K][2][n_canon] (or null).
template <int U>
__global__ void __launch_bounds__(kSwapThreads, 3) swap_kernel(SwapArgs g, SwapCands cand, int K,
                                                               int32_t* __restrict__ dcounts,
                                                               float* __restrict__ partial) {
  constexpr bool MANY = U > 0;
  constexpr int kU = MANY ? U : 1;
  extern __shared__ __align__(16) uint32_t smw[];
  // per group (at most one per warp): whether some translation is in one of
  // the planes, and its vector (the candidates' loop reads no global memory
  // but the candidates: its loads used to set the pace of small cells)
  __shared__ int s_any[kSwapWarps], s_n[kSwapWarps];
  __shared__ short2 s_vec[kSwapWarps];
  __shared__ float s_dd[kSwapWarps][2];
  const int H = g.H, W = g.W, S = g.S;
  const int img_words = ((H + g.ry) * S + 3) & ~3;
  const int ext_words = img_words;  // words of a plane with halo (padded: groups start on 16 bytes)
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nthr = blockDim.x, nwarps = nthr >> 5;
  uint32_t* s_img = smw;
  int* s_col = reinterpret_cast<int*>(s_img + img_words);  // column (32 k - r32) mod W
  uint32_t* s_groups = reinterpret_cast<uint32_t*>(s_col + ((S + 3) & ~3));
  const int plane_words = MANY ? g.words * 16 : (g.words * 3 + 3) & ~3;  // planes; many: then the sum tables
  const int group_words = plane_words + (MANY ? 4 * ext_words : 0) + 3 * g.nmax;
  const int gi = tid / g.tg, gt = tid - gi * g.tg;
  uint32_t* base = s_groups + gi * group_words;
  uint4* ext = reinterpret_cast<uint4*>(base + plane_words);  // {U, X1, X0, 0} by word of the packed rows
  uint32_t* segA = base + group_words - 3 * g.nmax;
  uint32_t* segB = segA + g.nmax;
  short2* segP = reinterpret_cast<short2*>(segB + g.nmax);

  for (int i = tid; i < (H + g.ry) * S; i += nthr) s_img[i] = __ldg(g.img + i);
  for (int k = tid; k < S; k += nthr) {
    int c = (32 * k - g.r32) % W;
    s_col[k] = c < 0 ? c + W : c;
  }
  const int ch = blockIdx.x / g.split, sub = blockIdx.x - ch * g.split;
  const int c0 = g.chunk[ch], nc = g.chunk[ch + 1] - c0;
  const int v0 = c0 + (int)((int64_t)nc * sub / g.split), v1 = c0 + (int)((int64_t)nc * (sub + 1) / g.split);
  const int k_lo = (int)((int64_t)K * blockIdx.y / gridDim.y), k_hi = (int)((int64_t)K * (blockIdx.y + 1) / gridDim.y);
  float* part = partial ? partial + (int64_t)blockIdx.x * K : nullptr;
  if (part) {
    if (MANY)
      for (int k = k_lo + tid; k < k_hi; k += nthr) part[k] = 0.0f;
    else if (lane == 0)
      for (int k = k_lo + warp; k < k_hi; k += nwarps) part[k] = 0.0f;
  }

  for (int vb = v0; vb < v1; vb += g.G) {
    // ---- the planes of vector vb + gi
    const int v = vb + gi;
    const bool mine = v < v1;
    const int o0 = mine ? __ldg(g.dptr + v) : 0, n = mine ? __ldg(g.dptr + v + 1) - o0 : 0;
    const short2* seg = reinterpret_cast<const short2*>(g.off16) + o0;
    for (int i = gt; i < n; i += g.tg) {
      const short2 s = __ldg(seg + i);
      segP[i] = s;
      segA[i] = (uint32_t)(s.y * S + ((s.x + g.r32) >> 5)) << 5 | (uint32_t)(s.x & 31);
      if (MANY) segB[i] = (uint32_t)((g.ry - s.y) * S + ((g.r32 - s.x) >> 5)) << 5 | (uint32_t)(-s.x & 31);
    }
    if (gt == 0) {
      s_any[gi] = 0;
      s_n[gi] = n;
      if (mine) {
        s_vec[gi] = __ldg(reinterpret_cast<const short2*>(g.vec16) + v);
        if (part) {
          s_dd[gi][0] = g.target[v] - (float)g.counts[v] * g.inv_norm;
          s_dd[gi][1] = g.target[g.n_full + v] - (float)g.counts[g.n_full + v] * g.inv_norm;
        }
      }
    }
    __syncthreads();  // (also: the packed rows, and the last round's reads of the planes)
    if (mine) {
      for (int w0 = gt; w0 - lane < g.words; w0 += 2 * g.tg) {  // two words at a time (whole warps)
        uint32_t all1[2], all0[2], one1[2], one0[2];
        const uint32_t* p[2];
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int w = w0 + h * g.tg;
          const bool on = w < g.words;
          const int j = on ? fast_div(w, g.inv_H) : 0, y = on ? w - j * H : 0;
          const int rem = W - 32 * j;
          uint32_t m = on ? (rem >= 32 ? 0xffffffffu : (1u << rem) - 1u) : 0u;
          if (g.sel) m &= __ldg(g.sel + y + H * j);
          all1[h] = all0[h] = m;
          one1[h] = one0[h] = 0u;
          p[h] = s_img + y * S + j;
        }
        int i = 0;
        bool live = true;
        for (; live && i + 8 <= n; i += 8) {  // eight pixels, their loads together, then one vote
          const uint4 s0 = *reinterpret_cast<const uint4*>(segA + i), s1 = *reinterpret_cast<const uint4*>(segA + i + 4);
          const uint32_t e[8] = {s0.x, s0.y, s0.z, s0.w, s1.x, s1.y, s1.z, s1.w};
          uint32_t any = 0;
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            uint32_t c[8];
#pragma unroll
            for (int t = 0; t < 8; ++t) {
              const uint32_t* q = p[h] + (e[t] >> 5);
              c[t] = __funnelshift_r(q[0], q[1], e[t]);
            }
#pragma unroll
            for (int t = 0; t < 8; ++t) walk_masks(c[t], all1[h], all0[h], one1[h], one0[h]);
            any |= all1[h] | all0[h] | one1[h] | one0[h];
          }
          live = __any_sync(0xffffffffu, any != 0);  // else nothing is left for the rest of the segment
        }
        for (; live && i < n; ++i) {
          const uint32_t s = segA[i];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint32_t* q = p[h] + (s >> 5);
            walk_masks(__funnelshift_r(q[0], q[1], s), all1[h], all0[h], one1[h], one0[h]);
          }
        }
        uint32_t any = 0;
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int w = w0 + h * g.tg;
          if (w >= g.words) continue;
          const uint32_t u = all1[h] | all0[h];
          base[w] = u;
          base[g.words + w] = one1[h];
          base[2 * g.words + w] = one0[h];
          any |= u | one1[h] | one0[h];
        }
        if (any) s_any[gi] = 1;
      }
    }
    __syncthreads();
    if (MANY) {
      // ---- the planes with their periodic halo
      if (mine && s_any[gi])
        for (int e = gt; e < (H + g.ry) * S; e += g.tg) {
          const int r = fast_div(e, g.inv_S), k = e - r * S;
          const int y = r >= g.ry ? r - g.ry : r - g.ry + H;
          ext[e] = plane_columns(base, g.words, y, s_col[k], H, W, g.nw);
        }
      __syncthreads();
      // ---- sums along the segment for every pixel, into byte tables (over the planes without halo)
      if (mine && s_any[gi])
        for (int w = gt; w < g.words; w += g.tg) {
          const int j = fast_div(w, g.inv_H), y = w - j * H;
          const uint32_t chi = s_img[y * S + j + (g.r32 >> 5)];
          const uint4* p = ext + y * S + j;
          BitCounter cu, cn;
#pragma unroll
          for (int q = 0; q < 8; ++q) cu.c[q] = cn.c[q] = 0u;
          int i = 0;
          for (; i + 8 <= n; i += 8) add_pixels<true>(cu, cn, p, segB + i, chi, 8);
          if (i < n) add_pixels<false>(cu, cn, p, segB + i, chi, n - i);
          to_bytes(cu);
          to_bytes(cn);
          uint4* tu = reinterpret_cast<uint4*>(base + 8 * w);
          uint4* tn = reinterpret_cast<uint4*>(base + 8 * g.words + 8 * w);
          tu[0] = make_uint4(cu.c[0], cu.c[1], cu.c[2], cu.c[3]);
          tu[1] = make_uint4(cu.c[4], cu.c[5], cu.c[6], cu.c[7]);
          tn[0] = make_uint4(cn.c[0], cn.c[1], cn.c[2], cn.c[3]);
          tn[1] = make_uint4(cn.c[4], cn.c[5], cn.c[6], cn.c[7]);
        }
      __syncthreads();
    }
    // ---- the candidates, vector by vector
    for (int q = 0; q < g.G && vb + q < v1; ++q) {
      const int vq = vb + q;
      const bool any = s_any[q] != 0;
      if (!any && !dcounts) continue;
      const uint32_t* pl = s_groups + q * group_words;
      const int nq = s_n[q];
      const short2* sq = reinterpret_cast<const short2*>(pl + group_words - g.nmax);
      const short2 dv = s_vec[q];
      const float dd0 = part ? s_dd[q][0] : 0.0f, dd1 = part ? s_dd[q][1] : 0.0f;
      if (MANY) {
        const uint8_t* tu = reinterpret_cast<const uint8_t*>(pl);
        const uint8_t* tn = tu + 32 * g.words;
        const uint4* pext = reinterpret_cast<const uint4*>(pl + plane_words);
        uint2 next[kU];  // the next round's candidates, loaded a round ahead
        auto fetch = [&](int k0) {
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const int k = k0 + lane + u * nthr;
            next[u] = k < k_hi ? __ldg(cand.table + k) : make_uint2(0u, 0u);
          }
        };
        if (any) fetch(k_lo + warp * 32);
        for (int k0 = k_lo + warp * 32; k0 < k_hi; k0 += kU * nthr) {
          int d0[kU], d1[kU];
#pragma unroll
          for (int u = 0; u < kU; ++u) d0[u] = d1[u] = 0;
          if (any) {
            uint2 pix[kU];
            uint32_t hit = 0;  // bit u: pix[u] is loaded
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              const uint2 t = next[u];
              pix[u] = make_uint2(0u, 0u);
              if (t.x != t.y) {
                const int na = tn[t.x], nb = tn[t.y];
                d0[u] = na - (int)tu[t.y];
                d1[u] = nb - (int)tu[t.x];
                if (na | nb) {
                  pix[u] = __ldg(cand.pixel + k0 + lane + u * nthr);
                  hit |= 1u << u;
                }
              }
            }
            fetch(k0 + kU * nthr);
#pragma unroll
            for (int u = 0; u < kU; ++u) {
              const bool share = (hit >> u & 1u) &&
                                 swap_maybe_both(dv.x, dv.y, (int)(pix[u].y & 0xffff) - (int)(pix[u].x & 0xffff),
                                                 (int)(pix[u].y >> 16) - (int)(pix[u].x >> 16), H, W);
              // translations through both pixels (a warp per such candidate, lanes over the segment)
              for (unsigned m = __ballot_sync(0xffffffffu, share); m; m &= m - 1) {
                const int src = __ffs(m) - 1;
                const uint32_t A = __shfl_sync(0xffffffffu, pix[u].x, src), B = __shfl_sync(0xffffffffu, pix[u].y, src);
                const int px = A & 0xffff, py = A >> 16, qx = B & 0xffff, qy = B >> 16;
                int both = 0;  // phase 0 | phase 1 << 16
                for (int i = lane; i < nq; i += 32) {
                  const short2 s = sq[i];
                  int x, y;
                  swap_start(px, py, s, H, W, x, y);
                  if ((pext[(y + g.ry) * S + ((x + g.r32) >> 5)].y >> (x & 31)) & 1u)
                    both += swap_on_segment(sq, dv.x, dv.y, x, y, qx, qy, H, W);
                  swap_start(qx, qy, s, H, W, x, y);
                  if ((pext[(y + g.ry) * S + ((x + g.r32) >> 5)].z >> (x & 31)) & 1u)
                    both += (int)swap_on_segment(sq, dv.x, dv.y, x, y, px, py, H, W) << 16;
                }
                both = __reduce_add_sync(0xffffffffu, both);
                if (lane == src) {
                  d0[u] -= both & 0xffff;
                  d1[u] -= both >> 16;
                }
              }
            }
          }
          float acc[kU];
#pragma unroll
          for (int u = 0; u < kU; ++u) {
            const int k = k0 + lane + u * nthr;
            acc[u] = part && (d0[u] | d1[u]) ? part[k] : 0.0f;
            if (dcounts && k < k_hi) {
              int32_t* dk = dcounts + (int64_t)k * 2 * g.n_canon + vq;
              dk[0] = d0[u];
              dk[g.n_canon] = d1[u];
            }
          }
#pragma unroll
          for (int u = 0; u < kU; ++u)
            if (part && (d0[u] | d1[u])) part[k0 + lane + u * nthr] = swap_add_error(acc[u], d0[u], d1[u], dd0, dd1, g);
        }
      } else {
        for (int k = k_lo + warp; k < k_hi; k += nwarps) {
          int d0 = 0, d1 = 0;
          const uint2 c = __ldg(cand.pixel + k);
          if (any && c.x != c.y) {
            const int ax = c.x & 0xffff, ay = c.x >> 16, bx = c.y & 0xffff, by = c.y >> 16;
            int e0 = 0, e1 = 0;
            for (int i = lane; i < nq; i += 32) {
              const short2 s = sq[i];
              int x, y;
              swap_start(ax, ay, s, H, W, x, y);
              int at = y + H * (x >> 5);
              e1 -= (int)((pl[at] >> (x & 31)) & 1u);
              if ((pl[g.words + at] >> (x & 31)) & 1u) e0 += !swap_on_segment(sq, dv.x, dv.y, x, y, bx, by, H, W);
              swap_start(bx, by, s, H, W, x, y);
              at = y + H * (x >> 5);
              e0 -= (int)((pl[at] >> (x & 31)) & 1u);
              if ((pl[2 * g.words + at] >> (x & 31)) & 1u) e1 += !swap_on_segment(sq, dv.x, dv.y, x, y, ax, ay, H, W);
            }
            d0 = __reduce_add_sync(0xffffffffu, e0);
            d1 = __reduce_add_sync(0xffffffffu, e1);
          }
          if (lane == 0) {
            if (dcounts) {
              int32_t* dk = dcounts + (int64_t)k * 2 * g.n_canon + vq;
              dk[0] = d0;
              dk[g.n_canon] = d1;
            }
            if (part && (d0 | d1)) part[k] = swap_add_error(part[k], d0, d1, dd0, dd1, g);
          }
        }
      }
    }
    __syncthreads();  // every read of the planes and segments is done
  }
}

// ---------------------------------------------------------------------------
// Host side

static int swap_threads_per_vector(int words) {
  return std::min(kSwapThreads, std::max(32, ((words + 1) / 2 + 31) / 32 * 32));
}

// Chunks hold equally many pixels, but long segments leave the walk early and
// mostly have nothing for the candidates: whole chunks kept the SMs busy for
// 64 % of the time (the short vectors' chunks ran on alone), and small windows
// have fewer chunks than the SMs take blocks.  Parts in 1, 2, 4, 8, 16: 743,
// 527, 496, 481, 476 us (4096 candidates, 128x128, window 64) and 104, 72, 66,
// 76, 105 us (64 candidates, 50x50, full domain; four vectors side by side),
// the sums over the parts 6, 4, 7, 11, 25 us of the first; so four, but a part
// has vectors for all groups of its block.
int swap_planes_split(const DeltaArgs& d) {
  const int groups = kSwapThreads / swap_threads_per_vector(d.H * ((d.W + 31) / 32));
  return (int)std::max<int64_t>(1, std::min<int64_t>(4, d.n_canon / std::max(1, d.n_chunks) / groups));
}

// The kernel's arguments for this cell and window, but for the candidates' part.
static SwapArgs swap_args(const DeltaArgs& d, int split) {
  SwapArgs g{};
  g.H = d.H;
  g.W = d.W;
  g.rx = d.rx;
  g.ry = d.ry;
  g.split = split;
  g.nw = (d.W + 31) / 32;
  g.r32 = ((d.rx + 31) / 32) * 32;
  g.S = (g.nw + ((g.r32 + d.rx) >> 5) + 1) | 1;  // odd: 32 rows in 32 banks
  g.words = g.H * g.nw;
  g.nmax = (std::max(d.rx, d.ry) + 1 + 7) & ~7;
  g.inv_H = g.H > 1 ? (uint32_t)(((uint64_t(1) << 32) + g.H - 1) / g.H) : 0u;
  g.inv_S = g.S > 1 ? (uint32_t)(((uint64_t(1) << 32) + g.S - 1) / g.S) : 0u;
  g.dptr = d.dptr;
  g.off16 = d.off16;
  g.vec16 = d.vec16;
  g.chunk = d.chunk;
  g.n_canon = d.n_canon;
  g.n_full = d.n_full;
  g.target = d.target ? d.target + d.base : nullptr;
  g.counts = d.counts ? d.counts + d.base : nullptr;
  g.phase_mask = d.phase_mask;
  g.inv_norm = d.inv_norm;
  // threads per vector: two words each, so that what a pixel step reads of
  // the segment serves two words; vectors side by side fill small blocks
  g.tg = swap_threads_per_vector(g.words);
  g.G = kSwapThreads / g.tg;
  return g;
}

// Segments of up to 255 pixels, of cells whose packed rows and one vector's
// planes fit in shared memory.  Nearly all cells whose extended copy (a byte
// per pixel) fits do: 32 columns take 16 bytes here.  But high cells of little
// more than 32 columns pad them to two words (6000 rows of 33, window 1x1: 264
// KB against 216 KB of the extended copy).
bool swap_planes_apply(const DeltaArgs& d) {
  if (std::max(d.rx, d.ry) + 1 > kSwapMaxPixels) return false;
  SwapArgs g = swap_args(d, 1);
  g.G = 1;
  return swap_smem(g, false) <= (size_t)delta_max_smem();
}

int swap_planes_run(const uint8_t* img_dev, lpf_paths* paths, const int32_t* pairs_dev, int K, int32_t* dcounts_dev,
                    float* partial_dev, const DeltaArgs& d, int split, bool first, cudaStream_t s) {
  SwapArgs g = swap_args(d, split);
  const int max_smem = delta_max_smem();
  // Sums for every pixel cost the same for 1 and 256 candidates, lookups a
  // warp's pass over the segment for each.  Lookups against sums in us:
  // 64x64, window 32: 35, 45, 65 against 38 (16, 32, 64 candidates); 123x69,
  // 17x30: 39, 57, 85 against 52; 128x128, 64: 223, 327, 541 against 354 (64,
  // 128, 256); 250x200, 40: 198, 280 against 453 (128, 256).  Equal near
  // H W / 250 while a block has fewer than two words per thread, near H W / 96
  // beyond (the tables then leave room for three blocks on an SM or fewer).
  bool many = (int64_t)K * (g.words < 2 * kSwapThreads ? 256 : 96) > (int64_t)g.H * g.W;
  if (many) {
    SwapArgs one = g;
    one.G = 1;
    if (swap_smem(one, true) > (size_t)max_smem) many = false;  // the tables of a large cell do not fit
  }
  while (g.G > 1 && swap_smem(g, many) > (size_t)max_smem / 3) --g.G;
  const size_t smem = swap_smem(g, many);  // (at most max_smem: swap_planes_apply)
  const size_t img_words = (size_t)swap_img_words(g.H, g.ry, g.S), sel_words = d.sel_ext ? (size_t)g.words : 0;
  const size_t at_cand = (img_words + sel_words + 3) & ~size_t(3), need = at_cand + 4 * (size_t)K;
  // A larger area replaces the one there is, which is kept until the handle
  // goes: graphs that recorded calls with count changes alone still use it, as
  // they could while that area did not depend on K (areas at least double: the
  // old ones together are smaller than the one in use).
  if (need > paths->swap_cap) {
    const size_t cap = std::max(need, 2 * paths->swap_cap);
    uint32_t* area = nullptr;
    if (cudaError_t e = cudaMalloc(&area, cap * 4)) return set_cuda_error(e);
    if (paths->d_swap) paths->swap_old.push_back(paths->d_swap);
    paths->d_swap = area;
    paths->swap_cap = cap;
  }
  uint32_t* sel = sel_words ? paths->d_swap + img_words : nullptr;
  SwapCands cand;
  cand.table = reinterpret_cast<uint2*>(paths->d_swap + at_cand);
  cand.pixel = cand.table + K;
  g.img = paths->d_swap;
  g.sel = sel;
  const int n = (int)std::max<int64_t>({(int64_t)img_words, (int64_t)sel_words, (int64_t)K});
  swap_prep_kernel<<<std::min((n + 127) / 128, 4096), 128, 0, s>>>(img_dev, g, paths->d_swap, d.sel_ext, d.We, sel,
                                                                   pairs_dev, K, cand, paths->d_status,
                                                                   paths->checked);
  if (paths->ev_start && first) cudaEventRecord(paths->ev_start, s);
  // small windows have few parts: shares of the candidates (at least one per
  // warp, or a block's threads' worth) fill the SMs' three blocks, each share
  // with its own walk (79x101, window 25x19, 28 candidates: 162 us without)
  const int share = many ? kSwapThreads : kSwapWarps, parts = d.n_chunks * split;
  const dim3 grid(parts, std::max(1, std::min(3 * delta_num_sms() / parts, (K + share - 1) / share)));
  // several candidates at a time hide the latency of their loads (4096 of
  // them: 929 us one by one, 815 by two, 746 by four, 817 by eight, before the
  // parts), but cost where a thread has one at most (64: 110, 119, 123, 174)
  const bool several = (K + (int)grid.y - 1) / (int)grid.y > g.G * g.tg;
  auto kernel = !many ? swap_kernel<0> : several ? swap_kernel<kSwapUnroll> : swap_kernel<1>;
  kernel<<<grid, g.G * g.tg, smem, s>>>(g, cand, K, dcounts_dev, partial_dev);
  if (paths->ev_stop) cudaEventRecord(paths->ev_stop, s);
  return LPF_OK;
}

int swap_planes_attributes(int optin, int* max_static) {
  cudaFuncAttributes fa;
  for (const void* fn : {(const void*)swap_kernel<0>, (const void*)swap_kernel<1>, (const void*)swap_kernel<kSwapUnroll>}) {
    cudaError_t e = cudaFuncGetAttributes(&fa, fn);
    if (e == cudaSuccess)
      e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
    if (e != cudaSuccess) return set_cuda_error(e);
    *max_static = std::max(*max_static, (int)fa.sharedSizeBytes);
  }
  return LPF_OK;
}

}  // namespace lpf
