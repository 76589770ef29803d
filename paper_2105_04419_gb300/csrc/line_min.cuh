// Minima of d^2 + f along staged lines: for one line f(0 .. n-1), every output i needs min over j of
// f(j) + (i - j)^2 (the separable exact transform).  The lines are staged in shared memory, a word per lane
// and position (one line's 32-bit value, or two neighbouring lines' 16-bit values), positions 32 words
// apart, with the minimum of every brick (eight positions) and of every eight bricks; a warp takes a brick
// of eight outputs at a time.  Against an envelope stack per line (one dependent load per pop, from global
// or local memory) the reads are independent and conflict-free, and all of a line's bricks are worked on at
// once by different warps.  Two forms:
//
// Walk (16-bit, bounded distances): evaluate the output brick's own positions, then go outward brick by
// brick on both sides; a brick is evaluated only when, on some line, its minimum plus the squared gap is
// below the outputs' current maximum, and the walk ends when the line's minimum plus it is not.  64
// candidates a lane for eight loads and 15 squares, uniform over the warp.  No bookkeeping, but 4.4 bricks
// per output brick in a tunnel scene, and more the farther the obstacles are.
//
// Brackets (32-bit, any distance): the argument of the minimum is monotone in i.  For p < q with arguments
// a(p), a(q) (any of several equal ones), every output between p and q takes its minimum over the positions
// between a(p) and a(q) -- a position j below both loses to the lower of the two by an amount that only
// grows with i, and likewise above; this holds for any values f, so missing inputs need no case of their
// own.  line_argmin finds the argument at a position by searching the staged bricks outward from it: a
// brick is read only when its minimum plus the squared gap to it is below the best so far, and the
// search ends when the squared gap plus the line's minimum is not.  It runs at every eighth brick
// boundary over the whole line, then at the boundaries between two of those over the bricks
// between their arguments only (nine per boundary on average, whatever the distances).  line_outputs
// evaluates a brick's eight outputs over the positions between its two boundaries' arguments -- eight on
// average over a line, since the brackets tile it; the widest of 32 lanes has 13.  (Measured no better:
// arguments kept as bricks, with whole bricks evaluated between them; the searches made uniform over the
// warp and each started from the previous boundary's argument; the walk, 1.3 to 2.5 times slower on far
// distances.)
#pragma once

#include <stdint.h>

namespace vdbedt {

constexpr int kLineStride = 32;               // words between positions (and between bricks' minima)
constexpr int kBrickWords = 8 * kLineStride;  // words of a staged brick

// ---- two 16-bit lines to a word ----
// squares, saturated above every dmax^2 (181^2 = 32,761) and low enough that a sum with one fits 16 bits: an
// offset whose square is saturated costs more than dmax^2 either way, so no minimum depends on it
__device__ __forceinline__ uint32_t line16_square(int u) { return (uint32_t)min(u * u, 65535 - 181 * 181) * 0x10001u; }

// a + b below c in either half
__device__ __forceinline__ bool line16_below(uint32_t a, uint32_t b, uint32_t c) { return __viaddmin_u16x2(a, b, c) != c; }

// Minimum of a brick's positions.
__device__ __forceinline__ uint32_t line16_min8(const uint32_t* __restrict__ v) {
  const uint32_t a = __vimin3_u16x2(v[0], v[kLineStride], v[2 * kLineStride]);
  const uint32_t b = __vimin3_u16x2(v[3 * kLineStride], v[4 * kLineStride], v[5 * kLineStride]);
  return __vimin3_u16x2(__vminu2(a, b), v[6 * kLineStride], v[7 * kLineStride]);
}

// The eight outputs of brick B of the lines v (nb bricks; m: brick minima, m8: minima over eight bricks,
// least: over the line).  sq[u]: the squares of u, -8 nb <= u < 8 nb + 16, rows of 16 words at multiples of
// 8 being 16-byte aligned.  Lanes without `some` need nothing.
__device__ __forceinline__ void line16_outputs(const uint32_t* __restrict__ v, const uint32_t* __restrict__ m,
                                               const uint32_t* __restrict__ m8, const uint32_t* __restrict__ sq,
                                               uint32_t least, int nb, int B, bool some, uint32_t (&acc)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = ~0u;
  uint32_t mxa, mxb;  // maxima of outputs 0 .. 3 and 4 .. 7; 0 where nothing is needed
  auto eval = [&](int b) {
    const uint32_t* c = v + b * kBrickWords;
    uint32_t s[16];  // squares of 8 (B - b) - 8 .. 8 (B - b) + 7
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint4 w = *reinterpret_cast<const uint4*>(sq + 8 * (B - b) - 8 + 4 * q);
      s[4 * q] = w.x;
      s[4 * q + 1] = w.y;
      s[4 * q + 2] = w.z;
      s[4 * q + 3] = w.w;
    }
    // a plain add sums both halves (no carry between them)
#pragma unroll
    for (int j = 0; j < 8; j += 2) {
      const uint32_t f = c[j * kLineStride], h = c[(j + 1) * kLineStride];
#pragma unroll
      for (int k = 0; k < 8; ++k) acc[k] = __vimin3_u16x2(acc[k], f + s[8 + k - j], h + s[7 + k - j]);
    }
    mxa = some ? __vimax3_u16x2(__vmaxu2(acc[0], acc[1]), acc[2], acc[3]) : 0u;
    mxb = some ? __vimax3_u16x2(__vmaxu2(acc[4], acc[5]), acc[6], acc[7]) : 0u;
  };
  eval(B);
  for (int t = 1;;) {
    const int r = B + t, l = B - t;
    const bool in_r = r < nb, in_l = l >= 0;
    if (!in_r && !in_l) break;
    // gaps of the brick's nearest position to the outputs on its side and to the other four
    const uint32_t g1 = sq[8 * t - 7], g2 = sq[8 * t - 3];
    if (t >= 8) {  // eight bricks at a time: both aligned groups that they touch on either side
      const uint32_t mx = __vmaxu2(mxa, mxb);
      const int r0 = min(r, nb - 1) >> 3, r1 = min(r + 7, nb - 1) >> 3, l0 = max(l, 0) >> 3, l1 = max(l - 7, 0) >> 3;
      const uint32_t mr = __vminu2(m8[r0 * kLineStride], m8[r1 * kLineStride]);
      const uint32_t ml = __vminu2(m8[l0 * kLineStride], m8[l1 * kLineStride]);
      if (!__any_sync(0xffffffffu, (in_r && line16_below(mr, g1, mx)) || (in_l && line16_below(ml, g1, mx)))) {
        if (!__any_sync(0xffffffffu, line16_below(least, g1, mx))) break;
        t += 8;
        continue;
      }
    }
    const uint32_t br = in_r ? m[r * kLineStride] : 0u, bl = in_l ? m[l * kLineStride] : 0u;
    const bool nr = __any_sync(0xffffffffu, in_r && (line16_below(br, g1, mxb) || line16_below(br, g2, mxa)));
    const bool nl = __any_sync(0xffffffffu, in_l && (line16_below(bl, g1, mxa) || line16_below(bl, g2, mxb)));
    if (nr) eval(r);
    if (nl) eval(l);
    if (!nr && !nl && !__any_sync(0xffffffffu, line16_below(least, g1, __vmaxu2(mxa, mxb)))) break;
    ++t;
  }
}

// ---- one 32-bit line to a word ----
// Minimum of a brick's positions.
__device__ __forceinline__ uint32_t line_brick_min(const uint32_t* __restrict__ v) {
  uint32_t r = v[0];
#pragma unroll
  for (int j = 1; j < 8; ++j) r = min(r, v[j * kLineStride]);
  return r;
}

// The least f(j) + (p - j)^2 over the positions of bricks lo .. hi of the line v (brick minima m; least:
// a bound below every value of those bricks), and its position.  On entry best is that sum for some
// position a, kept in arg (~0u: none).  Searched from p outward; lanes of a warp may pass different
// arguments, and a lane with best = 0 searches nothing.
__device__ __forceinline__ void line_argmin(const uint32_t* __restrict__ v, const uint32_t* __restrict__ m, uint32_t least, int p, int lo,
                                            int hi, uint32_t& best, int& arg) {
  const int kb = p >> 3, pm = p & 7;
  int abrick = -1;  // the brick that improved best last
  auto eval = [&](int b) {
    const uint32_t* c = v + b * 8 * kLineStride;
    uint32_t r = best;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int d = 8 * b + j - p;
      r = min(r, c[j * kLineStride] + (uint32_t)(d * d));
    }
    if (r < best) {
      best = r;
      abrick = b;
    }
  };
  // t bricks away on the right, then on the left; gaps from p to the brick's nearest position
  for (int t = max(0, max(lo - kb, kb - hi));; ++t) {
    const int r = kb + t, l = kb - t;
    const int gr = t ? 8 * t - pm : 0, gl = 8 * t - 7 + pm;
    const uint32_t gr2 = (uint32_t)(gr * gr), gl2 = (uint32_t)(gl * gl);
    const bool right = r <= hi && least + gr2 < best, left = t > 0 && l >= lo && least + gl2 < best;
    if (!right && !left) break;
    if (right && m[r * kLineStride] + gr2 < best) eval(r);
    if (left && m[l * kLineStride] + gl2 < best) eval(l);
  }
  if (abrick >= 0) {
    const uint32_t* c = v + abrick * 8 * kLineStride;
    int a = arg;
#pragma unroll
    for (int j = 7; j >= 0; --j) {
      const int d = 8 * abrick + j - p;
      if (c[j * kLineStride] + (uint32_t)(d * d) == best) a = 8 * abrick + j;
    }
    arg = a;
  }
}

// Two candidates, positions j and j2, into the eight outputs from x0 on: (s + k)^2 = s^2 + 2 s k + k^2 with
// s = x0 - j takes one multiply-add and half a three-way minimum per candidate and output; the sums carry
// a bias of 64 so that they stay non-negative without k^2.
__device__ __forceinline__ void line_take2(const uint32_t* __restrict__ v, int x0, int j, int j2, uint32_t (&acc)[8]) {
  const int s = x0 - j, s2 = x0 - j2;
  const uint32_t a = v[j * kLineStride] + (uint32_t)(s * s + 64);
  const uint32_t b = v[j2 * kLineStride] + (uint32_t)(s2 * s2 + 64);
  const uint32_t w = (uint32_t)(2 * s), w2 = (uint32_t)(2 * s2);
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = __vimin3_u32(acc[k], a + w * k, b + w2 * k);
}

// The eight outputs x0 .. x0 + 7 over the positions lo .. hi (hi < lo: none, every output ~0u - 64 or more).
// Where some lane's bracket is long (two obstacles far apart with a change of the nearest between them), its
// two ends come first and a brick between them is evaluated only when its minimum plus the squared gap is
// below the outputs' maximum.
__device__ __forceinline__ void line_outputs(const uint32_t* __restrict__ v, const uint32_t* __restrict__ m, int x0, int lo,
                                             int hi, uint32_t (&out)[8]) {
  uint32_t acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = ~0u;
  if (!__any_sync(__activemask(), hi - lo > 24)) {
    for (int j = lo; j <= hi; j += 2) line_take2(v, x0, j, min(j + 1, hi), acc);
  } else if (lo <= hi) {
    line_take2(v, x0, lo, hi, acc);
    for (int b = lo >> 3; b <= hi >> 3; ++b) {
      const int x = b - (x0 >> 3), gap = x == 0 ? 0 : 8 * abs(x) - 7;
      uint32_t mx = 0u;  // of the outputs themselves: acc carries 64 - k^2
#pragma unroll
      for (int k = 0; k < 8; ++k) mx = max(mx, acc[k] + (uint32_t)(k * k));
      if (m[b * kLineStride] + (uint32_t)(gap * gap + 64) < mx) {
#pragma unroll
        for (int j = 0; j < 8; j += 2) line_take2(v, x0, 8 * b + j, 8 * b + j + 1, acc);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) out[k] = acc[k] + (uint32_t)(k * k - 64);
}

}  // namespace vdbedt
