// Minima of d^2 + f along staged lines, by bracketed arguments.
//
// For one line f(0 .. n-1) every output i needs min over j of f(j) + (i - j)^2 (the separable exact
// transform).  The argument of that minimum is monotone in i: for p < q with arguments a(p), a(q) (any
// of several equal ones), every output between p and q takes its minimum over the positions between
// a(p) and a(q) -- a position j below both loses to the lower of the two by an amount that only grows
// with i, and likewise above.  This holds for any values f, so saturated or missing inputs need no case
// of their own.  So:
//   1. line_argmin finds the argument at a position by searching the staged bricks outward from it: a
//      brick is read only when its minimum plus the squared gap to it is below the best so far, and the
//      search ends when the squared gap plus the line's minimum is not.  It runs at every eighth brick
//      boundary over the whole line, then at the boundaries between two of those over the bricks
//      between their arguments only (nine per boundary on average, whatever the distances);
//   2. line_outputs evaluates a brick's eight outputs over the positions between its two boundaries'
//      arguments -- nine on average over a line, since the brackets tile it.
// Against an envelope stack per line (one dependent load per pop, from global or local memory) the
// reads are independent and in shared memory, a lane per line with consecutive lanes on consecutive
// words, and all of a line's bricks are worked on at once by different warps.
#pragma once

#include <stdint.h>

namespace vdbedt {

// Brick minima of one line: eight staged positions to one word.  T: the staged type (16-bit or 32-bit
// unsigned compare: missing inputs are the largest value), STRIDE: elements between positions.
template <typename T, int STRIDE>
__device__ __forceinline__ uint32_t line_brick_min(const T* __restrict__ v) {
  uint32_t r = (uint32_t)v[0];
#pragma unroll
  for (int j = 1; j < 8; ++j) r = min(r, (uint32_t)v[j * STRIDE]);
  return r;
}

// The least f(j) + (p - j)^2 over the positions of bricks lo .. hi of the line v (brick minima m; least:
// a bound below every value of those bricks), and its position.  On entry best is that sum for some
// position a, kept in arg (~0u: none).  Searched from p outward; lanes of a warp may pass different
// arguments, and a lane with best = 0 searches nothing.
template <typename T, int STRIDE>
__device__ __forceinline__ void line_argmin(const T* __restrict__ v, const T* __restrict__ m, uint32_t least, int p, int lo,
                                            int hi, uint32_t& best, int& arg) {
  const int kb = p >> 3, pm = p & 7;
  int abrick = -1;  // the brick that improved best last
  auto eval = [&](int b) {
    const T* c = v + b * 8 * STRIDE;
    uint32_t r = best;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int d = 8 * b + j - p;
      r = min(r, (uint32_t)c[j * STRIDE] + (uint32_t)(d * d));
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
    if (right && (uint32_t)m[r * STRIDE] + gr2 < best) eval(r);
    if (left && (uint32_t)m[l * STRIDE] + gl2 < best) eval(l);
  }
  if (abrick >= 0) {
    const T* c = v + abrick * 8 * STRIDE;
    int a = arg;
#pragma unroll
    for (int j = 7; j >= 0; --j) {
      const int d = 8 * abrick + j - p;
      if ((uint32_t)c[j * STRIDE] + (uint32_t)(d * d) == best) a = 8 * abrick + j;
    }
    arg = a;
  }
}

// The eight outputs x0 .. x0 + 7 over the positions lo .. hi (hi < lo: none, every output ~0u - 64 or
// more).  (s + k)^2 = s^2 + 2 s k + k^2 with s = x0 - j: one multiply-add and half a three-way minimum
// per candidate and output; the sums carry a bias of 64 so that they stay non-negative without k^2.
template <typename T, int STRIDE>
__device__ __forceinline__ void line_outputs(const T* __restrict__ v, int x0, int lo, int hi, uint32_t (&out)[8]) {
  uint32_t acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) acc[k] = ~0u;
  for (int j = lo; j <= hi; j += 2) {
    const int j2 = min(j + 1, hi);
    const int s = x0 - j, s2 = x0 - j2;
    const uint32_t a = (uint32_t)v[j * STRIDE] + (uint32_t)(s * s + 64);
    const uint32_t b = (uint32_t)v[j2 * STRIDE] + (uint32_t)(s2 * s2 + 64);
    const uint32_t w = (uint32_t)(2 * s), w2 = (uint32_t)(2 * s2);
#pragma unroll
    for (int k = 0; k < 8; ++k) acc[k] = __vimin3_u32(acc[k], a + w * k, b + w2 * k);
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) out[k] = acc[k] + (uint32_t)(k * k - 64);
}

}  // namespace vdbedt
