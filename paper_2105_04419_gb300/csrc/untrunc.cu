// Untruncated transform (VDBEDT_FLAG_UNTRUNCATED): Eq. 1 without the truncation, i.e. the exact
// squared distance to the nearest occupied voxel anywhere in a bounded grid (the paper's
// dmax = infinity runs, Table II).  With no truncation every voxel is in reach of every obstacle,
// so every brick is stored, brick (bx, by, bz) at slot bx + BX (by + BY bz), and the transform runs
// over whole lines of the grid, one axis after the other (Eq. 1's minimum taken per axis):
//   x: per row, the distance to the nearest occupied voxel on either side, g1 = dx^2 (k_ut_x);
//   y, z: per line, the minimum over i of f(i) + (t - i)^2 (f: g1, then g2).  Lines of up to kLineMax
//      positions are staged whole in shared memory (k_ut_line, by the bracketed minima of
//      line_min.cuh).  Longer ones: the lower envelope of the parabolas rooted at the line's
//      finite values, built on a stack in one sweep, read back in a second.  Two
//      parabolas are compared through their intersection with the denominators multiplied out,
//      exactly: the grid's size limit keeps every f(p) + p^2 below 2^31, so the differences are
//      int32 and each product one widening multiply (below 2^48).
// kNone marks a row, plane or grid without an obstacle.  Only voxels inside the grid are read or
// written; g1 and g2 hold int32 here (their arrays are allocated twice as large).
#include <algorithm>

#include "line_min.cuh"
#include "vdbedt_internal.cuh"

namespace vdbedt {
namespace {

constexpr int kUT = 256;

__device__ __forceinline__ int ut_slot(const GridView& g, int bx, int by, int bz) {
  return bx + g.BX * (by + g.BY * bz);
}

__device__ __forceinline__ int ut_vox(int x, int y, int z) { return (x & 7) + 8 * (y & 7) + 64 * (z & 7); }
// g1 is stored y-major, so that the y pass reads planes
__device__ __forceinline__ int ut_vox_g1(int x, int y, int z) { return (x & 7) + 8 * (z & 7) + 64 * (y & 7); }

// A line's stack in the scratch, interleaved with the other 31 lines of its group of 32 (entry m
// of line t at ((t >> 5) n + m) 32 + (t & 31)): lanes of a warp that push or pop at similar depths
// touch the same 32-byte sectors instead of 32 separate regions.
struct LineStack {
  int2* p;
  __device__ __forceinline__ LineStack(int2* stack, int64_t t, int n)
      : p(stack + (size_t)(t >> 5) * 32 * n + (size_t)(t & 31)) {}
  __device__ __forceinline__ int2& operator[](int m) const { return p[(size_t)m * 32]; }
};

unsigned ut_blocks(int64_t threads) {
  const int64_t b = (threads + kUT - 1) / kUT;
  return (unsigned)(b < 1 ? 1 : (b > 152 * 64 ? 152 * 64 : b));
}

// Interior nodes of every key of the grid (node indices in creation order).
__global__ void k_ut_nodes(GridView g) {
  const int64_t nk = (int64_t)g.NX * g.NY * g.NZ;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < nk; k += (int64_t)gridDim.x * blockDim.x)
    get_or_create_node(g, (unsigned long long)k);
}

// Every brick of the grid at its fixed slot, with an empty occupancy.
__global__ void k_ut_bricks(GridView g) {
  const int64_t nb = (int64_t)g.BX * g.BY * g.BZ;
  if (blockIdx.x == 0 && threadIdx.x == 0) g.counters[C_NBRICKS] = (int)nb;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += (int64_t)gridDim.x * blockDim.x) {
    const int bx = (int)(b % g.BX), r = (int)(b / g.BX), by = r % g.BY, bz = r / g.BY;
    const int node = find_node(g, node_key_of(g, bx, by, bz));
    if (node < 0) {
      set_error(g, kErrInternal);
      continue;
    }
    g.child[(size_t)node * kNodeBricks + local_brick(bx, by, bz)] = (int)b;
    g.bcoord[b] = make_int4(bx, by, bz, node);
    g.bflags[b] = 0u;
    g.bepoch[b] = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) g.occ[(size_t)b * 8 + q] = 0ull;
  }
}

// Empty occupancy, flags and brick epochs; the counters start over except the stored bricks and
// nodes.
__global__ void k_ut_reset(GridView g) {
  const int64_t nb = (int64_t)g.BX * g.BY * g.BZ;
  if (blockIdx.x == 0 && (int)threadIdx.x < C_NUM && threadIdx.x != C_NBRICKS && threadIdx.x != C_NNODES)
    g.counters[threadIdx.x] = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nb * 8; i += (int64_t)gridDim.x * blockDim.x) {
    g.occ[i] = 0ull;
    if ((i & 7) == 0) {
      g.bflags[i >> 3] = 0u;
      g.bepoch[i >> 3] = 0;  // the update epoch starts over with the counters
    }
  }
}

// Occupancy from a dense uint8 grid [nz][ny][nx] (nonzero = occupied): a thread per (brick,
// plane) assembles the plane's 64-bit word (bit x + 8 y) from eight rows of eight bytes.
__global__ void k_ut_dense(GridView g, const uint8_t* __restrict__ grid) {
  const int64_t nw = (int64_t)g.BX * g.BY * g.BZ * 8;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nw; i += (int64_t)gridDim.x * blockDim.x) {
    // i = bx + BX (pz + 8 (by + BY bz)): neighbouring threads read neighbouring 8-byte row pieces
    const int bx = (int)(i % g.BX);
    const int64_t r = i / g.BX;
    const int pz = (int)(r & 7);
    const int64_t rb = r >> 3;
    const int by = (int)(rb % g.BY), bz = (int)(rb / g.BY);
    const int z = 8 * bz + pz;
    unsigned long long w = 0ull;
    if (z < g.nz) {
      for (int py = 0; py < 8; ++py) {
        const int y = 8 * by + py;
        if (y >= g.ny) break;
        const uint8_t* row = grid + ((size_t)z * g.ny + y) * g.nx;
        for (int px = 0; px < 8; ++px) {
          const int x = 8 * bx + px;
          if (x < g.nx && row[x]) w |= 1ull << (px + 8 * py);
        }
      }
    }
    g.occ[(size_t)ut_slot(g, bx, by, bz) * 8 + pz] = w;
  }
}

// A row piece of eight words (32-byte aligned) with one 256-bit store: the lanes of a warp write to as many
// lines, and two 16-byte stores would pass them through the load-store unit twice.
__device__ __forceinline__ void store_row(void* dst, const int (&d)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(dst), "r"(d[0]), "r"(d[1]), "r"(d[2]),
               "r"(d[3]), "r"(d[4]), "r"(d[5]), "r"(d[6]), "r"(d[7])
               : "memory");
}

// x pass: a warp per (by, bz, plane z): eight x-rows at once, 32 bricks of the row per step (a lane's
// 64-bit mask word holds its brick's eight rows of the plane).  Per row one ballot gives the bricks of the
// step that hold an occupied voxel, from which a lane has the nearest ones before and after its brick by
// a count of leading and of trailing zeros; what lies outside the step comes from two carries per row: the
// last occupied voxel before it, followed as the steps advance, and the first one after it, taken from a
// sweep over the steps from the far end (kept in shared memory, eight words per step).  g1 = d^2 (kNone:
// empty row) is written once, 32 bytes per brick and row.  Bound by those writes.  512 x 512 x 256 tunnel
// scene: 0.064 ms (a thread per row walking it forward and back, with a carry per brick through memory:
// 0.097); the rows of a lidar frame 0.027 ms (0.093).
// INCR (an update): only the rows whose dirty bit is set (a byte per plane, cleared once read); each g1 is
// compared with the stored one, the row pieces that changed are written and the y-line byte (x, z) of
// every changed voxel set with a plain store.
constexpr int kUtXWarps = 8;
template <bool INCR>
__global__ void __launch_bounds__(32 * kUtXWarps) k_ut_x(GridView g) {
  extern __shared__ int32_t after_sh[];  // [kUtXWarps][steps][8]
  int32_t* __restrict__ g1 = reinterpret_cast<int32_t*>(g.g1);
  const int lane = threadIdx.x & 31, steps = (g.BX + 31) >> 5;
  int32_t* after = after_sh + (size_t)(threadIdx.x >> 5) * steps * 8;
  constexpr int kFar = 1 << 20;  // beyond every distance of a row
  const int64_t ntask = (int64_t)g.BY * g.BZ * 8, nw = (int64_t)gridDim.x * kUtXWarps;
  for (int64_t t = (int64_t)blockIdx.x * kUtXWarps + (threadIdx.x >> 5); t < ntask; t += nw) {
    const int pz = (int)(t & 7);
    const int64_t line = t >> 3;  // by + BY bz
    const int by = (int)(line % g.BY), bz = (int)(line / g.BY), z = 8 * bz + pz;
    uint32_t rows = 0xFFu >> max(0, 8 * by + 8 - g.ny);  // rows of the plane inside the grid
    if (z >= g.nz) continue;
    if (INCR) {
      uint8_t* dirty = reinterpret_cast<uint8_t*>(g.ut_bits) + t;  // bit (y & 7) + 8 (z & 7) of the line's 64
      rows = *dirty;
      if (!rows) continue;  // warp-uniform
      __syncwarp();
      if (lane == 0) {
        *dirty = 0;
        atomicAdd(&g.items_ctr[0], __popc(rows));
      }
    }
    const size_t s0 = (size_t)ut_slot(g, 0, by, bz);
    const unsigned long long* occ = g.occ + s0 * 8 + pz;
    // first occupied voxel after each step, per row (lane r < 8 keeps row r's)
    int first = kFar * 2;
    for (int k = steps - 1; k >= 0; --k) {
      if (lane < 8) after[8 * k + lane] = first;
      const int bx = 32 * k + lane;
      const unsigned long long w = bx < g.BX ? occ[(size_t)bx * 8] : 0ull;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const uint32_t byte = (uint32_t)(w >> (8 * r)) & 0xFFu;
        const unsigned m = __ballot_sync(0xffffffffu, byte != 0u);
        if (!m) continue;
        const int b = __ffs(m) - 1;
        const uint32_t fb = __shfl_sync(0xffffffffu, byte, b);
        if (lane == r) first = 8 * (32 * k + b) + __ffs(fb) - 1;
      }
    }
    __syncwarp();
    int last[8];
#pragma unroll
    for (int r = 0; r < 8; ++r) last[r] = -kFar;
    uint8_t* yflag = INCR ? reinterpret_cast<uint8_t*>(g.ut_bits + ut_row_words(g)) + (size_t)ut_nxp(g) * z : nullptr;
    for (int k = 0; k < steps; ++k) {
      const int bx = 32 * k + lane;
      const unsigned long long w = bx < g.BX ? occ[(size_t)bx * 8] : 0ull;
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const uint32_t byte = (uint32_t)(w >> (8 * r)) & 0xFFu;
        const unsigned m = __ballot_sync(0xffffffffu, byte != 0u);
        if (!((rows >> r) & 1u)) continue;  // warp-uniform
        // the nearest occupied voxels before and after this lane's brick
        const unsigned ml = m & ((1u << lane) - 1u), mr = (m >> lane) >> 1;
        const int lb = ml ? 31 - __clz(ml) : lane, rb = mr ? lane + __ffs(mr) : lane;
        const uint32_t lbyte = __shfl_sync(0xffffffffu, byte, lb), rbyte = __shfl_sync(0xffffffffu, byte, rb);
        int dl = 8 * bx - 1 - (ml ? 8 * (32 * k + lb) + 31 - __clz(lbyte) : last[r]);
        int dr = (mr ? 8 * (32 * k + rb) + __ffs(rbyte) - 1 : after[8 * k + r]) - (8 * bx + 8);
        if (m) {
          const int b = 31 - __clz(m);
          const uint32_t eb = __shfl_sync(0xffffffffu, byte, b);
          last[r] = 8 * (32 * k + b) + 31 - __clz(eb);
        }
        if (bx >= g.BX) continue;
        int d[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          dl = (byte >> i) & 1u ? 0 : dl + 1;
          d[i] = dl;
        }
#pragma unroll
        for (int i = 7; i >= 0; --i) {
          dr = (byte >> i) & 1u ? 0 : dr + 1;
          d[i] = min(d[i], dr);
          d[i] = d[i] >= kFar / 2 || 8 * bx + i >= g.nx ? kNone : d[i] * d[i];  // the last brick's padding holds kNone
        }
        int4* dst = reinterpret_cast<int4*>(g1 + (s0 + bx) * kBrickVox + ut_vox_g1(0, r, pz));
        if (INCR) {
          const int4 oa = dst[0], ob = dst[1];
          const int old[8] = {oa.x, oa.y, oa.z, oa.w, ob.x, ob.y, ob.z, ob.w};
          uint32_t ch = 0u;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (8 * bx + i < g.nx && d[i] != old[i]) ch |= 1u << i;
          if (!ch) continue;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if ((ch >> i) & 1u) yflag[8 * bx + i] = 1;  // the rows of every y write the same y lines
        }
        store_row(dst, d);
      }
    }
    __syncwarp();  // the carries are rewritten by the next task
  }
}

// Voxel i of line (x, c) along AXIS (1: y, c = z; 2: z, c = y) in a pool of bricks at fixed slots:
// base + (i >> 3) * brick stride + (i & 7) * voxel stride.  IN: of the pass's input field (planes along
// the axis), else of its output.
template <int AXIS, bool IN>
struct LineAt {
  size_t base, bstride;
  __device__ __forceinline__ LineAt(const GridView& g, int x, int c) {
    base = AXIS == 1 ? (size_t)ut_slot(g, x >> 3, 0, c >> 3) * kBrickVox + (IN ? ut_vox_g1(x, 0, c) : ut_vox(x, 0, c))
                     : (size_t)ut_slot(g, x >> 3, c >> 3, 0) * kBrickVox + ut_vox(x, c, 0);
    bstride = (size_t)kBrickVox * (AXIS == 1 ? g.BX : (size_t)g.BX * g.BY);
  }
  __device__ __forceinline__ size_t operator()(int i) const {
    return base + (size_t)(i >> 3) * bstride + (size_t)((i & 7) * (AXIS == 1 && !IN ? 8 : 64));
  }
};

// Lower envelope of the parabolas f(i) + (t - i)^2 over the line's finite values, built on the
// line's stack: entries (p, F = f(p) + p^2), the top two also in registers.  The grid's size limit
// keeps every F below 2^31, so differences of F are int32 and each intersection test compares two
// widening 32 x 32 -> 64-bit products exactly.  The inputs are loaded a brick (8 positions) at a
// time, all eight before any is used.  Returns the entry count.
template <int AXIS>
__device__ __forceinline__ int env_build(const LineStack& st, const LineAt<AXIS, true>& at, const int32_t* __restrict__ in,
                                         int n) {
  int m = 0, p0 = 0, F0 = 0, p1 = 0, F1 = 0;
  for (int i0 = 0; i0 < n; i0 += 8) {
    int fv[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) fv[j] = i0 + j < n ? in[at(i0 + j)] : kNone;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int i = i0 + j;
      if (fv[j] == kNone) continue;
      const int Fi = fv[j] + i * i;
      while (m >= 2) {
        // drop the top when the new parabola undercuts it no later than the top undercuts the one
        // below: (Fi - F1) / (i - p1) <= (F1 - F0) / (p1 - p0)
        if ((long long)(Fi - F1) * (p1 - p0) > (long long)(F1 - F0) * (i - p1)) break;
        --m;
        p1 = p0;
        F1 = F0;
        if (m >= 2) {
          const int2 e = st[m - 2];
          p0 = e.x;
          F0 = e.y;
        }
      }
      st[m] = make_int2(i, Fi);
      p0 = p1;
      F0 = F1;
      p1 = i;
      F1 = Fi;
      ++m;
    }
  }
  return m;
}

// Reading an envelope back in increasing position: the lowest parabola only moves forward.
// Entries k, k + 1 and (loaded ahead) k + 2 in registers.
struct EnvRead {
  const LineStack& st;
  int m, k;
  int2 cur, nxt, ahead;
  __device__ __forceinline__ EnvRead(const LineStack& s, int count) : st(s), m(count), k(0) {
    cur = nxt = ahead = make_int2(0, 0);
    if (m > 0) {
      cur = st[0];
      nxt = m > 1 ? st[1] : cur;
      ahead = m > 2 ? st[2] : cur;
    }
  }
  // the envelope at i (i non-decreasing between calls); kNone for an empty envelope
  __device__ __forceinline__ int at(int i) {
    if (m == 0) return kNone;
    while (k + 1 < m) {
      // the next parabola is no higher at i: F(nxt) - F(cur) <= 2 i (nxt - cur)
      if ((long long)(nxt.y - cur.y) > (long long)(2 * i) * (nxt.x - cur.x)) break;
      ++k;
      cur = nxt;
      nxt = ahead;
      if (k + 2 < m) ahead = st[k + 2];
    }
    const int d = i - cur.x;
    return (cur.y - cur.x * cur.x) + d * d;  // f(p) + (i - p)^2
  }
};

// y (AXIS 1: g1 -> g2) or z (AXIS 2: g2 -> D) pass: a thread per line, lines (x, z) or (x, y)
// with x fastest, the line's stack in `stack` (LineStack).
template <int AXIS>
__global__ void k_ut_env(GridView g, const int32_t* __restrict__ in, int32_t* __restrict__ out, int2* __restrict__ stack) {
  const int n = AXIS == 1 ? g.ny : g.nz;
  const int64_t nlines = (int64_t)g.nx * (AXIS == 1 ? g.nz : g.ny);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nlines; t += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(t % g.nx), c = (int)(t / g.nx);  // c: z (AXIS 1) or y (AXIS 2)
    const LineAt<AXIS, true> at(g, x, c);
    const LineAt<AXIS, false> to(g, x, c);
    const LineStack st(stack, t, n);
    EnvRead env(st, env_build<AXIS>(st, at, in, n));
    for (int i = 0; i < n; ++i) out[to(i)] = env.at(i);
  }
}

// The update's y (AXIS 1) or z (AXIS 2) pass over the dirty lines: lines (x, c) with x padded to
// NXP, so that a warp's 32 lanes are 32 lines along x at one c and read 32 dirty-line bytes,
// cleared once read.  Each dirty lane builds its line's envelope as k_ut_env does and reads it
// back; the y pass writes the g2 values that changed and sets the z-line byte (x, y) of each.
// The z pass writes D on its dirty lines.
template <int AXIS>
__global__ void k_ut_env_upd(GridView g, const int32_t* __restrict__ in, int32_t* __restrict__ out,
                             int2* __restrict__ stack) {
  const int n = AXIS == 1 ? g.ny : g.nz;
  const int nxp = ut_nxp(g);
  const int64_t nlines = (int64_t)nxp * (AXIS == 1 ? g.nz : g.ny);  // a multiple of 32
  uint8_t* yflag = reinterpret_cast<uint8_t*>(g.ut_bits + ut_row_words(g));
  uint8_t* zflag = reinterpret_cast<uint8_t*>(g.ut_bits + ut_row_words(g) + ut_yline_words(g));
  uint8_t* flag = AXIS == 1 ? yflag : zflag;  // this pass's dirty lines
  const int lane = threadIdx.x & 31;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nlines; t += (int64_t)gridDim.x * blockDim.x) {
    const bool f = flag[t] != 0;
    const uint32_t w = __ballot_sync(0xffffffffu, f);
    if (f) flag[t] = 0;
    if (!w) continue;  // warp-uniform
    if (lane == 0) atomicAdd(&g.items_ctr[AXIS], __popc(w));
    const bool dirty = (w >> lane) & 1u;  // set only for x < nx
    if (!dirty) continue;
    const int x = (int)(t % nxp), c = (int)(t / nxp);  // c: z (AXIS 1) or y (AXIS 2)
    const LineAt<AXIS, true> at(g, x, c);
    const LineAt<AXIS, false> to(g, x, c);
    const LineStack st(stack, t, n);
    EnvRead env(st, env_build<AXIS>(st, at, in, n));
    for (int i = 0; i < n; ++i) {
      const int val = env.at(i);
      const size_t a = to(i);
      if (AXIS == 1) {
        if (out[a] != val) {
          out[a] = val;
          zflag[(size_t)nxp * i + x] = 1;
        }
      } else {
        out[a] = val;
      }
    }
  }
}

// Brick flags after the transform: obstacle bits, and finite D (voxel (0, 0, 0) of every brick lies
// inside the grid; with an obstacle anywhere every voxel is finite).
__global__ void k_ut_flags(GridView g) {
  const int64_t nb = (int64_t)g.BX * g.BY * g.BZ;
  for (int64_t b = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += (int64_t)gridDim.x * blockDim.x) {
    unsigned long long any = 0ull;
#pragma unroll
    for (int q = 0; q < 8; ++q) any |= g.occ[(size_t)b * 8 + q];
    uint32_t f = any ? F_OBST : 0u;
    if (g.dist[(size_t)b * kBrickVox] != kNone) f |= F_FINITE | F_G2FIN | F_G1FIN;
    g.bflags[b] = f;
  }
}

// y (AXIS 1: g1 -> g2) or z (AXIS 2: g2 -> D) pass of lines that fit shared memory: a block per tile of
// 32 lines (8 along x times 4 across; half of a brick column), staged whole as planes of 32 words, then
// the bracketed minima of line_min.cuh, each warp on its own bricks.  Missing inputs (kNone, and the
// ragged end of the line) stay the largest candidates: kNone + d^2 is at least kNone and fits 32 bits.
// UPD (an update): only the lines of the tile whose dirty byte is set (cleared once read); the y pass
// writes the g2 values that changed and sets the z-line byte of each.
// Bound by issue (searches and candidates, about 40 instructions a voxel) with 8 B of memory traffic a
// voxel under it.  512 x 512 x 256 tunnel scene: y 0.24 ms, z 0.21 ms (the stack kernels 0.58 and 0.66;
// memory alone would take 0.08); dirty lines of its first lidar frames 0.18 and 0.17 ms (0.42 and 0.26).
// Isolated obstacles far apart (2e-5 of the voxels) take y 0.31, z 0.22 (0.19 and 0.34).
// kLineMax is what shared memory holds: 152 B a position with minima and arguments, of 227 KB.
constexpr int kLineMax = 1496;
__host__ __device__ inline int line_bricks(int n) { return (n + 7) >> 3; }
__host__ __device__ inline size_t line_smem(int n) {
  const size_t nb = (size_t)line_bricks(n);
  return nb * 8 * 128 + nb * 128 + (nb + 1) * 64;
}

template <int AXIS, bool UPD>
__global__ void k_ut_line(GridView g, const int32_t* __restrict__ in, int32_t* __restrict__ out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int n = AXIS == 1 ? g.ny : g.nz, nb = line_bricks(n), nc = AXIS == 1 ? g.nz : g.ny;
  uint32_t* val = reinterpret_cast<uint32_t*>(smem);               // [8 nb][32]
  uint32_t* bmin = val + (size_t)nb * 256;                         // [nb][32]
  uint16_t* args = reinterpret_cast<uint16_t*>(bmin + nb * 32);    // [nb + 1][32]
  __shared__ uint32_t lmin[32];                                    // the lines' minima
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
  // tile: brick column (bx, bc), lines c = 8 bc + 4 h + (lane >> 3)
  const int h = (int)(blockIdx.x & 1), bx = (int)((blockIdx.x >> 1) % g.BX), bc = (int)((blockIdx.x >> 1) / g.BX);
  const int x = 8 * bx + (lane & 7), c = 8 * bc + 4 * h + (lane >> 3);
  bool live = x < g.nx && c < nc;
  if (UPD) {
    uint8_t* flag = reinterpret_cast<uint8_t*>(g.ut_bits + ut_row_words(g) + (AXIS == 1 ? 0 : ut_yline_words(g)));
    const size_t fi = (size_t)ut_nxp(g) * c + x;
    live = live && flag[fi] != 0;
    const unsigned dirty = __ballot_sync(0xffffffffu, live);
    if (!dirty) return;  // block-uniform: every warp read the same 32 bytes
    __syncthreads();     // all of them, before they are cleared
    if (warp == 0) {
      if (live) flag[fi] = 0;
      if (lane == 0) atomicAdd(&g.items_ctr[AXIS], __popc(dirty));
    }
  }
  const size_t bstride = (size_t)kBrickVox * (AXIS == 1 ? (size_t)g.BX : (size_t)g.BX * g.BY);
  const size_t base = (size_t)(AXIS == 1 ? ut_slot(g, bx, 0, bc) : ut_slot(g, bx, bc, 0)) * kBrickVox;
  if (warp == 0) lmin[lane] = (uint32_t)kNone;
  // stage: 16 bytes per copy, eight to a plane; positions past the line's end are kNone
  for (int i = threadIdx.x; i < nb * 64; i += blockDim.x) {
    const int pos = i >> 3;
    if (pos < n) {
      const int32_t* src = in + base + (size_t)(pos >> 3) * bstride + 64 * (pos & 7) + 32 * h + 4 * (i & 7);
      asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(val + 4 * i)),
                   "l"(src)
                   : "memory");
    } else {
      reinterpret_cast<int4*>(val)[i] = make_int4(kNone, kNone, kNone, kNone);
    }
  }
  asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  for (int b = warp; b < nb; b += nw) {
    const uint32_t m = line_brick_min(val + b * 256 + lane);
    bmin[b * 32 + lane] = m;
    atomicMin(&lmin[lane], m);
  }
  __syncthreads();
  const uint32_t least = lmin[lane];
  const bool some = live && least != (uint32_t)kNone;  // a line without a finite input is kNone throughout
  // arguments at the brick boundaries 8 b (the last one at n - 1): every eighth first, then the rest
  for (int q = warp; 8 * q < nb + 8; q += nw) {
    const int b = min(8 * q, nb), p = min(8 * b, n - 1);
    uint32_t best = some ? ~0u : 0u;
    int arg = 0;
    line_argmin(val + lane, bmin + lane, least, p, 0, nb - 1, best, arg);
    args[b * 32 + lane] = (uint16_t)arg;
  }
  __syncthreads();
  for (int b = warp; b < nb; b += nw) {
    if ((b & 7) == 0) continue;
    const int p = 8 * b, a0 = args[(b & ~7) * 32 + lane], a1 = args[min((b & ~7) + 8, nb) * 32 + lane];
    const uint32_t c0 = val[a0 * 32 + lane] + (uint32_t)((p - a0) * (p - a0));
    const uint32_t c1 = val[a1 * 32 + lane] + (uint32_t)((p - a1) * (p - a1));
    uint32_t best = some ? min(c0, c1) : 0u;
    int arg = c0 <= c1 ? a0 : a1;
    line_argmin(val + lane, bmin + lane, least, p, min(a0, a1) >> 3, max(a0, a1) >> 3, best, arg);
    args[b * 32 + lane] = (uint16_t)arg;
  }
  __syncthreads();
  for (int b = warp; b < nb; b += nw) {
    if (!live) continue;
    const int a0 = args[b * 32 + lane], a1 = args[b * 32 + 32 + lane];
    uint32_t r[8];
    line_outputs(val + lane, bmin + lane, 8 * b, min(a0, a1), some ? max(a0, a1) : -1, r);
    int32_t* dst = out + base + (size_t)b * bstride + (AXIS == 1 ? ut_vox(x, 0, c) : 32 * h + lane);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      const int o = (int)min(r[k], (uint32_t)kNone), at = k * (AXIS == 1 ? 8 : 64);
      if (8 * b + k >= n) break;
      if (UPD && AXIS == 1) {
        if (dst[at] != o) {
          dst[at] = o;
          reinterpret_cast<uint8_t*>(g.ut_bits + ut_row_words(g) + ut_yline_words(g))[(size_t)ut_nxp(g) * (8 * b + k) + x] = 1;
        }
      } else {
        dst[at] = o;
      }
    }
  }
}

template <bool INCR>
cudaError_t launch_x(const GridView& g, cudaStream_t st) {
  // at most 46,341 voxels along x (the grid's size limit): 182 steps, 46,592 bytes of carries
  const size_t smem = (size_t)kUtXWarps * ((g.BX + 31) / 32) * 8 * sizeof(int32_t);
  VDB_LAUNCH(k_ut_x<INCR>, ut_blocks((int64_t)g.BY * g.BZ * 8 * 32), 32 * kUtXWarps, smem, st, g);
  return cudaGetLastError();
}

template <int AXIS, bool UPD>
cudaError_t launch_line(const GridView& g, const int32_t* in, int32_t* out, cudaStream_t st) {
  const int n = AXIS == 1 ? g.ny : g.nz;
  const int64_t tiles = 2ll * g.BX * (AXIS == 1 ? g.BZ : g.BY);
  const cudaError_t e = cudaFuncSetAttribute(k_ut_line<AXIS, UPD>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                            (int)line_smem(kLineMax));
  if (e != cudaSuccess) return e;
  // blocks of up to 1,024 where the compiled kernel's registers allow them (any whole number of warps serves;
  // declared bounds or registers made the compiler's code 1 % slower)
  static const int most = [] {
    cudaFuncAttributes a{};
    return cudaFuncGetAttributes(&a, k_ut_line<AXIS, UPD>) == cudaSuccess ? a.maxThreadsPerBlock & ~31 : 256;
  }();
  const int threads = std::min(n <= 64 ? 128 : (n <= 128 ? 256 : (n <= 768 ? 512 : 1024)), most);
  VDB_LAUNCH((k_ut_line<AXIS, UPD>), (unsigned)tiles, threads, line_smem(n), st, g, in, out);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ut_init(const GridView& g, cudaStream_t st) {
  VDB_LAUNCH(k_ut_nodes, ut_blocks((int64_t)g.NX * g.NY * g.NZ), kUT, 0, st, g);
  VDB_LAUNCH(k_ut_bricks, ut_blocks((int64_t)g.BX * g.BY * g.BZ), kUT, 0, st, g);
  return cudaGetLastError();
}

cudaError_t launch_ut_reset(const GridView& g, cudaStream_t st) {
  VDB_LAUNCH(k_ut_reset, ut_blocks((int64_t)g.BX * g.BY * g.BZ * 8), kUT, 0, st, g);
  return cudaGetLastError();
}

cudaError_t launch_ut_dense(const GridView& g, const uint8_t* grid, cudaStream_t st) {
  VDB_LAUNCH(k_ut_dense, ut_blocks((int64_t)g.BX * g.BY * g.BZ * 8), kUT, 0, st, g, grid);
  return cudaGetLastError();
}

// Where lines are too long to be staged: the line stacks (8 bytes per voxel of lines padded along x to a
// multiple of 32).
size_t ut_scratch_bytes(const GridView& g) {
  return g.ny > kLineMax || g.nz > kLineMax ? (size_t)ut_nxp(g) * g.ny * g.nz * sizeof(int2) : 0;
}

cudaError_t launch_ut_pass(const GridView& g, int axis, void* scratch, cudaStream_t st) {
  int32_t* g1 = reinterpret_cast<int32_t*>(g.g1);
  int32_t* g2 = reinterpret_cast<int32_t*>(g.g2);
  int2* stack = static_cast<int2*>(scratch);
  if (axis == 0) {
    return launch_x<false>(g, st);
  } else if (axis == 1 && g.ny <= kLineMax) {
    return launch_line<1, false>(g, g1, g2, st);
  } else if (axis == 1) {
    VDB_LAUNCH(k_ut_env<1>, ut_blocks((int64_t)g.nx * g.nz), kUT, 0, st, g, g1, g2, stack);
  } else {
    if (g.nz <= kLineMax) {
      const cudaError_t e = launch_line<2, false>(g, g2, g.dist, st);
      if (e != cudaSuccess) return e;
    } else {
      VDB_LAUNCH(k_ut_env<2>, ut_blocks((int64_t)g.nx * g.ny), kUT, 0, st, g, g2, g.dist, stack);
    }
    VDB_LAUNCH(k_ut_flags, ut_blocks((int64_t)g.BX * g.BY * g.BZ), kUT, 0, st, g);
  }
  return cudaGetLastError();
}

cudaError_t launch_ut_update_pass(const GridView& g, int axis, void* scratch, cudaStream_t st) {
  int32_t* g1 = reinterpret_cast<int32_t*>(g.g1);
  int32_t* g2 = reinterpret_cast<int32_t*>(g.g2);
  if (axis == 0) {
    return launch_x<true>(g, st);
  } else if (axis == 1 && g.ny <= kLineMax) {
    return launch_line<1, true>(g, g1, g2, st);
  } else if (axis == 1) {
    VDB_LAUNCH(k_ut_env_upd<1>, ut_blocks((int64_t)ut_nxp(g) * g.nz), kUT, 0, st, g, g1, g2, static_cast<int2*>(scratch));
  } else {
    if (g.nz <= kLineMax) {
      const cudaError_t e = launch_line<2, true>(g, g2, g.dist, st);
      if (e != cudaSuccess) return e;
    } else {
      VDB_LAUNCH(k_ut_env_upd<2>, ut_blocks((int64_t)ut_nxp(g) * g.ny), kUT, 0, st, g, g2, g.dist,
                 static_cast<int2*>(scratch));
    }
    VDB_LAUNCH(k_ut_flags, ut_blocks((int64_t)g.BX * g.BY * g.BZ), kUT, 0, st, g);
  }
  return cudaGetLastError();
}

}  // namespace vdbedt
