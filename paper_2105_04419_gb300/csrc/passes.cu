// The separable transform passes over the sparse brick grid.
//
// D(v) = min(dmax^2, min over occupied o of |v - o|^2) (paper Eq. 1 with the truncation of
// Sec. III) factorises along the axes because min distributes over +:
//   g1(x,y,z) = min over occupied (x',y,z) of (x'-x)^2          (x pass; saturated at dmax^2)
//   g2(x,y,z) = min over |d| <= W of d^2 + g1(x,y+d,z)         (y pass)
//   D(x,y,z)  = min over |d| <= W of d^2 + g2(x,y,z+d)         (z pass)
// with any window W >= dmax - 1 (offsets of dmax or more cost at least dmax^2 and can never beat
// the d = 0 term, which is already saturated).  Here W = 8R, R = floor((dmax + 6) / 8): exactly the
// halo of R bricks a pass reads on each side.  A brick that is not stored has no obstacle within
// R bricks, so every intermediate value in it is dmax^2: absent bricks read as dmax^2.
//
// All three passes run in one warp-specialised kernel, k_pass<R, RUN, AXIS>.  A work item is a run
// of RUN bricks along the pass axis; its slot list (the run plus R bricks of halo on each side) is
// prepared when the item is queued.  A producer warp streams each item's brick inputs into a
// three-stage shared-memory ring with bulk asynchronous copies (cp.async.bulk global -> shared,
// completion counted in bytes on a "full" mbarrier per stage) and fills absent bricks itself;
// RUN consumer warps each own one output brick of the item, wait on the stage's full barrier,
// compute, write, and release the stage on its "empty" barrier.  No block-wide barrier sits on
// the main path, so warps whose windows exit early run ahead.
//   x (AXIS 0): inputs are the 64-byte occupancy masks.  Each lane expands two x-lines: the line's
//     occupancy is gathered from the masks of bricks bx-R..bx+R (one byte each), the nearest set bits outside
//     the brick found by counts of leading and trailing zeros (x_compute_rows).  g1 is stored y-major so
//     that the y pass reads it as planes.
//   y, z (AXIS 1, 2): inputs are 1 KB bricks of g1 / g2.  In the staged column a plane along the
//     pass axis is 32 words (two voxels per word) and a lane's line is one word per plane, so the
//     32 lanes of a consumer read 32 consecutive words.
//
// Arithmetic of the windowed minimum: 16-bit integers, two voxels per 32-bit lane.  Every value is
// saturated at dmax^2 <= 2025 before it enters a window and a squared offset is at most 48^2, so a plain
// 32-bit add sums both halves (no carry between them).  Each lane owns 8 consecutive outputs of two
// neighbouring lines, pairing offsets +d and -d (window_min8).  The pruned form stops when (d + 1)^2
// reaches every output's current minimum in the warp, and skips windows whose input bricks hold no
// value below dmax^2.
//
// Grids with dmax above 45 (up to 181), and any grid tuned to variant 8, take the envelope kernels at
// the end of the file, whose work per voxel follows the distances, not the window.
#include "line_min.cuh"
#include "vdbedt_internal.cuh"

namespace vdbedt {

namespace {

// n in both halves of a word
__host__ __device__ constexpr uint32_t twice(uint32_t n) { return n * 0x10001u; }

// Sets or clears one bit of a brick's flags with a reduction (no value returned, so the warp does
// not wait for the word's round trip); each pass owns the bit it writes.
__device__ __forceinline__ void set_flag_bit(const GridView& g, int slot, uint32_t bit, bool on) {
  if (on)
    atomicOr(&g.bflags[slot], bit);
  else
    atomicAnd(&g.bflags[slot], ~bit);
}

// ---- asynchronous bulk copies and mbarriers (inline PTX) ----
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// Ordering between this thread's earlier generic-proxy accesses to shared memory and async-proxy
// writes issued after it.
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void bulk_copy_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
// Bounded wait for a phase of an mbarrier: gives up after one second of global time (or
// kWaitMaxPolls polls), sets the device error word and reports failure.
__device__ __forceinline__ bool mbar_wait_bounded(const GridView& g, uint64_t* bar, uint32_t parity) {
  const unsigned long long t0 = global_ns();
  for (uint32_t i = 0; i < kWaitMaxPolls; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((i & 63u) == 63u && global_ns() - t0 > kWaitLimitNs) break;
    if (i > 16) __nanosleep(64);
  }
  set_error(g, kErrTimeout);
  return false;
}

// One 8-output window minimum on packed registers:
//   out[k] = min over |d| <= W of v[k + W + d] + d^2, pairing +d and -d,
// where v[j] is plane j of the lane's staged column (c[j * 32]).  Planes are loaded when first
// needed: the 8 centre planes, then at offset d the two planes that enter the window (W - d and
// W + 7 + d), so only about 16 planes are live at a time and the early exit also skips the loads.
// With `prune`, the offsets stop once (d + 1)^2 is at least every output's current minimum in the
// warp (a farther candidate costs at least (d + 1)^2, so none can lower any output); the test runs
// every 4 offsets and is warp-uniform.
// The eight candidates of four offsets go in as three pairs of adds with a three-way minimum and two fused
// add-minima: the adds issue beside the minima, so the mix takes 1.4 cycles a candidate where fused
// add-minima alone take 2.0, adds with three-way minima 1.6 and fp16 adds with them 1.8 (fp16 fields
// before: y 0.330 and z 0.354 ms, now 0.313 and 0.332; 1024 x 1024 x 256 tunnel scene, dmax 32, runs of 4).
template <int W>
__device__ __forceinline__ void window_min8(const uint32_t* __restrict__ c, uint32_t (&out)[8], bool prune) {
  static_assert(W % 4 == 0, "window is a multiple of 4 offsets");
  uint32_t v[8 + 2 * W];
  uint32_t acc[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    v[k + W] = c[(k + W) * 32];
    acc[k] = v[k + W];
  }
  bool live = true;  // warp-uniform
#pragma unroll
  for (int ch = 0; ch < W / 4; ++ch) {
    if (live) {
      const int d = 4 * ch + 1;  // offsets d .. d + 3
#pragma unroll
      for (int dd = 0; dd < 4; ++dd) {
        v[W - d - dd] = c[(W - d - dd) * 32];
        v[W + 7 + d + dd] = c[(W + 7 + d + dd) * 32];
      }
      constexpr auto sq = [](int n) { return twice((uint32_t)(n * n)); };
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        uint32_t r = acc[k];
        r = __vimin3_u16x2(r, v[k + W - d] + sq(d), v[k + W + d] + sq(d));
        r = __viaddmin_u16x2(v[k + W - d - 1], sq(d + 1), r);
        r = __vimin3_u16x2(r, v[k + W + d + 1] + sq(d + 1), v[k + W - d - 2] + sq(d + 2));
        r = __viaddmin_u16x2(v[k + W + d + 2], sq(d + 2), r);
        r = __vimin3_u16x2(r, v[k + W - d - 3] + sq(d + 3), v[k + W + d + 3] + sq(d + 3));
        acc[k] = r;
      }
      if (prune && ch + 1 < W / 4) {
        const uint32_t mx = __vimax3_u16x2(__vimax3_u16x2(acc[0], acc[1], acc[2]), __vimax3_u16x2(acc[3], acc[4], acc[5]),
                                           __vmaxu2(acc[6], acc[7]));
        const uint32_t next = sq(d + 4);  // the next offset's square
        live = !__all_sync(0xffffffffu, __vmaxu2(mx, next) == next);
      }
    }
  }
#pragma unroll
  for (int k = 0; k < 8; ++k) out[k] = acc[k];
}

// ================================================================================================
// The three passes: warp-specialised kernel with a bulk-copy ring
// ================================================================================================
template <int R, int RUN, int AXIS>
struct ColShape {
  static constexpr int NB = RUN + 2 * R;                     // staged bricks per item
  static constexpr int NS = AXIS == 0 ? 8 : 3;               // ring stages (x stages are 64 B per brick)
  static constexpr int UNIT = AXIS == 0 ? 64 : 1024;         // bytes staged per brick
  static constexpr int STAGE_BYTES = NB * UNIT;
  static constexpr int META = 2 * NB;                        // slots, then input flags
  static constexpr int THREADS = 32 * (RUN + 1);
  static constexpr size_t DATA_BYTES = (size_t)NS * STAGE_BYTES;
  static constexpr size_t META_BYTES = (size_t)NS * META * 4;
  static constexpr size_t TABLE_BYTES = AXIS == 0 ? 4096 : 0;  // x pass: ByteTable
  static constexpr size_t SMEM = DATA_BYTES + ((META_BYTES + 15) & ~(size_t)15) + 2 * NS * 8 + TABLE_BYTES + 16;
};

// Distances inside one byte: entry m holds, for voxels 0 .. 7, the distance to the nearest set bit of m (1024:
// none), two voxels to a word.
struct ByteTable {
  uint32_t w[256][4];
  constexpr ByteTable() : w{} {
    for (int m = 0; m < 256; ++m)
      for (int x = 0; x < 8; ++x) {
        uint32_t best = 1024;
        for (int j = 0; j < 8; ++j)
          if ((m >> j) & 1) {
            const uint32_t d = (uint32_t)(j < x ? x - j : j - x);
            if (d < best) best = d;
          }
        w[m][x / 2] |= best << (16 * (x & 1));
      }
  }
};
__device__ const ByteTable kByteTable{};

// The table in shared memory, copied by the whole block (no barrier).
__device__ __forceinline__ void load_byte_table(uint4* table) {
  for (int i = threadIdx.x; i < 256; i += blockDim.x) table[i] = reinterpret_cast<const uint4*>(kByteTable.w)[i];
}

// Squared distances, at most dmax^2 (dmax2: dmax twice), of the eight voxels of a row's byte, two to a word: t the
// distances inside the byte, A and B those from its first voxel to the nearest bit before it and from its last to the
// nearest after it.
__device__ __forceinline__ uint4 x_squares(const uint4& t, int A, int B, uint32_t dmax2) {
  const uint32_t in[4] = {t.x, t.y, t.z, t.w}, a2 = twice((uint32_t)A), b2 = twice((uint32_t)B);
  uint32_t w[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const uint32_t l = a2 + (uint32_t)(2 * q | (2 * q + 1) << 16), h = b2 + (uint32_t)((7 - 2 * q) | (6 - 2 * q) << 16);
    const uint32_t d = __vminu2(__vimin3_u16x2(l, h, in[q]), dmax2);
    const uint32_t lo = d & 0xFFFFu;
    w[q] = (d >> 16) * (d & 0xFFFF0000u) + lo * lo;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// x pass of one brick from the masks of bricks bx - R .. bx + R (64 B each; byte y + 8 z is the x-row (y, z)).
// Lane: z = lane & 7, rows y0 = 2 (lane >> 3) and y0 + 1, whose bytes of brick b are rows2[b] (low, high).  g1 is
// stored y-major.  A row's nearest bits outside the brick are one count of leading zeros (left) and one of
// trailing zeros (right) of the four neighbouring bytes on that side (and of two more for R > 4); from those
// distances A and B the eight voxels have A + x and B + 7 - x, two to a word, against the distances inside
// the brick's own byte (a table), and the minimum, at most dmax, is squared.  Bound by issue: about 140
// instructions a brick and lane for 1 KB written; 1024 x 1024 x 256 tunnel scene, dmax 32: 0.115 ms, 0.106 in runs of 8 (a
// funnel shift and a count per voxel and side with a table of squares: 0.139).
template <int R>
__device__ __forceinline__ void x_compute_rows(const GridView& g, const uint32_t (&rows2)[2 * R + 1], int slot,
                                               const uint4* __restrict__ table) {
  const int lane = threadIdx.x & 31;
  const int z = lane & 7, y0 = (lane >> 3) * 2;
  const uint32_t dmax2 = twice((uint32_t)g.dmax);
  auto at = [&](int b) -> uint32_t { return b >= 0 && b <= 2 * R ? rows2[b] : 0u; };
  // the four bytes of bricks b .. b + 3 of either row
  auto four = [&](int b, uint32_t (&w)[2]) {
    const uint32_t t01 = __byte_perm(at(b), at(b + 1), 0x5140), t23 = __byte_perm(at(b + 2), at(b + 3), 0x5140);
    w[0] = __byte_perm(t01, t23, 0x5410);
    w[1] = __byte_perm(t01, t23, 0x7632);
  };
  uint32_t lw[2], rw[2];
  four(R - 4, lw);
  four(R + 1, rw);
  bool fin = false;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const uint32_t own = (rows2[R] >> (8 * r)) & 0xFFu;
    uint32_t w[4];
    int A = __clz(lw[r]) + 1, B = __clz(__brev(rw[r])) + 1;  // 33: none in the four bytes
    if constexpr (R > 4) {
      // the next two bytes on either side, the nearer one on top (left) or below (right)
      const uint32_t lf = ((at(R - 5) >> (8 * r)) & 0xFFu) << 8 | ((at(R - 6) >> (8 * r)) & 0xFFu);
      const uint32_t rf = ((at(R + 5) >> (8 * r)) & 0xFFu) | ((at(R + 6) >> (8 * r)) & 0xFFu) << 8;
      if (lw[r] == 0u) A = 33 + (lf ? __clz(lf << 16) : 32);
      if (rw[r] == 0u) B = 33 + (rf ? __ffs(rf) - 1 : 32);
    }
    if (own == 0u && min(A, B) >= g.dmax) {
      w[0] = w[1] = w[2] = w[3] = twice((uint32_t)g.INF);
    } else {
      fin = true;
      const uint4 v = x_squares(table[own], A, B, dmax2);
      w[0] = v.x, w[1] = v.y, w[2] = v.z, w[3] = v.w;
    }
    *reinterpret_cast<uint4*>(g.g1 + (size_t)slot * kBrickVox + (y0 + r) * 64 + z * 8) = make_uint4(w[0], w[1], w[2], w[3]);
  }
  const unsigned anyfin = __any_sync(0xffffffffu, fin);
  if (lane == 0) set_flag_bit(g, slot, F_G1FIN, anyfin);
}

template <int R>
__device__ __forceinline__ void x_compute(const GridView& g, const uint8_t* masks, int slot, const uint4* table) {
  const int lane = threadIdx.x & 31;
  const int z = lane & 7, y0 = (lane >> 3) * 2;
  uint32_t rows2[2 * R + 1];
#pragma unroll
  for (int b = 0; b <= 2 * R; ++b) rows2[b] = *reinterpret_cast<const uint16_t*>(masks + b * 64 + y0 + 8 * z);
  x_compute_rows<R>(g, rows2, slot, table);
}

// y or z pass of one brick: the staged column holds planes along the pass axis, 32 words each
// (two voxels per word); lane (xpair, a) reads one word per plane.
//   AXIS 1: g1 (y-major) -> g2 (z-major) + F_G2FIN;   AXIS 2: g2 -> D + F_FINITE.
template <int R, int AXIS>
__device__ __forceinline__ void window_compute(const GridView& g, const uint32_t* col, const int* fin_flags, int slot,
                                               int w, bool prune, uint32_t inf2) {
  constexpr int W = 8 * R;
  const int lane = threadIdx.x & 31;
  const int xp = lane & 3, a = lane >> 2;
  bool any_fin = !prune;
#pragma unroll
  for (int b = 0; b <= 2 * R; ++b) any_fin |= fin_flags[w + b] != 0;
  uint32_t out[8];
  if (any_fin) {
    // plane w * 8 of the stage is plane 0 of this output brick's window (output 0 minus W)
    window_min8<W>(col + a * 4 + xp + (size_t)w * 8 * 32, out, prune);
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) out[q] = inf2;
  }
  bool fin = false;
  if (AXIS == 1) {
    // g2, z-major: word z * 32 + y * 4 + xpair, here z = a and y = q
    uint32_t* dst = reinterpret_cast<uint32_t*>(g.g2 + (size_t)slot * kBrickVox) + a * 32 + xp;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      dst[q * 4] = out[q];
      fin |= out[q] != inf2;  // every value is at most dmax^2
    }
  } else {
    // D, z-major int32: pair index z * 32 + y * 4 + xpair, here y = a and z = q
    int2* dst = reinterpret_cast<int2*>(g.dist + (size_t)slot * kBrickVox) + a * 4 + xp;
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      fin |= out[q] != inf2;
      dst[q * 32] = make_int2((int)(out[q] & 0xFFFFu), (int)(out[q] >> 16));
    }
  }
  const unsigned anyfin = __any_sync(0xffffffffu, fin);
  if (lane == 0) {
    const uint32_t bit = AXIS == 1 ? F_G2FIN : F_FINITE;
    set_flag_bit(g, slot, bit, anyfin);
  }
}

// One work item = a run of RUN bricks along AXIS.  Warp 0 produces: it reads the item's slot list
// (prefetched two items ahead, with the input flags one item ahead), fills absent bricks of the
// stage, and starts one bulk copy per present brick (64 B masks for x, 1 KB g1 / g2 for y / z).
// Warps 1..RUN consume: warp w computes output brick w of the item from the stage, then
// releases it.  Every wait is bounded; on a timeout the error word is set and the block drains.
// Resident blocks per SM the window passes ask the register allocator for (at most 80 registers
// for RUN 4, 72 for RUN 8): enough warps to keep the packed-min pipe busy.
__host__ __device__ constexpr int pass_min_blocks(int run, int axis) {
  return axis == 0 ? (run == 4 ? 10 : (run == 8 ? 7 : 3)) : (run == 4 ? 5 : (run == 8 ? 3 : 1));
}

template <int R, int RUN, int AXIS>
__global__ void __launch_bounds__(32 * (RUN + 1), pass_min_blocks(RUN, AXIS))
    k_pass(GridView g, const int32_t* __restrict__ islots, int max_items, bool prune) {
  pdl_enter();
  using S = ColShape<R, RUN, AXIS>;
  constexpr int NB = S::NB, NS = S::NS;
  extern __shared__ __align__(16) unsigned char smem[];
  unsigned char* data = smem;
  int* meta = reinterpret_cast<int*>(smem + S::DATA_BYTES);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::DATA_BYTES + ((S::META_BYTES + 15) & ~(size_t)15));
  uint64_t* empty = full + NS;
  uint4* table = reinterpret_cast<uint4*>(empty + NS);  // 16-byte aligned: whole pairs of barriers before it
  const int nitems = min(g.items_ctr[AXIS], max_items);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t inf2 = twice((uint32_t)g.INF);
  if (threadIdx.x == 0) {
    for (int s = 0; s < NS; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], RUN);
    }
  }
  if (AXIS == 0) load_byte_table(table);
  __syncthreads();

  if (warp == 0) {
    // ---------------- producer ----------------
    const void* src_base = AXIS == 0 ? (const void*)g.occ : (AXIS == 1 ? (const void*)g.g1 : (const void*)g.g2);
    const uint32_t in_fin = AXIS == 1 ? F_G1FIN : F_G2FIN;
    auto slot_of = [&](int item) -> int {
      return (item < nitems && lane < NB) ? islots[(size_t)item * kItemSlots + lane] : -1;
    };
    auto flag_of = [&](int slot) -> int { return (AXIS == 0 || slot < 0) ? 0 : ((g.bflags[slot] & in_fin) != 0); };
    int it = blockIdx.x;
    int sl_cur = slot_of(it), sl_nxt = slot_of(it + (int)gridDim.x);
    int fl_cur = flag_of(sl_cur);
    int k = 0;
    for (; it < nitems; it += gridDim.x, ++k) {
      const int sl_nn = slot_of(it + 2 * (int)gridDim.x);  // prefetch two items ahead
      const int fl_nxt = flag_of(sl_nxt);                  // and the next item's flags
      const int s = k % NS, u = k / NS;
      if (u > 0 && !mbar_wait_bounded(g, &empty[s], (u - 1) & 1)) break;
      if (lane < NB) {
        meta[s * S::META + lane] = sl_cur;
        meta[s * S::META + NB + lane] = fl_cur;
      }
      const unsigned present = __ballot_sync(0xffffffffu, lane < NB && sl_cur >= 0);
      unsigned absent = __ballot_sync(0xffffffffu, lane < NB && sl_cur < 0);
      uint4* stage = reinterpret_cast<uint4*>(data + (size_t)s * S::STAGE_BYTES);
      constexpr int U16 = S::UNIT / 16;  // 16-byte words per staged brick
      while (absent) {
        const int b = __ffs(absent) - 1;
        absent &= absent - 1;
        const uint32_t fill = AXIS == 0 ? 0u : inf2;
        for (int q = lane; q < U16; q += 32) stage[b * U16 + q] = make_uint4(fill, fill, fill, fill);
      }
      __syncwarp();
      if (lane == 0) {
        fence_proxy_async_smem();
        mbar_arrive_expect_tx(&full[s], (uint32_t)__popc(present) * (uint32_t)S::UNIT);
      }
      __syncwarp();
      if ((present >> lane) & 1u)
        bulk_copy_g2s(data + (size_t)s * S::STAGE_BYTES + lane * S::UNIT,
                      reinterpret_cast<const unsigned char*>(src_base) + (size_t)sl_cur * S::UNIT, (uint32_t)S::UNIT,
                      &full[s]);
      sl_cur = sl_nxt;
      fl_cur = fl_nxt;
      sl_nxt = sl_nn;
    }
    // after a timeout, let copies already issued land before the block can exit
    if (it < nitems)
      for (int j = max(0, k - NS); j < k; ++j) mbar_wait_bounded(g, &full[j % NS], (j / NS) & 1);
    return;
  }

  // ---------------- consumers ----------------
  const int w = warp - 1;  // output brick of the item
  int k = 0;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x, ++k) {
    const int s = k % NS, u = k / NS;
    if (!mbar_wait_bounded(g, &full[s], u & 1)) break;
    const int* m = meta + s * S::META;
    const int slot = m[w + R];
    if (slot >= 0) {
      const unsigned char* stage = data + (size_t)s * S::STAGE_BYTES;
      if (AXIS == 0)
        x_compute<R>(g, stage + w * 64, slot, table);
      else
        window_compute<R, AXIS>(g, reinterpret_cast<const uint32_t*>(stage), m + NB, slot, w, prune, inf2);
    }
    __syncwarp();
    if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&empty[s])) : "memory");
  }
}

// x pass with plain loads: one warp per output brick of the queued runs; each lane reads its two
// mask bytes of the 2R + 1 bricks of the window straight from global memory (the masks of
// neighbouring bricks are shared through L1 / L2) and writes its 32 bytes of g1.
template <int R>
__global__ void __launch_bounds__(256) k_x_direct(GridView g, const int32_t* __restrict__ islots, int max_items,
                                                  int run) {
  pdl_enter();
  constexpr int NBX = 2 * R + 1;
  const int nitems = min(g.items_ctr[0], max_items);
  const int lane = threadIdx.x & 31;
  const int z = lane & 7, y0 = (lane >> 3) * 2;
  const int64_t total = (int64_t)nitems * run;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const unsigned char* occ = reinterpret_cast<const unsigned char*>(g.occ);
  __shared__ uint4 table[256];
  load_byte_table(table);
  __syncthreads();
  for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w < total; w += nw) {
    const int item = (int)(w / run), j = (int)(w % run);
    const int32_t* sl = islots + (size_t)item * kItemSlots + j;
    const int s = lane < NBX ? __ldg(sl + lane) : -1;
    const int slot = __shfl_sync(0xffffffffu, s, R);
    if (slot < 0) continue;  // warp-uniform
    uint32_t rows2[NBX];
#pragma unroll
    for (int b = 0; b < NBX; ++b) {
      const int sb = __shfl_sync(0xffffffffu, s, b);
      rows2[b] = sb >= 0 ? (uint32_t)__ldg(reinterpret_cast<const uint16_t*>(occ + (size_t)sb * 64 + y0 + 8 * z)) : 0u;
    }
    x_compute_rows<R>(g, rows2, slot, table);
  }
}

// ------------------------------------------------------------------------------------------------
// Envelope kernels (any dmax up to 181; the only form above 45, variant 8 below it).
//
// Fields as in the windowed kernels (16-bit integers, g1 y-major, g2 z-major).  A work
// item is a run of kEnvRun bricks along the pass axis (a node's length); each kernel finds the
// run's bricks and their R bricks of halo on each side through the node tables.
//   x: the distance to the nearest occupied voxel of an x-line, from the line's bits.
//   y, z: for one line f(0 .. n-1) along the axis (the run and its halo, n = 8 (kEnvRun + 2R)),
//      every output i needs min over j of (i - j)^2 + f(j) (any input farther than the halo costs at
//      least (W + 1)^2 >= dmax^2): the walk of line_min.cuh.  Work per voxel follows the distances, not the
//      window.
// ------------------------------------------------------------------------------------------------
constexpr int kEnvRun = 16;

// x pass (nearest set bit of a binary line): a block per item at a time, the masks of the run and its
// halo staged in shared memory (17 words apart, so that a byte of 32 neighbouring bricks takes 32
// banks).  A warp takes two x-rows at a time, neighbours along z: ballots over the staged bricks (at
// most 62) give a 64-bit word of the bricks that hold a bit of the row, from which each of the run's
// bricks has its nearest set bits beyond itself by one count of leading and one of trailing zeros --
// lanes 0-15 for one row, 16-31 for the other, whose 16-byte results share a sector.  Bound by issue:
// 512 x 512 x 256 tunnel scene, dmax 64: 0.060 ms (the brick's voxels one by one instead of x_squares: 0.075; the
// neighbours' bytes scanned outward: 0.149).
constexpr int kEnvMaxNB = kEnvRun + 2 * 23;
__global__ void __launch_bounds__(256) k_env_x(GridView g, const unsigned long long* __restrict__ items, int max_items) {
  pdl_enter();
  __shared__ int slots[kEnvMaxNB];
  __shared__ uint32_t masks[64 * 17];  // bricks past the halo stay empty
  __shared__ uint32_t fin[kEnvRun];
  __shared__ uint4 table[256];
  load_byte_table(table);
  const int R = g.R, NB = kEnvRun + 2 * R, dmax = g.dmax;
  const uint32_t inf2 = twice((uint32_t)g.INF), dmax2 = twice((uint32_t)dmax);
  const int nitems = min(g.items_ctr[0], max_items);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int i = threadIdx.x; i < 64 * 17; i += blockDim.x) masks[i] = 0u;
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    int bx0, by, bz;
    unpack_brick(items[it], bx0, by, bz);
    __syncthreads();  // the previous item's shared memory is no longer read
    if ((int)threadIdx.x < NB) slots[threadIdx.x] = find_brick(g, bx0 - R + (int)threadIdx.x, by, bz);
    if (threadIdx.x < kEnvRun) fin[threadIdx.x] = 0u;
    __syncthreads();
    for (int i = threadIdx.x; i < NB * 16; i += blockDim.x) {
      const int s = slots[i >> 4];
      masks[(i >> 4) * 17 + (i & 15)] = s >= 0 ? __ldg(reinterpret_cast<const uint32_t*>(g.occ) + (size_t)s * 16 + (i & 15)) : 0u;
    }
    __syncthreads();
    auto row_byte = [&](int b, int row) { return (masks[b * 17 + (row >> 2)] >> (8 * (row & 3))) & 0xFFu; };
    const int o = R + (lane & 15);  // this lane's brick of the run
    const int slot = slots[o];
    bool any = false;
    for (int u = warp; u < 32; u += 8) {
      const int y = u & 7, z = 2 * (u >> 3);  // rows (y, z) and (y, z + 1): bytes y + 8 z and y + 8 z + 8
      unsigned long long w[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int row = y + 8 * (z + h);
        const unsigned lo = __ballot_sync(0xffffffffu, row_byte(lane, row) != 0u);
        const unsigned hi = __ballot_sync(0xffffffffu, row_byte(lane + 32, row) != 0u);
        w[h] = ((unsigned long long)hi << 32) | lo;
      }
      const int row = y + 8 * (z + (lane >> 4));
      const unsigned long long m = lane < 16 ? w[0] : w[1];
      const uint32_t own = row_byte(o, row);
      const unsigned long long ml = m & ((1ull << o) - 1ull), mr = (m >> o) >> 1;
      // from the brick's first voxel to the nearest set bit before it, and from its last voxel to the nearest after
      int A = 1 << 10, B = 1 << 10;
      if (ml) {
        const int b = 63 - __clzll((long long)ml);
        A = 8 * (o - b) - (31 - __clz(row_byte(b, row)));
      }
      if (mr) {
        const int b = o + __ffsll((long long)mr);
        B = 8 * (b - o) - 8 + __ffs(row_byte(b, row));
      }
      uint4 w4 = make_uint4(inf2, inf2, inf2, inf2);
      if (own != 0u || min(A, B) < dmax) {
        any = true;
        w4 = x_squares(table[own], A, B, dmax2);
      }
      if (slot >= 0)  // g1 is y-major: voxel x + 8 z + 64 y
        *reinterpret_cast<uint4*>(g.g1 + (size_t)slot * kBrickVox + 64 * y + 8 * (row >> 3)) = w4;
    }
    if (any) atomicOr(&fin[lane & 15], 1u);
    __syncthreads();
    if (threadIdx.x < kEnvRun && slots[R + threadIdx.x] >= 0)
      set_flag_bit(g, slots[R + threadIdx.x], F_G1FIN, fin[threadIdx.x] != 0u);
  }
}

// y (AXIS 1: g1 -> g2) or z (AXIS 2: g2 -> D) pass: a block per item at a time, its run and halo staged
// whole in shared memory as planes of 64 lines (16-bit values; bricks that are absent or hold nothing
// below dmax^2 are filled with it), then line_min.cuh's walk, a lane per two lines and each warp on its own
// bricks.  Positions count from the first halo brick.
// Bound by issue; R halo bricks each side make the staged bytes (kEnvRun + 2R) / kEnvRun times the run's.
// 512 x 512 x 256 tunnel scene, dmax 64 / 128 / 181: y 0.16 / 0.23 / 0.31 ms, z 0.15 / 0.19 / 0.25 (a
// thread per line with its envelope in a local-memory deque: y 0.73 / 1.00 / 1.15, z 0.67 / 0.85 / 0.84; brackets
// over single lines: 0.26 and 0.22 at 64).  With isolated obstacles far apart the walk passes more bricks: at
// 2e-5 of the voxels and dmax 181 y takes 0.50 (0.40), z 0.23 (0.64), x 0.07 (0.37).
constexpr int kEnvBlock = 256;
// values, minima, squares of -8 NB .. 8 NB + 15
size_t env_smem(int R) { return (size_t)(kEnvRun + 2 * R) * (kBrickVox * 2 + 128 + 64) + 64; }

template <int AXIS>
__global__ void __launch_bounds__(kEnvBlock) k_env_line(GridView g, const unsigned long long* __restrict__ items,
                                                        int max_items) {
  pdl_enter();
  extern __shared__ __align__(16) uint32_t smem32[];
  __shared__ int slots[kEnvMaxNB];   // stored bricks of the run and its halo (-1: none)
  __shared__ int inslot[kEnvMaxNB];  // the same, -1 also where the brick's input is all dmax^2
  __shared__ uint32_t gmin[(kEnvMaxNB + 7) / 8 * 32];  // minima over eight bricks
  __shared__ __align__(16) uint32_t rows[kEnvBlock / 32][256];  // y pass: a warp's output brick, by row
  const int R = g.R, NB = kEnvRun + 2 * R, INF = g.INF;
  uint32_t* val = smem32;                  // [8 NB][32]
  uint32_t* bmin = val + NB * kBrickWords;  // [NB][32]
  uint32_t* sq = bmin + NB * 32 + 8 * NB;
  const int nitems = min(g.items_ctr[AXIS], max_items);
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  constexpr int nw = kEnvBlock / 32;
  const uint16_t* __restrict__ src = AXIS == 1 ? g.g1 : g.g2;
  const uint32_t in_fin = AXIS == 1 ? F_G1FIN : F_G2FIN;
  const uint32_t inf2 = twice((uint32_t)INF);
  for (int u = t - 8 * NB; u < 8 * NB + 16; u += kEnvBlock) sq[u] = line16_square(u);
  for (int it = blockIdx.x; it < nitems; it += gridDim.x) {
    int bx, by, bz;
    unpack_brick(items[it], bx, by, bz);
    __syncthreads();  // the previous item's shared memory is no longer read
    if (t < NB) {  // at most 62
      const int s = AXIS == 1 ? find_brick(g, bx, by - R + t, bz) : find_brick(g, bx, by, bz - R + t);
      slots[t] = s;
      inslot[t] = (s >= 0 && (g.bflags[s] & in_fin)) ? s : -1;
    }
    const bool some = __syncthreads_or(t < NB && inslot[t] >= 0);
    uint32_t least = inf2;
    if (some) {
      for (int i = t; i < NB * 64; i += kEnvBlock) {  // 16 bytes each, 64 to a brick
        const int s = inslot[i >> 6];
        if (s >= 0)
          asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(val + 4 * i)),
                       "l"(src + (size_t)s * kBrickVox + 8 * (i & 63))
                       : "memory");
        else
          reinterpret_cast<uint4*>(val)[i] = make_uint4(inf2, inf2, inf2, inf2);
      }
      asm volatile("cp.async.commit_group;\n\tcp.async.wait_group 0;" ::: "memory");
      __syncthreads();
      for (int q = warp; 8 * q < NB; q += nw) {
        uint32_t m8 = ~0u;
        for (int b = 8 * q; b < min(8 * q + 8, NB); ++b) {
          const uint32_t m = inslot[b] >= 0 ? line16_min8(val + b * kBrickWords + lane) : inf2;
          bmin[b * 32 + lane] = m;
          m8 = __vminu2(m8, m);
        }
        gmin[q * 32 + lane] = m8;
      }
      __syncthreads();
      for (int q = 0; 8 * q < NB; ++q) least = __vminu2(least, gmin[q * 32 + lane]);
    }
    const bool live = least != inf2;  // (lines without an input below dmax^2 are dmax^2)
    for (int b = warp; b < kEnvRun; b += nw) {
      const int slot = slots[R + b];
      if (slot < 0) continue;  // warp-uniform
      uint32_t r[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) r[k] = inf2;
      if (__any_sync(0xffffffffu, live))
        line16_outputs(val + lane, bmin + lane, gmin + lane, sq, least, NB, R + b, live, r);
      uint32_t least_out = inf2;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        r[k] = __vminu2(r[k], inf2);
        least_out = __vminu2(least_out, r[k]);
      }
      if (AXIS == 1) {
        // g2 is z-major: a lane's word of eight rows of plane z = lane >> 2, gathered so that a lane
        // stores rows
        uint32_t* w = rows[warp];
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k) w[32 * (lane >> 2) + 4 * k + (lane & 3)] = r[k];
        __syncwarp();
        uint4* dst = reinterpret_cast<uint4*>(g.g2 + (size_t)slot * kBrickVox);
        dst[lane] = reinterpret_cast<const uint4*>(w)[lane];
        dst[lane + 32] = reinterpret_cast<const uint4*>(w)[lane + 32];
      } else {
        int2* dst = reinterpret_cast<int2*>(g.dist + (size_t)slot * kBrickVox) + lane;
#pragma unroll
        for (int k = 0; k < 8; ++k) dst[32 * k] = make_int2((int)(r[k] & 0xFFFFu), (int)(r[k] >> 16));
      }
      const bool f = __any_sync(0xffffffffu, least_out != inf2);
      if (lane == 0) set_flag_bit(g, slot, AXIS == 1 ? F_G2FIN : F_FINITE, f);
    }
  }
}

int g_num_sms = 0;
int num_sms() {
  if (!g_num_sms) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&g_num_sms, cudaDevAttrMultiProcessorCount, dev);
    if (g_num_sms <= 0) g_num_sms = 1;
  }
  return g_num_sms;
}

// Persistent launch of an envelope kernel: as many blocks as fit on the GPU at once (items are
// taken grid-stride; blocks beyond the queued count exit at once).
template <typename K>
cudaError_t launch_env_kernel(K kernel, int threads, size_t smem, const GridView& g, const unsigned long long* items,
                              bool chained, cudaStream_t st) {
  if (g.item_cap <= 0) return cudaSuccess;
  // the largest radius's shared memory, whatever this grid's: concurrent callers set the same value
  cudaError_t e = smem ? cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)env_smem(23)) : cudaSuccess;
  if (e != cudaSuccess) return e;
  int per_sm = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, threads, smem);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  int grid = num_sms() * per_sm;
  if (grid > g.item_cap) grid = g.item_cap;
  if (chained)
    VDB_LAUNCH_PDL(kernel, grid, threads, smem, st, g, items, (int)g.item_cap);
  else
    VDB_LAUNCH(kernel, grid, threads, smem, st, g, items, g.item_cap);
  return cudaGetLastError();
}

// Envelope pass along `axis`.
cudaError_t launch_env(const GridView& g, int axis, const Items& it, bool chained, cudaStream_t st) {
  if (axis == 0) return launch_env_kernel(k_env_x, 256, 0, g, it.run[0], chained, st);
  if (axis == 1) return launch_env_kernel(k_env_line<1>, kEnvBlock, env_smem(g.R), g, it.run[1], chained, st);
  return launch_env_kernel(k_env_line<2>, kEnvBlock, env_smem(g.R), g, it.run[2], chained, st);
}

template <int R, int RUN, int AXIS>
cudaError_t pass_window(const GridView& g, const int32_t* islots, int max_items, bool chained, cudaStream_t st,
                        bool prune) {
  using S = ColShape<R, RUN, AXIS>;
  auto kernel = k_pass<R, RUN, AXIS>;
  if (max_items <= 0) return cudaSuccess;
  // attributes and resident blocks per SM, set up once per device (0: not yet)
  static int per_sm_dev[64] = {};
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  int per_sm = dev >= 0 && dev < 64 ? per_sm_dev[dev] : 0;
  if (per_sm == 0) {
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)S::SMEM);
    if (e != cudaSuccess) return e;
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, 100);
    if (e != cudaSuccess) return e;
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, S::THREADS, S::SMEM);
    if (e != cudaSuccess) return e;
    if (per_sm < 1) per_sm = 1;
    if (dev >= 0 && dev < 64) per_sm_dev[dev] = per_sm;
  }
  int grid = num_sms() * per_sm;
  if (grid > max_items) grid = max_items;
  if (chained)
    VDB_LAUNCH_PDL(kernel, grid, S::THREADS, S::SMEM, st, g, islots, max_items, prune);
  else
    VDB_LAUNCH(kernel, grid, S::THREADS, S::SMEM, st, g, islots, max_items, prune);
  return cudaGetLastError();
}

template <int RUN, int AXIS>
cudaError_t pass_window_r(const GridView& g, const int32_t* islots, int max_items, bool chained, cudaStream_t st,
                          bool prune) {
  switch (g.R) {
    case 1: return pass_window<1, RUN, AXIS>(g, islots, max_items, chained, st, prune);
    case 2: return pass_window<2, RUN, AXIS>(g, islots, max_items, chained, st, prune);
    case 3: return pass_window<3, RUN, AXIS>(g, islots, max_items, chained, st, prune);
    case 4: return pass_window<4, RUN, AXIS>(g, islots, max_items, chained, st, prune);
    case 5: return pass_window<5, RUN, AXIS>(g, islots, max_items, chained, st, prune);
    case 6: return pass_window<6, RUN, AXIS>(g, islots, max_items, chained, st, prune);
  }
  return cudaErrorInvalidValue;
}

template <int AXIS>
cudaError_t pass_window_run(const GridView& g, int run, const int32_t* islots, int max_items, bool chained,
                            cudaStream_t st, bool prune) {
  switch (run) {
    case 4: return pass_window_r<4, AXIS>(g, islots, max_items, chained, st, prune);
    case 8: return pass_window_r<8, AXIS>(g, islots, max_items, chained, st, prune);
    case 16: return pass_window_r<16, AXIS>(g, islots, max_items, chained, st, prune);
  }
  return cudaErrorInvalidValue;
}

// Self-test of the bounded waits: one thread waits on a phase that never completes (which = 0: an
// mbarrier with no arrivals, the wait of the pass kernels) or looks up a node whose insertion was
// left pending (which = 1: the wait of node creation).  Each gives up after its poll limit, sets
// the error word and returns.
__global__ void k_wait_selftest(GridView g, int which) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  if (which == 0) {
    mbar_init(&bar, 1);
    mbar_wait_bounded(g, &bar, 0);
  } else {
    const unsigned long long key = 0;
    g.hslots[hash_key(key) & g.hmask] = (key << kIndexBits) | kPending;
    get_or_create_node(g, key);
  }
}

template <int R>
cudaError_t x_direct_r(const GridView& g, const int32_t* islots, int max_items, int run, cudaStream_t st) {
  auto kernel = k_x_direct<R>;
  if (max_items <= 0) return cudaSuccess;
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, 256, 0);
  if (e != cudaSuccess) return e;
  if (per_sm < 1) per_sm = 1;
  VDB_LAUNCH(kernel, num_sms() * per_sm, 256, 0, st, g, islots, max_items, run);
  return cudaGetLastError();
}

cudaError_t x_direct(const GridView& g, const int32_t* islots, int max_items, int run, cudaStream_t st) {
  switch (g.R) {
    case 1: return x_direct_r<1>(g, islots, max_items, run, st);
    case 2: return x_direct_r<2>(g, islots, max_items, run, st);
    case 3: return x_direct_r<3>(g, islots, max_items, run, st);
    case 4: return x_direct_r<4>(g, islots, max_items, run, st);
    case 5: return x_direct_r<5>(g, islots, max_items, run, st);
    case 6: return x_direct_r<6>(g, islots, max_items, run, st);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_wait_selftest(const GridView& g, int which, cudaStream_t st) {
  VDB_LAUNCH(k_wait_selftest, 1, 32, 0, st, g, which);
  return cudaGetLastError();
}

bool windowed_form(const GridView& g) { return g.windowed != 0; }


// The windowed kernels address bricks by pool slot (the slot lists hold local slot + slot_base):
// their view has the per-brick pointers moved back to the first slot of the pool.
GridView pool_view(const GridView& g) {
  GridView p = g;
  const size_t b = (size_t)g.slot_base;
  p.occ = g.occ - b * 8;
  p.g1 = g.g1 - b * kBrickVox;
  p.g2 = g.g2 - b * kBrickVox;
  p.dist = g.dist - b * kBrickVox;
  p.bcoord = g.bcoord - b;
  p.bflags = g.bflags - b;
  p.bepoch = g.bepoch - b;
  p.slot_base = 0;
  return p;
}

// Passes over at most this many bricks of capacity are chained to the kernel before them (programmatic
// launch): there a launch costs as much as the pass (160^3: 65.7 us a call with its export, 70.2 without).
// A pass that fills the GPU is launched on its own: started early, its blocks take the places that the
// previous pass's leave one by one, and y and z together took 0.82 ms where they take 0.65 (1024 x 1024 x 256
// tunnel scene, dmax 32).  Nearer the line (transform alone, random cubes, dmax 16, chained / not): 8,000 bricks 37.8 / 44.6 us,
// 15,625 49.1 / 56.0, 17,576 51.9 / 59.7, 32,768 72.5 / 80.5, 64,000 116 / 122 -- chaining gains 7 us on either side of it, and
// loses only where the passes are long against that.  By capacity, which the host knows, not by the work: a map of 131,072
// bricks that holds few gives up the same 7 us.
constexpr int kChainBricks = 16384;

// Runs of 8 bricks share their halo over twice as many outputs as runs of 4 and halve the work lists: for whole
// transforms that fill the GPU, with halos of three bricks or more (1024 x 1024 x 256 tunnel scene: dmax 32
// lists 22 us, x 115, y 313, z 336 with 4, 16, 107, 305, 317 with 8; dmax 24 249 and 278, 248 and 266; at dmax
// 8 y takes 121 and 131).  Around the line both take the same (random cubes, dmax 32, 4 / 8: 15,625 bricks 57.5 / 58.3 us, 17,576
// 65.5 / 67.3, 32,768 90.4 / 91.1, 64,000 146 / 144), and so do large maps that hold few bricks (48 us for 3,000 voxels).
// Updates keep 4: their dirty runs are short.
constexpr int kLongRunBricks = 16384;
int effective_run(const GridView& g, const Tuning& t, int axis, bool whole) {
  if (!windowed_form(g)) return kEnvRun;
  if (t.run[axis]) return t.run[axis];
  return whole && g.item_cap > kLongRunBricks && g.R >= 3 ? 8 : 4;
}

cudaError_t launch_pass(const GridView& g, const Tuning& t, int axis, const Items& it, bool chained, cudaStream_t st) {
  chained = chained && g.item_cap <= kChainBricks;
  const bool prune = (t.variant & 3) != 1;
  if (windowed_form(g)) {
    const GridView p = pool_view(g);
    if (axis == 0 && (t.variant & kVariantXDirect)) return x_direct(p, it.slots[0], g.item_cap, t.run[0], st);
    if (axis == 0) return pass_window_run<0>(p, t.run[0], it.slots[0], g.item_cap, chained, st, prune);
    if (axis == 1) return pass_window_run<1>(p, t.run[1], it.slots[1], g.item_cap, chained, st, prune);
    return pass_window_run<2>(p, t.run[2], it.slots[2], g.item_cap, chained, st, prune);
  }
  // the envelope kernels find bricks through the grid's own tables (local slots)
  return launch_env(g, axis, it, chained, st);
}

}  // namespace vdbedt
