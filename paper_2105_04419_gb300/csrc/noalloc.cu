// vdbedt_edt_dense_noalloc: the exact truncated transform of a small dense grid that allocates
// nothing.
//
// Some callers cannot call cudaMalloc: code running while another part of the application holds a
// stream capture open, real-time control loops that must not enter the allocator, and embedded or
// plugin hosts whose device memory budget is fixed when the library is loaded.  For them this entry
// point computes the same D as a handle (vdbedt_create + vdbedt_set_occupancy_dense +
// vdbedt_global) but keeps its two intermediate fields (the x-line and in-plane squared distances)
// in a file-scope device array of fixed size instead of allocating them.  That array exists on
// every GPU that loads the library, for as long as the process runs.
//
// The array is shared by every call on a device and keeps the last call's contents; each call
// writes every scratch element it later reads, so nothing needs clearing.  Calls whose work
// overlaps on the GPU (on different streams, or from different threads without ordering) race on
// the array.
//
// Host code must not pass the array's name to a kernel (in host code it is a host-side stand-in,
// not a device address): the device address comes from cudaGetSymbolAddress, called with the
// device current.  Each call made while its stream is not being captured looks the address up
// again and refreshes the per-device cache, so a context torn down and recreated in between (for
// example by cudaDeviceReset) is followed; a call made during a stream capture uses the cached
// address, which is why the first call on a device must come before any capture.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <atomic>

#include "../../include/vdbedt.h"
#include "vdbedt_internal.cuh"

namespace {

constexpr int64_t kMaxVoxels = VDBEDT_NOALLOC_MAX_VOXELS;
constexpr int kMaxDevices = 64;

// g1 (x-line squared distance) at [0, kMaxVoxels), g2 (in-plane) at [kMaxVoxels, 2 kMaxVoxels).
static __device__ __align__(256) uint16_t g_noalloc_scratch[2 * kMaxVoxels];

std::atomic<uint16_t*> g_scratch_ptr[kMaxDevices];

// x: nearest occupied voxel along the x-line within dmax - 1, squared, saturated at dmax^2.  A warp per
// stretch of WORDS words of 32 voxels of a row: ballots over its bytes and HALO words more on each side
// (at least dmax - 1 voxels) give the words of bits, one per lane, and a word of those that are not empty, so
// that a voxel has its nearest set bits by counts of leading and trailing zeros of its own word and of the
// nearest other one.  117 x 96 x 83, dmax 24: 4.6 us (a thread per voxel scanning bytes outward: 27).
// Stretches of 20 words; of four where a few long rows would leave the GPU idle while a warp each works through
// twenty (a call on 1000 x 1000 x 1, dmax 12: 20 us, was 43).
template <int WORDS, int HALO>
__global__ void __launch_bounds__(128) k_dense_x(const uint8_t* __restrict__ occ, int nx, int64_t nrows, int dmax,
                                                 uint16_t* __restrict__ g1) {
  static_assert(WORDS + 2 * HALO <= 32, "a word per lane");
  vdbedt::pdl_enter();
  const int lane = threadIdx.x & 31, cap = dmax * dmax;
  const int nch = (nx + 32 * WORDS - 1) / (32 * WORDS);
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t < nrows * nch; t += nw) {
    const int64_t row = nch == 1 ? t : t / nch;
    const int x0 = ((int)(t - row * nch) * WORDS - HALO) * 32;  // position of word 0's first bit
    const uint8_t* src = occ + row * nx;
    const int j0 = max(0, -(x0 >> 5)), j1 = min(WORDS + 2 * HALO, (nx - x0 + 31) >> 5);  // words inside the row
    uint32_t word = 0u;  // this lane's word
    for (int j = j0; j < j1; j += 4) {
      uint8_t v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int x = x0 + 32 * (j + q) + lane;
        v[q] = j + q < j1 && x < nx ? __ldg(src + x) : (uint8_t)0;
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint32_t w = __ballot_sync(0xffffffffu, v[q] != 0);
        if (lane == j + q) word = w;
      }
    }
    const uint32_t some = __ballot_sync(0xffffffffu, word != 0u);
    for (int c = HALO; c < min(j1, HALO + WORDS); ++c) {
      const uint32_t w = __shfl_sync(0xffffffffu, word, c);
      const uint32_t before = some & ((1u << c) - 1u), after = (some >> c) >> 1;
      const int b = before ? 31 - __clz(before) : 0, a = after ? c + __ffs(after) : 31;
      const uint32_t wb = __shfl_sync(0xffffffffu, word, b), wa = __shfl_sync(0xffffffffu, word, a);
      const uint32_t le = w & ((2u << lane) - 1u), ge = w >> lane;
      const int dl = le ? lane - (31 - __clz(le)) : (before ? lane + 32 * (c - b) - (31 - __clz(wb)) : dmax);
      const int dr = ge ? __ffs(ge) - 1 : (after ? 32 * (a - c) - lane + __ffs(wa) - 1 : dmax);
      const int d = min(min(dl, dr), dmax), x = x0 + 32 * c + lane;
      if (x < nx) g1[row * nx + x] = (uint16_t)min(d * d, cap);
    }
  }
}

// The same for rows of at most 32 voxels: a warp per 32 / nx whole rows, one load and one ballot for all of
// them.  A call on 1 x 2048 x 1024, dmax 12: 34 us (354 with a warp per row, 84 with a thread per voxel).
__global__ void __launch_bounds__(128) k_dense_x_narrow(const uint8_t* __restrict__ occ, int nx, int64_t nrows, int dmax,
                                                        uint16_t* __restrict__ g1) {
  vdbedt::pdl_enter();
  const int lane = threadIdx.x & 31, cap = dmax * dmax;
  const int per = 32 / nx, r = lane / nx, x = lane - r * nx;  // rows of a warp, this lane's row and voxel
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; t * per < nrows; t += nw) {
    const bool in = r < per && t * per + r < nrows;
    const int64_t at = t * per * nx + lane;
    const uint32_t all = __ballot_sync(0xffffffffu, in && __ldg(occ + at) != 0);
    const uint32_t w = (all >> (lane - x)) & (0xffffffffu >> (32 - nx));
    const uint32_t le = w & ((2u << x) - 1u), ge = w >> x;
    const int dl = le ? x - (31 - __clz(le)) : dmax, dr = ge ? __ffs(ge) - 1 : dmax, d = min(min(dl, dr), dmax);
    if (in) g1[at] = (uint16_t)min(d * d, cap);
  }
}

// y (AXIS 1) or z (AXIS 2) of lines of up to kShortLine positions: a thread per output, outward along its line
// (eight outputs a thread would mostly lie past the end).  A call on 1000 x 1000 x 2 takes 30.3 us, 31.1 by eights;
// on 666 x 1000 x 3 30.1 and 28.1.
constexpr int kShortLine = 2;
template <int AXIS>
__global__ void __launch_bounds__(128) k_dense_short(const uint16_t* __restrict__ in, int nx, int ny, int nz, int dmax,
                                                     int reach, uint16_t* __restrict__ out16, int32_t* __restrict__ out32) {
  vdbedt::pdl_enter();
  const int64_t n = (int64_t)nx * ny * nz, stride = AXIS == 1 ? (int64_t)nx : (int64_t)nx * ny;
  const int cap = dmax * dmax, len = AXIS == 1 ? ny : nz;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int c = len == 1 ? 0 : (AXIS == 1 ? (int)((i / nx) % ny) : (int)(i / stride));
    int best = min((int)__ldg(in + i), cap);
    for (int d = 1; d < reach && d * d < best; ++d) {
      if (c - d >= 0) best = min(best, d * d + (int)__ldg(in + i - d * stride));
      if (c + d < len) best = min(best, d * d + (int)__ldg(in + i + d * stride));
    }
    if (AXIS == 2)
      out32[i] = best;
    else
      out16[i] = (uint16_t)best;
  }
}

// y (AXIS 1) or z (AXIS 2): min over |d| < dmax of d^2 + the previous field at offset d.  A thread per
// eight outputs along the axis (a warp's threads along x): the eight inputs among themselves, then plane by
// plane outward on both sides, each loaded once for all eight; every fourth plane the walk stops
// when the square of the next offset reaches the largest minimum.  (d + k)^2 = d^2 + 2 d k + k^2: the
// minima are kept less k^2, a multiply-add and half a three-way minimum per candidate and output.  Bound by
// the latency of the loads at such sizes: 117 x 96 x 83, dmax 24: about 6 us each, their launches
// overlapping the pass before (a thread per output: 14.5).  reach: where the walk ends, at most dmax.
template <int AXIS>
__global__ void __launch_bounds__(128) k_dense_win(const uint16_t* __restrict__ in, int nx, int ny, int nz, int dmax, int reach,
                                                   uint16_t* __restrict__ out16, int32_t* __restrict__ out32) {
  vdbedt::pdl_enter();
  const int cap = dmax * dmax, len = AXIS == 1 ? ny : nz, nb = (len + 7) / 8;
  const int64_t stride = AXIS == 1 ? (int64_t)nx : (int64_t)nx * ny;
  const int64_t n = AXIS == 1 ? (int64_t)nx * nb * nz : (int64_t)nx * ny * nb;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    int b;          // eighth of the line
    int64_t line;   // its first voxel
    if (AXIS == 1) {
      const int64_t r = i / nx;
      b = (int)(r % nb);
      line = i - r * nx + (r / nb) * nx * ny;
    } else {
      b = (int)(i / stride);
      line = i - b * stride;
    }
    const int c0 = 8 * b;
    auto at = [&](int c) -> int { return c >= 0 && c < len ? (int)__ldg(in + line + c * stride) : cap; };
    int acc[8];  // minimum of output k, less k^2
    {
      int f[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) f[k] = at(c0 + k);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        int m = f[k];
#pragma unroll
        for (int j = 0; j < 8; ++j) m = min(m, f[j] + (k - j) * (k - j));
        acc[k] = m - k * k;
      }
    }
    for (int d = 1; d < reach; d += 4) {
      int lo[4], hi[4], mx = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) mx = max(mx, acc[k] + k * k);
      if (d * d >= mx) break;
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        lo[q] = at(c0 - d - q);
        hi[q] = at(c0 + 7 + d + q);
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int e = d + q, h = e + 7;
        const int a = lo[q] + e * e, z = hi[q] + h * h;
#pragma unroll
        for (int k = 0; k < 8; ++k) acc[k] = __vimin3_s32(acc[k], a + 2 * e * k, z - 2 * h * k);
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if (c0 + k >= len) break;
      const int v = min(acc[k] + k * k, cap);
      if (AXIS == 2)
        out32[line + (c0 + k) * stride] = v;
      else
        out16[line + (c0 + k) * stride] = (uint16_t)v;
    }
  }
}

}  // namespace

namespace {

vdbedt_status noalloc_fail(vdbedt_status s, const char* msg) {
  vdbedt::set_last_error(msg);
  return s;
}

}  // namespace

extern "C" vdbedt_status vdbedt_edt_dense_noalloc(const uint8_t* occ, int32_t nx, int32_t ny, int32_t nz,
                                                  int32_t dmax, int32_t* out, void* stream) {
  if (!occ || !out) return noalloc_fail(VDBEDT_EINVAL, "vdbedt_edt_dense_noalloc: null pointer");
  if (nx < 1 || ny < 1 || nz < 1) return noalloc_fail(VDBEDT_EINVAL, "vdbedt_edt_dense_noalloc: size < 1");
  if (dmax < 1 || dmax > VDBEDT_DMAX_LIMIT)
    return noalloc_fail(VDBEDT_EINVAL, "vdbedt_edt_dense_noalloc: dmax outside [1, VDBEDT_DMAX_LIMIT]");
  const int64_t n = (int64_t)nx * ny * nz;
  if (n > kMaxVoxels)
    return noalloc_fail(VDBEDT_EINVAL, "vdbedt_edt_dense_noalloc: more than VDBEDT_NOALLOC_MAX_VOXELS voxels");
  // an error left pending by earlier work on this thread is not ours to report or to clear
  if (cudaPeekAtLastError() != cudaSuccess)
    return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: a CUDA error from earlier work is pending "
                                      "(read it with cudaGetLastError first)");
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices)
    return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: no current device");
  cudaStream_t st = (cudaStream_t)stream;
  cudaStreamCaptureStatus cs = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(st, &cs) != cudaSuccess) {
    cudaGetLastError();
    return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: invalid stream");
  }
  uint16_t* scratch = g_scratch_ptr[dev].load(std::memory_order_acquire);
  if (cs == cudaStreamCaptureStatusNone) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_noalloc_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: scratch address lookup failed");
    }
    scratch = static_cast<uint16_t*>(p);
    g_scratch_ptr[dev].store(scratch, std::memory_order_release);
  } else if (!scratch) {
    return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: first call on this device made during a stream "
                                      "capture (call it once before capturing)");
  }
  const auto blocks = [](int64_t threads) {
    const int64_t k = (threads + 127) / 128;
    return (unsigned)(k > 152 * 32 ? 152 * 32 : k);
  };
  uint16_t* g1 = scratch;
  uint16_t* g2 = scratch + kMaxVoxels;
  const int64_t nrows = (int64_t)ny * nz;
  if (nx <= 32) {
    VDB_LAUNCH(k_dense_x_narrow, blocks((nrows + 32 / nx - 1) / (32 / nx) * 32), 128, 0, st, occ, nx, nrows, dmax, g1);
  } else {
    // (rows of up to four words are one stretch either way)
    const bool few = nx > 128 && nrows * ((nx + 639) / 640) < 8192;
    const int64_t warps = nrows * (few ? (nx + 127) / 128 : (nx + 639) / 640);
    const auto kernel = !few ? k_dense_x<20, 6> : (dmax <= 32 ? k_dense_x<4, 1> : k_dense_x<4, 6>);
    VDB_LAUNCH(kernel, blocks(warps * 32), 128, 0, st, occ, nx, nrows, dmax, g1);
  }
  if (cudaGetLastError() != cudaSuccess) return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: x launch");
  const auto line = [&](auto wide, auto brief, int len, const uint16_t* in, uint16_t* out16, int32_t* out32) {
    const bool is_short = len <= kShortLine;
    // no offset reaches past the line; eight positions or fewer are all among themselves
    const int reach = is_short || len > 8 ? std::min((int)dmax, len) : 1;
    VDB_LAUNCH_PDL(is_short ? brief : wide, blocks(is_short ? n : n / len * ((len + 7) / 8)), 128, 0, st, in, (int)nx, (int)ny,
                   (int)nz, (int)dmax, reach, out16, out32);
    return cudaGetLastError();
  };
  if (line(k_dense_win<1>, k_dense_short<1>, ny, g1, g2, nullptr) != cudaSuccess)
    return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: y launch");
  if (line(k_dense_win<2>, k_dense_short<2>, nz, g2, nullptr, out) != cudaSuccess)
    return noalloc_fail(VDBEDT_ECUDA, "vdbedt_edt_dense_noalloc: z launch");
  return VDBEDT_OK;
}
