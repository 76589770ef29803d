// Reading the field: point queries, dense export, and the differentiable clearance cost.
//
// Query: D at voxel coordinates through the two-level interior (hash probe, child table); voxels
// outside the grid or in unstored bricks return the background dmax^2 (the paper's tile value,
// Sec. IV-A).  Nearest-obstacle query: the occupied voxel a cell's distance is measured to (the
// obstacle the paper keeps per cell, Sec. IV-B), found through the passes' per-axis fields.
//
// Clearance cost (Eq. 2, clearance term, as a squared hinge): per point p (metres),
//   u = p / vs (float32), i0 = floor(u) clamped to [0, n-2], t = u - i0,
//   corner distance d_c = vs * sqrt(D_c), d = trilinear(d_c, t), c = max(0, tau - d)^2,
//   cost[traj] = sum of c over the trajectory's points.
// Backward: dc/dp = -2 max(0, tau - d) (1 / vs) grad_t(trilinear), scaled by the upstream
// gradient of the trajectory's cost.  One warp per trajectory, points strided over the lanes,
// a warp shuffle sum for the forward.
#include "vdbedt_internal.cuh"

namespace vdbedt {

namespace {

__device__ __forceinline__ int sqdist_at(const GridView& g, int x, int y, int z) {
  if ((unsigned)x >= (unsigned)g.nx || (unsigned)y >= (unsigned)g.ny || (unsigned)z >= (unsigned)g.nz) return g.INF;
  int s = find_brick(g, x >> 3, y >> 3, z >> 3);
  if (s < 0) return g.INF;
  return g.dist[(size_t)s * kBrickVox + (x & 7) + 8 * (y & 7) + 64 * (z & 7)];
}

// caller coordinates are stored shifted by g.off (an unbounded grid's signed coordinates)
__global__ void k_query(GridView g, const int32_t* __restrict__ xyz, int64_t n, int32_t* __restrict__ out) {
  pdl_enter();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    out[i] = sqdist_at(g, xyz[3 * i] + g.off, xyz[3 * i + 1] + g.off, xyz[3 * i + 2] + g.off);
}

// The dense field: a warp per plane of a row of 16 bricks along x (one interior node's width, so one
// hash probe and 16 neighbouring child slots serve 8 x 128 outputs); unstored bricks are filled with
// the background without a read.  Bound by memory: 4 B written per voxel and 4 B read per stored one.
// VEC (rows and output aligned to 16 bytes): lane pairs read a brick's 32-byte row as two int4 and
// the warp writes 512 contiguous bytes per row, a plane's eight loads issued before its stores.
// Otherwise 4-byte stores, 128 contiguous bytes per warp.  1024 x 1024 x 256 with 89 % of the bricks
// stored: 0.32 ms, about 2.0 GB at 6.3 TB/s (a thread per voxel, each with its own probe and child
// read: 1.48 ms); the 4-byte form serves widths that are no multiple of 4.
template <bool VEC>
__global__ void __launch_bounds__(256) k_export_dense(GridView g, int32_t* __restrict__ out) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t units = (int64_t)g.NX * g.BY * g.BZ * 8;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; u < units; u += nw) {
    const int plane = (int)(u & 7);
    const int64_t r = u >> 3;
    const int qx = (int)(r % g.NX);
    const int64_t rb = r / g.NX;
    const int by = (int)(rb % g.BY), bz = (int)(rb / g.BY);
    const int z = 8 * bz + plane, x0 = 128 * qx, ny = min(8, g.ny - 8 * by);
    if (z >= g.nz) continue;  // warp-uniform
    // lanes 2j, 2j + 1: brick j of the row
    const int node = find_node(g, node_key_at(g, qx, by >> 4, bz >> 4));
    const int bx = 16 * qx + (lane >> 1);
    const int slot = node >= 0 && bx < g.BX ? g.child[(size_t)node * kNodeBricks + local_brick(bx, by, bz)] : -1;
    int32_t* dst = out + ((int64_t)z * g.ny + 8 * by) * g.nx + x0;
    if (VEC) {
      const int x = 4 * lane;
      const int4* src = reinterpret_cast<const int4*>(g.dist + (size_t)max(slot, 0) * kBrickVox + 64 * plane) + (lane & 1);
      int4 v[8];
#pragma unroll
      for (int y = 0; y < 8; ++y) v[y] = slot >= 0 ? __ldg(src + 2 * y) : make_int4(g.INF, g.INF, g.INF, g.INF);
      if (x0 + x < g.nx) {
#pragma unroll
        for (int y = 0; y < 8; ++y)
          if (y < ny) __stcs(reinterpret_cast<int4*>(dst + (int64_t)y * g.nx + x), v[y]);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int x = 32 * q + lane;
        const int s = __shfl_sync(0xffffffffu, slot, 8 * q + 2 * (lane >> 3));  // brick 4 q + lane / 8
        const int32_t* src = g.dist + (size_t)max(s, 0) * kBrickVox + 64 * plane + (lane & 7);
        int v[8];
#pragma unroll
        for (int y = 0; y < 8; ++y) v[y] = s >= 0 ? __ldg(src + 8 * y) : g.INF;
        if (x0 + x < g.nx) {
#pragma unroll
          for (int y = 0; y < 8; ++y)
            if (y < ny) __stcs(dst + (int64_t)y * g.nx + x, v[y]);
        }
      }
    }
  }
}

// Fields narrower than a brick: a thread per voxel.  A warp per plane of a brick row would have 8 x nx outputs:
// 1 x 1024 x 1024 takes 25 us, 50 so; 7 x 1024 x 512 25 and 28; from a brick's width on the warp is faster (8 x 1024 x
// 1024: 53 and 47).
__global__ void __launch_bounds__(256) k_export_narrow(GridView g, int32_t* __restrict__ out) {
  pdl_enter();
  const int64_t total = (int64_t)g.nx * g.ny * g.nz;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = i / g.nx;
    out[i] = sqdist_at(g, (int)(i - r * g.nx), (int)(r % g.ny), (int)(r / g.ny));
  }
}

// A thread's last node lookup (key, node): the bricks of one query mostly fall in one interior node,
// so most lookups skip the hash table.
struct NodeCache {
  unsigned long long key = ~0ull;  // no node looked up yet
  int node = -1;
  // slot of brick (bx, by, bz) (inside the grid), or -1
  __device__ __forceinline__ int brick(const GridView& g, int bx, int by, int bz) {
    const unsigned long long k = node_key_of(g, bx, by, bz);
    if (k != key) {
      key = k;
      node = find_node(g, k);
    }
    return node < 0 ? -1 : g.child[(size_t)node * kNodeBricks + local_brick(bx, by, bz)];
  }
};

__device__ __forceinline__ bool occupied_at(const GridView& g, int x, int y, int z, NodeCache& nc) {
  const int s = nc.brick(g, x >> 3, y >> 3, z >> 3);
  return s >= 0 && ((g.occ[(size_t)s * 8 + (z & 7)] >> ((x & 7) + 8 * (y & 7))) & 1ull) != 0ull;
}

__device__ __forceinline__ int isqrt_floor(int v) {
  int r = (int)sqrtf((float)v);
  while (r * r > v) --r;
  while ((r + 1) * (r + 1) <= v) ++r;
  return r;
}

// Smallest position o of [c - isqrt(want), c + isqrt(want)] along y (AXIS 1, field g1) or z (AXIS 2,
// field g2) through (x, y, z) with field(o) = want - (o - c)^2, its value in `rest`; -1: none.  A
// brick's values in range are loaded together (planes 128 B apart: a sector each).
template <int AXIS>
__device__ __forceinline__ int line_match(const GridView& g, int x, int y, int z, int want, NodeCache& nc,
                                          int& rest) {
  const int c = AXIS == 1 ? y : z, n = AXIS == 1 ? g.ny : g.nz, r = isqrt_floor(want);
  const int b1 = min(c + r, n - 1) >> 3;
  for (int b = max(c - r, 0) >> 3; b <= b1; ++b) {
    const int s = AXIS == 1 ? nc.brick(g, x >> 3, b, z >> 3) : nc.brick(g, x >> 3, y >> 3, b);
    if (s < 0) continue;
    // g1 is stored x + 8 z + 64 y, g2 x + 8 y + 64 z
    const uint16_t* p = (AXIS == 1 ? g.g1 : g.g2) + (size_t)s * kBrickVox + (x & 7) + 8 * ((AXIS == 1 ? z : y) & 7);
    uint16_t v[8];
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = abs(8 * b + q - c) <= r ? __ldg(p + 64 * q) : (uint16_t)0xFFFFu;
    int at = -1;
#pragma unroll
    for (int q = 7; q >= 0; --q) {
      const int d = 8 * b + q - c, f = (int)v[q];
      if (f == want - d * d) {
        at = 8 * b + q;
        rest = f;
      }
    }
    if (at >= 0) return at;
  }
  return -1;
}

// Nearest occupied voxel of a query voxel; ties to the smallest (z, y, x), (-1, -1, -1) outside the
// grid or when D = dmax^2 (no obstacle closer than dmax).  The passes' own fields lead to it: D(v) is
// reached in the plane oz with g2(x, y, oz) = D - (oz - z)^2, that value on the row oy with
// g1(x, oy, oz) = g2 - (oy - y)^2, and g1 is the squared distance to the obstacle along x; the first
// match on each line is the smallest oz, then oy.  2 sqrt(D) + 1 reads a line instead of the
// O(D) rows of the lattice sphere |o - v|^2 = D.  Bound by the random sector reads (about 30 per
// query at dmax 32): 2^20 voxels of a 512 x 512 x 256 tunnel scene 0.18 ms = 5.8e9 queries/s (walking
// the sphere in (z, y, x) order and testing occupancy bits: 3.7 ms).
// Where every lane of a warp has an obstacle within one voxel on every axis (D <= 3; maps occupied to 30 % and
// more), the few rows of that sphere are walked: their occupancy bits mostly lie in the voxel's own brick, a sector
// or two against one per field value.  2^20 voxels of a 200^3 map occupied to 50 / 30 / 10 %, dmax 8: 32 / 43 / 59 us
// (along the fields 45 / 52 / 58; the walk in every lane with such a D costs 82 at 10 %).
constexpr int kNearD = 3;
__global__ void __launch_bounds__(128) k_query_nearest(GridView g, const int32_t* __restrict__ xyz, int64_t n,
                                                       int32_t* __restrict__ out) {
  pdl_enter();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const int x = xyz[3 * i] + g.off, y = xyz[3 * i + 1] + g.off, z = xyz[3 * i + 2] + g.off;
    int rx = -1 + g.off, ry = -1 + g.off, rz = -1 + g.off;
    if ((unsigned)x < (unsigned)g.nx && (unsigned)y < (unsigned)g.ny && (unsigned)z < (unsigned)g.nz) {
      NodeCache nc;
      const int s = nc.brick(g, x >> 3, y >> 3, z >> 3);
      const int D = s >= 0 ? g.dist[(size_t)s * kBrickVox + (x & 7) + 8 * (y & 7) + 64 * (z & 7)] : g.INF;
      const bool near = __all_sync(__activemask(), D <= kNearD || D >= g.INF);
      if ((unsigned)D < (unsigned)g.INF) {
        bool found = false;
        if (near) {
          // the sphere's points in (z, y, x) order, all within one voxel on every axis
          for (int r = 0; r < 9 && !found; ++r) {
            const int dz = r / 3 - 1, dy = r % 3 - 1, oz = z + dz, oy = y + dy;
            const int dx = D - dz * dz - dy * dy;  // 0 or 1: its own square
            if ((unsigned)dx > 1u || (unsigned)oy >= (unsigned)g.ny || (unsigned)oz >= (unsigned)g.nz) continue;
            int ox = x - dx;
            found = ox >= 0 && occupied_at(g, ox, oy, oz, nc);
            if (!found && dx) {
              ox = x + dx;
              found = ox < g.nx && occupied_at(g, ox, oy, oz, nc);
            }
            if (found) rx = ox, ry = oy, rz = oz;
          }
        } else {
          int plane = 0, dx2 = 0, oy = -1;
          const int oz = line_match<2>(g, x, y, z, D, nc, plane);
          if (oz >= 0) oy = line_match<1>(g, x, y, oz, plane, nc, dx2);
          if (oy >= 0) {
            const int dx = isqrt_floor(dx2);
            int ox = x - dx;
            found = ox >= 0 && occupied_at(g, ox, oy, oz, nc);
            if (!found) {
              ox = x + dx;
              found = ox < g.nx && occupied_at(g, ox, oy, oz, nc);
            }
            if (found) rx = ox, ry = oy, rz = oz;
          }
        }
        if (!found) set_error(g, kErrInternal);  // a finite D always has an obstacle at its distance
      }
    }
    out[3 * i] = rx - g.off;  // (-1, -1, -1) when there is none
    out[3 * i + 1] = ry - g.off;
    out[3 * i + 2] = rz - g.off;
  }
}

struct Corner8 {
  float d[8];  // index a + 2b + 4c for corner (i0+a, j0+b, k0+c)
};

// Corner distances (metres) of the cell holding u; returns the in-cell coordinates.
__device__ __forceinline__ void cell_of(const GridView& g, float vs, float px, float py, float pz, int& i0, int& j0,
                                        int& k0, float& tx, float& ty, float& tz) {
  float ux = px / vs, uy = py / vs, uz = pz / vs;
  float fx = floorf(ux), fy = floorf(uy), fz = floorf(uz);
  // cells in stored coordinates (shifted by g.off); t measured from the cell in caller coordinates
  const float o = (float)g.off;
  i0 = (int)fminf(fmaxf(fx + o, 0.f), (float)(g.nx - 2));
  j0 = (int)fminf(fmaxf(fy + o, 0.f), (float)(g.ny - 2));
  k0 = (int)fminf(fmaxf(fz + o, 0.f), (float)(g.nz - 2));
  tx = ux - (float)(i0 - g.off);
  ty = uy - (float)(j0 - g.off);
  tz = uz - (float)(k0 - g.off);
}

// Corner distances vs sqrt(D).  The cell's eight voxels lie in one brick, or in two, four or eight where it
// straddles brick faces: the bricks it touches (subsets of the axes it straddles) are looked up through
// one cached node, their child reads and then the eight values being independent loads.  (Looking each
// corner up by itself on the straddling third of the cells cost a warp eight chains of three dependent
// loads in a row: 2^20 points of 8,192 trajectories in a 512 x 512 x 256 tunnel scene now take 35 us for
// the cost, 28 for its gradient and 30 for distance and gradient, before 89, 59 and 63.)  Bound by the
// latency of that chain (point, hash slot, child, value).
__device__ __forceinline__ void corners(const GridView& g, float vs, int i0, int j0, int k0, Corner8& c) {
  const int bx = i0 >> 3, by = j0 >> 3, bz = k0 >> 3;
  const int across = ((i0 & 7) == 7 ? 1 : 0) | ((j0 & 7) == 7 ? 2 : 0) | ((k0 & 7) == 7 ? 4 : 0);
  NodeCache nc;
  int slot[8];
  slot[0] = nc.brick(g, bx, by, bz);
  const int32_t* child = g.child + (size_t)max(nc.node, 0) * kNodeBricks;
  // straddling a node face too: each brick through its own node
  const bool nodes = nc.node < 0 || ((across & 1) && (bx & 15) == 15) || ((across & 2) && (by & 15) == 15) ||
                     ((across & 4) && (bz & 15) == 15);
#pragma unroll
  for (int q = 1; q < 8; ++q) {
    slot[q] = -1;
    if ((q & ~across) == 0) {
      const int x = bx + (q & 1), y = by + ((q >> 1) & 1), z = bz + (q >> 2);
      slot[q] = nodes ? nc.brick(g, x, y, z) : child[local_brick(x, y, z)];
    }
  }
  int D[8];
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    int s = slot[0];
#pragma unroll
    for (int r = 1; r <= q; ++r)
      if (r == (q & across)) s = slot[r];
    const int a = q & 1, b = (q >> 1) & 1, e = q >> 2;
    D[q] = s >= 0 ? g.dist[(size_t)s * kBrickVox + ((i0 + a) & 7) + 8 * ((j0 + b) & 7) + 64 * ((k0 + e) & 7)] : g.INF;
  }
  // rounded by themselves: a difference of equal corners stays zero, which a product fused into it would not
#pragma unroll
  for (int q = 0; q < 8; ++q) c.d[q] = __fmul_rn(vs, sqrtf((float)D[q]));
}

__device__ __forceinline__ float trilinear(const Corner8& c, float tx, float ty, float tz) {
  float c00 = c.d[0] + tx * (c.d[1] - c.d[0]);
  float c10 = c.d[2] + tx * (c.d[3] - c.d[2]);
  float c01 = c.d[4] + tx * (c.d[5] - c.d[4]);
  float c11 = c.d[6] + tx * (c.d[7] - c.d[6]);
  float c0 = c00 + ty * (c10 - c00);
  float c1 = c01 + ty * (c11 - c01);
  return c0 + tz * (c1 - c0);
}

__global__ void k_clearance_fwd(GridView g, float vs, const float* __restrict__ pts, int64_t T, int64_t P, float tau,
                                float* __restrict__ cost) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t t = warp; t < T; t += nw) {
    float acc = 0.f;
    for (int64_t p = lane; p < P; p += 32) {
      const float* q = pts + (t * P + p) * 3;
      int i0, j0, k0;
      float tx, ty, tz;
      cell_of(g, vs, q[0], q[1], q[2], i0, j0, k0, tx, ty, tz);
      Corner8 c;
      corners(g, vs, i0, j0, k0, c);
      float d = trilinear(c, tx, ty, tz);
      float h = fmaxf(0.f, tau - d);
      acc += h * h;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    if (lane == 0) cost[t] = acc;
  }
}

__global__ void k_clearance_bwd(GridView g, float vs, const float* __restrict__ pts, int64_t T, int64_t P, float tau,
                                const float* __restrict__ gcost, float* __restrict__ gpts) {
  pdl_enter();
  const int64_t n = T * P;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float* q = pts + i * 3;
    int i0, j0, k0;
    float tx, ty, tz;
    cell_of(g, vs, q[0], q[1], q[2], i0, j0, k0, tx, ty, tz);
    Corner8 c;
    corners(g, vs, i0, j0, k0, c);
    float d = trilinear(c, tx, ty, tz);
    float h = fmaxf(0.f, tau - d);
    float go = gcost[i / P];
    float gx = 0.f, gy = 0.f, gz = 0.f;
    if (h > 0.f) {
      float wx[2] = {1.f - tx, tx}, wy[2] = {1.f - ty, ty}, wz[2] = {1.f - tz, tz};
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          gx += (c.d[1 + 2 * b + 4 * e] - c.d[2 * b + 4 * e]) * wy[b] * wz[e];
          gy += (c.d[2 + b + 4 * e] - c.d[b + 4 * e]) * wx[b] * wz[e];
          gz += (c.d[4 + b + 2 * e] - c.d[b + 2 * e]) * wx[b] * wy[e];
        }
      float s = -2.f * h / vs * go;
      gx *= s;
      gy *= s;
      gz *= s;
    }
    gpts[i * 3] = gx;
    gpts[i * 3 + 1] = gy;
    gpts[i * 3 + 2] = gz;
  }
}

// Distance and its gradient at points (planners): d = trilinear(vs sqrt(D)) as in the clearance
// cost, grad = (1 / vs) grad_t(trilinear), a thread per point.
__global__ void k_distance_at(GridView g, float vs, const float* __restrict__ pts, int64_t n, float* __restrict__ dist,
                              float* __restrict__ grad) {
  pdl_enter();
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float* q = pts + i * 3;
    int i0, j0, k0;
    float tx, ty, tz;
    cell_of(g, vs, q[0], q[1], q[2], i0, j0, k0, tx, ty, tz);
    Corner8 c;
    corners(g, vs, i0, j0, k0, c);
    dist[i] = trilinear(c, tx, ty, tz);
    if (grad) {
      float gx = 0.f, gy = 0.f, gz = 0.f;
      const float wx[2] = {1.f - tx, tx}, wy[2] = {1.f - ty, ty}, wz[2] = {1.f - tz, tz};
#pragma unroll
      for (int b = 0; b < 2; ++b)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          gx += (c.d[1 + 2 * b + 4 * e] - c.d[2 * b + 4 * e]) * wy[b] * wz[e];
          gy += (c.d[2 + b + 4 * e] - c.d[b + 4 * e]) * wx[b] * wz[e];
          gz += (c.d[4 + b + 2 * e] - c.d[b + 2 * e]) * wx[b] * wy[e];
        }
      grad[i * 3] = gx / vs;
      grad[i * 3 + 1] = gy / vs;
      grad[i * 3 + 2] = gz / vs;
    }
  }
}

unsigned grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  if (b < 1) b = 1;
  if (b > 152 * 32) b = 152 * 32;
  return (unsigned)b;
}

}  // namespace

cudaError_t launch_query(const GridView& g, const int32_t* xyz, int64_t n, int32_t* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_query, grid_for(n, 256), 256, 0, st, g, xyz, n, out);
  return cudaGetLastError();
}

cudaError_t launch_distance_at(const GridView& g, float vs, const float* pts, int64_t n, float* dist, float* grad,
                               cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_distance_at, grid_for(n, 256), 256, 0, st, g, vs, pts, n, dist, grad);
  return cudaGetLastError();
}

cudaError_t launch_query_nearest(const GridView& g, const int32_t* xyz, int64_t n, int32_t* out, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_query_nearest, grid_for(n, 128), 128, 0, st, g, xyz, n, out);
  return cudaGetLastError();
}

// Bricks holding an obstacle and bricks holding a finite D, counted on the device (counters
// C_OBST and C_FINITE, cleared by the caller): one atomic per warp and flag.
__global__ void k_count_flags(GridView g) {
  // counts kept per warp over the grid-stride loop, then one atomic per block and counter (the
  // two counters would otherwise take an atomic from every warp)
  __shared__ int wobst[32], wfin[32];
  const int nb = min(g.counters[C_NBRICKS], g.cap);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int obst = 0, fin = 0;
  for (int base = blockIdx.x * blockDim.x; base < nb; base += gridDim.x * blockDim.x) {
    const int s = base + threadIdx.x;
    const uint32_t f = s < nb ? g.bflags[s] : 0u;
    obst += __popc(__ballot_sync(0xffffffffu, (f & F_OBST) != 0u));
    fin += __popc(__ballot_sync(0xffffffffu, (f & F_FINITE) != 0u));
  }
  if (lane == 0) {
    wobst[warp] = obst;
    wfin[warp] = fin;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int to = 0, tf = 0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
      to += wobst[w];
      tf += wfin[w];
    }
    if (to) atomicAdd(&g.counters[C_OBST], to);
    if (tf) atomicAdd(&g.counters[C_FINITE], tf);
  }
}

cudaError_t launch_count_flags(const GridView& g, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(g.counters + C_FINITE, 0, 2 * sizeof(int32_t), st);  // C_FINITE, C_OBST
  if (e != cudaSuccess) return e;
  VDB_LAUNCH(k_count_flags, 304, 256, 0, st, g);
  return cudaGetLastError();
}

namespace {
// Occupancy of a z-range as packed records (x | y << 21 | (z + dz) << 42 | occ << 63): a warp per
// brick (stored bricks, or the bricks the last update changed), a lane per two voxel rows of one
// z-plane pair; records are appended with one atomic per warp per plane pair.  mode 0: occupied
// voxels only (occ = 1); mode 1: every voxel of the brick in the range, occupied or not.
__global__ void k_export_occupancy(GridView g, const int32_t* __restrict__ changed, int z_lo, int z_hi, int dz,
                                   int mode, unsigned long long* __restrict__ out, int64_t max_n,
                                   unsigned long long* __restrict__ count) {
  const int nb = mode == 0 ? min(g.counters[C_NBRICKS], g.cap) : min(g.counters[C_CHANGED], g.cap);
  const int lane = threadIdx.x & 31;
  const int nw = (int)gridDim.x * (int)(blockDim.x >> 5);
  for (int i = (int)blockIdx.x * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5); i < nb; i += nw) {
    const int slot = mode == 0 ? i : changed[i];
    const int4 c = g.bcoord[slot];
    const int bz0 = 8 * c.z;
    if (bz0 + 8 <= z_lo || bz0 >= z_hi) continue;  // warp-uniform
    for (int zz = 0; zz < 8; ++zz) {
      const int z = bz0 + zz;
      if (z < z_lo || z >= z_hi) continue;  // warp-uniform
      const unsigned long long word = g.occ[(size_t)slot * 8 + zz];  // bit x + 8 y
      // lane: bits 2 lane, 2 lane + 1 of the plane
      const int b0 = 2 * lane;
      const int e0 = (int)((word >> b0) & 1ull), e1 = (int)((word >> (b0 + 1)) & 1ull);
      // voxels of a brick that hangs over the grid's edge are not part of the grid
      const int y = 8 * c.y + (b0 >> 3), x0 = 8 * c.x + (b0 & 7);
      const bool in0 = x0 < g.nx && y < g.ny, in1 = x0 + 1 < g.nx && y < g.ny;
      const int k0 = (mode == 0 ? e0 : 1) & (int)in0, k1 = (mode == 0 ? e1 : 1) & (int)in1;
      const int mine = k0 + k1;
      int incl = mine;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += v;
      }
      const int total = __shfl_sync(0xffffffffu, incl, 31);
      if (total == 0) continue;
      unsigned long long base = 0;
      if (lane == 31) base = atomicAdd(count, (unsigned long long)total);
      base = __shfl_sync(0xffffffffu, base, 31);
      unsigned long long p = base + (unsigned long long)(incl - mine);
      for (int q = 0; q < 2; ++q) {
        if (!(q ? k1 : k0)) continue;
        if ((int64_t)p < max_n)
          out[p] = pack_rec(x0 + q, y, z + dz, q ? e1 : e0);
        ++p;
      }
    }
  }
}
}  // namespace

cudaError_t launch_export_occupancy(const GridView& g, const int32_t* changed, int z_lo, int z_hi, int dz, int mode,
                                    unsigned long long* out, int64_t max_n, unsigned long long* count,
                                    cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(count, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  VDB_LAUNCH(k_export_occupancy, 152 * 8, 256, 0, st, g, changed, z_lo, z_hi, dz, mode, out, max_n, count);
  return cudaGetLastError();
}

cudaError_t launch_export_dense(const GridView& g, int32_t* out, cudaStream_t st) {
  const bool narrow = g.nx < kBrick, vec = g.nx % 4 == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
  const unsigned blocks = grid_for(narrow ? (int64_t)g.nx * g.ny * g.nz : (int64_t)g.NX * g.BY * g.BZ * 8 * 32, 256);
  const auto kernel = narrow ? k_export_narrow : (vec ? k_export_dense<true> : k_export_dense<false>);
  // small fields are chained to the pass before (as the passes are); behind one that fills the GPU the blocks
  // that start early keep its shared-memory split, and a 1024 x 1024 x 256 field takes 0.09 ms longer
  if ((int64_t)g.BX * g.BY * g.BZ <= 16384)
    VDB_LAUNCH_PDL(kernel, blocks, 256, 0, st, g, out);
  else
    VDB_LAUNCH(kernel, blocks, 256, 0, st, g, out);
  return cudaGetLastError();
}

cudaError_t launch_clearance_fwd(const GridView& g, float vs, const float* pts, int64_t T, int64_t P, float tau,
                                 float* cost, cudaStream_t st) {
  if (T <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_clearance_fwd, grid_for(T * 32, 256), 256, 0, st, g, vs, pts, T, P, tau, cost);
  return cudaGetLastError();
}

cudaError_t launch_clearance_bwd(const GridView& g, float vs, const float* pts, int64_t T, int64_t P, float tau,
                                 const float* gcost, float* gpts, cudaStream_t st) {
  if (T <= 0 || P <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_clearance_bwd, grid_for(T * P, 256), 256, 0, st, g, vs, pts, T, P, tau, gcost, gpts);
  return cudaGetLastError();
}

}  // namespace vdbedt
