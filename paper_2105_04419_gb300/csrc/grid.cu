// Building and maintaining the sparse brick grid on the device.
//
//   ingest (global form)  staged occupancy records -> brick keys of "set" records -> unique list
//            (one flag per brick of the grid, compacted with one atomic per block, when records are
//            many or the grid mostly has storage; an LSD radix sort + unique + compaction for few
//            records on large sparse grids) -> nodes created first
//            (one thread per flagged node key) -> bricks allocated (slots reserved with one
//            atomic per block) -> occupancy bits set (OR-ed into a dense mask during the count, or
//            per record).  Several records for one voxel: the last one wins -- a per-voxel
//            last-record table (atomicMax of the record index) picks it whenever a record clears a
//            voxel.
//   ingest (incremental form)  the bricks of "set" records that are not stored yet are claimed
//            and allocated by one record each; every voxel's last record is applied through the
//            last-record table and each flip's brick joins the changed list once.
//   dense ingest  a whole occupancy grid -> per-brick masks in a scratch (sector-complete loads),
//            then nodes, then the occupied bricks.
//   activation  the compute set: every brick within Chebyshev brick radius R of a brick holding
//            an obstacle (the paper grows the tree only where the limited transform reaches,
//            Sec. IV-A): obstacle bits in per-node 4096-bit masks, halo nodes created, each node's
//            dilation computed from its 3 x 3 x 3 node neighbourhood, absent bricks allocated.
//   items    work lists for the passes: runs of bricks along x, y and z with their slot lists.
//   incremental marking  bricks whose occupancy changed -> their dilation (allocated) -> dirty
//            runs as bits per node: x within dmax along x, in-plane within dmax, z within dmax in space ->
//            work lists from the bits.
//   batches  the per-grid kernels take a view source: one grid, or every grid of a batch with
//            block shares of one launch.
#include "vdbedt_internal.cuh"

namespace vdbedt {

namespace {

constexpr int kT = 256;

// Grid of a grid-stride kernel over n items: enough blocks to fill the GPU a few times over.
inline unsigned blocks_for(int64_t n, int t = kT) {
  int64_t b = (n + t - 1) / t;
  if (b < 1) b = 1;
  if (b > 152 * 16) b = 152 * 16;
  return (unsigned)b;
}

inline int bits_for(uint64_t maxval) {
  int b = 1;
  while (b < 32 && (1ull << b) <= maxval) ++b;
  return b;
}

// View sources of the kernels that run once per grid.  get() returns the grid of the calling block
// and the block's index and count within that grid's share of the launch: a single grid (the view
// is a kernel parameter, the whole launch is its share), or every grid of a batch (views in device
// memory; grid i owns blocks first[i] .. first[i + 1] - 1 of a one-dimensional launch, shares sized
// to each grid's work, found by binary search).
struct OneView {
  GridView g;
  __device__ __forceinline__ GridView get(int& bid, int& nblk, int& grid) const {
    bid = blockIdx.x;
    nblk = gridDim.x;
    grid = 0;
    return g;
  }
  __device__ __forceinline__ bool skip(const GridView&) const { return false; }
};
struct BatchViews {
  const GridView* v;
  const int* first;  // [k + 1], first[k] = blocks of the launch
  int k;
  __device__ __forceinline__ GridView get(int& bid, int& nblk, int& grid) const {
    const int b = (int)blockIdx.x;
    int lo = 0, hi = k;  // first[lo] <= b < first[hi]
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (first[mid] <= b) lo = mid; else hi = mid;
    }
    bid = b - first[lo];
    nblk = first[lo + 1] - first[lo];
    grid = lo;
    return v[lo];
  }
  __device__ __forceinline__ bool skip(const GridView&) const { return false; }
};
// The global form's activation and work-list kernels run inside an incremental update only for
// grids whose update switched to the global form (counters[C_BIG] set after the records were
// applied): one grid (the whole launch is its share), or grid blockIdx.y of a batch.
// An update's choice between its incremental and its global form (the marking would cost (2R + 1)^3
// brick visits per changed brick; beyond kBigUpdate visits per stored brick the global form's
// activation and work lists are cheaper -- measured crossover on the tunnel scene).  Taken from the
// changed-brick count, final once the records are applied, and the stored bricks when the update
// began, so that every kernel of the update, on either stream and at any time, decides alike.
__device__ __forceinline__ bool big_update(const GridView& g) {
  const int64_t nc = min(g.counters[C_CHANGED], g.cap), side = 2 * g.R + 1;
  return nc * side * side * side > (int64_t)kBigUpdate * max(g.counters[C_NB_START], 1);
}

struct GatedOne {
  GridView g;
  __device__ __forceinline__ GridView get(int& bid, int& nblk, int& grid) const {
    bid = blockIdx.x;
    nblk = gridDim.x;
    grid = 0;
    return g;
  }
  __device__ __forceinline__ bool skip(const GridView& v) const { return !big_update(v); }
};
struct GatedBatch {
  const UpdArgs* a;
  __device__ __forceinline__ GridView get(int& bid, int& nblk, int& grid) const {
    bid = blockIdx.x;
    nblk = gridDim.x;
    grid = (int)blockIdx.y;
    return a[blockIdx.y].g;
  }
  __device__ __forceinline__ bool skip(const GridView& v) const { return !big_update(v); }
};
struct OneSrc {
  const uint8_t* p;
  __device__ __forceinline__ const uint8_t* get(int) const { return p; }
};
struct BatchSrc {
  const uint8_t* p[kBatchMax];
  __device__ __forceinline__ const uint8_t* get(int grid) const { return p[grid]; }
};
// Argument sources of the incremental update's kernels: one grid, or the grid blockIdx.y of a batch.
struct UpdOne {
  UpdArgs a;
  __device__ __forceinline__ UpdArgs get() const { return a; }
};
struct UpdBatch {
  const UpdArgs* a;
  __device__ __forceinline__ UpdArgs get() const { return a[blockIdx.y]; }
};

// ---- reset ----
// clear, clear_words: more words to set to zero (a dense ingest's node flags)
template <class VS>
__global__ void k_reset_nodes(VS vs, int32_t* __restrict__ clear, int64_t clear_words) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  (void)gi;
  // per used node: 4096 child slots, 128 dirty-run words, 128 activity words and 384 work words, all
  // whole 16-byte vectors (the per-node arrays start at multiples of their node strides)
  const int64_t nn = min(g.counters[C_NNODES], g.node_cap);
  const int64_t stride = (int64_t)nblk * blockDim.x, t0 = (int64_t)bid * blockDim.x + threadIdx.x;
  const int4 none = make_int4(kNoSlot, kNoSlot, kNoSlot, kNoSlot), zero = make_int4(0, 0, 0, 0);
  for (int64_t i = t0; i < nn * (kNodeBricks / 4); i += stride) reinterpret_cast<int4*>(g.child)[i] = none;
  for (int64_t i = t0; i < nn * (kMarkWords / 4); i += stride) reinterpret_cast<int4*>(g.mark)[i] = zero;
  for (int64_t i = t0; i < nn * (128 / 4); i += stride) reinterpret_cast<int4*>(g.amask)[i] = zero;
  for (int64_t i = t0; i < nn * (384 / 4); i += stride) reinterpret_cast<int4*>(g.mwork)[i] = zero;
  for (int64_t i = t0; i < nn * (128 / 4); i += stride) reinterpret_cast<int4*>(g.nclaim)[i] = zero;
  for (int64_t i = t0; i <= (int64_t)g.hmask; i += stride) g.hslots[i] = ~0ull;
  for (int64_t i = t0; i < clear_words; i += stride) clear[i] = 0;
}

// Start of an incremental update: clear the per-update counters and advance the update epoch
// (kept on the device, so that a captured update replays with a fresh epoch each time).  In a batch
// every grid's block clears the shared run counters (all store 0).
template <class US>
__global__ void k_begin_update(US us) {
  pdl_enter();
  if (threadIdx.x == 0 && blockIdx.x == 0) {
    const GridView g = us.get().g;
    g.items_ctr[0] = 0;
    g.items_ctr[1] = 0;
    g.items_ctr[2] = 0;
    g.counters[C_CHANGED] = 0;
    g.counters[C_FLIPS] = 0;
    g.counters[C_NEW_BRICKS] = 0;
    g.counters[C_UNIQUE] = 0;
    g.counters[C_HAS_ZERO] = 0;
    g.counters[C_XB] = 0;
    g.counters[C_YB] = 0;
    g.counters[C_ZB] = 0;
    g.counters[C_BIG] = 0;
    g.counters[C_DIRTY_NODES] = 0;
    g.counters[C_NB_START] = g.counters[C_NBRICKS];
    g.counters[C_EPOCH] += 1;
  }
}

// Batched form: the same, plus the record count of grids staged without a device count.
__global__ void k_begin_batch_update(const UpdArgs* __restrict__ args, BatchCounts counts) {
  pdl_enter();
  if (threadIdx.x == 0) {
    const int i = (int)blockIdx.y;
    const UpdArgs a = args[i];
    if (counts.c[i] >= 0) *const_cast<int32_t*>(a.n_dev) = counts.c[i];
    const GridView& g = a.g;
    g.items_ctr[0] = 0;
    g.items_ctr[1] = 0;
    g.items_ctr[2] = 0;
    g.counters[C_CHANGED] = 0;
    g.counters[C_FLIPS] = 0;
    g.counters[C_NEW_BRICKS] = 0;
    g.counters[C_UNIQUE] = 0;
    g.counters[C_HAS_ZERO] = 0;
    g.counters[C_XB] = 0;
    g.counters[C_YB] = 0;
    g.counters[C_ZB] = 0;
    g.counters[C_BIG] = 0;
    g.counters[C_DIRTY_NODES] = 0;
    g.counters[C_NB_START] = g.counters[C_NBRICKS];
    g.counters[C_EPOCH] += 1;
  }
}

// ---- brick allocation ----
// Coordinates and flags of a freshly allocated brick (no plane holds a value below dmax^2).  Its g1, g2 and D are
// written by the passes, and before an update's by init_new_fields.
__device__ __forceinline__ void init_brick_meta(const GridView& g, int slot, int node, int bx, int by, int bz) {
  g.bcoord[slot] = make_int4(bx, by, bz, node);
  g.bflags[slot] = 0u;
  g.bepoch[slot] = 0;
}

// dmax^2 twice, as g1 and g2 hold it
__device__ __forceinline__ uint32_t field_inf2(const GridView& g) { return (uint32_t)g.INF * 0x10001u; }

// g1, g2 and D of `slot` at dmax^2, written by a whole warp (every lane passes the same slot): each
// store instruction covers 512 contiguous bytes.
__device__ __forceinline__ void init_fields_warp(const GridView& g, int slot, int lane) {
  const uint32_t p = field_inf2(g);
  const uint4 v = make_uint4(p, p, p, p);
  uint4* d1 = reinterpret_cast<uint4*>(g.g1 + (size_t)slot * kBrickVox);
  uint4* d2 = reinterpret_cast<uint4*>(g.g2 + (size_t)slot * kBrickVox);
  d1[lane] = v;
  d1[lane + 32] = v;
  d2[lane] = v;
  d2[lane + 32] = v;
  int4* dd = reinterpret_cast<int4*>(g.dist + (size_t)slot * kBrickVox);
  const int4 w = make_int4(g.INF, g.INF, g.INF, g.INF);
#pragma unroll
  for (int q = 0; q < 4; ++q) dd[lane + 32 * q] = w;
}

// The same with an empty occupancy.
__device__ __forceinline__ void init_brick(const GridView& g, int slot, int node, int bx, int by, int bz) {
  ulonglong2* occ = reinterpret_cast<ulonglong2*>(g.occ + (size_t)slot * 8);
#pragma unroll
  for (int q = 0; q < 4; ++q) occ[q] = make_ulonglong2(0ull, 0ull);
  init_brick_meta(g, slot, node, bx, by, bz);
}

__device__ __forceinline__ bool brick_has_obstacle(const GridView& g, int s) {
  const ulonglong2* w = reinterpret_cast<const ulonglong2*>(g.occ + (size_t)s * 8);
  ulonglong2 a = w[0], b = w[1], c = w[2], d = w[3];
  return (a.x | a.y | b.x | b.y | c.x | c.y | d.x | d.y) != 0ull;
}

// ---- record ingest ----
__device__ __forceinline__ bool rec_valid(const GridView& g, int4 r) {
  return (unsigned)r.x < (unsigned)g.nx && (unsigned)r.y < (unsigned)g.ny && (unsigned)r.z < (unsigned)g.nz &&
         (unsigned)r.w <= 1u;
}

// Block-wide aggregation: every thread of the block calls it; returns base + the thread's rank
// among the threads with `pred` (-1 without), after one atomicAdd of the block's total on ctr.
__device__ int block_agg_add(int* ctr, bool pred, int* block_total) {
  __shared__ int wsum[32];
  __shared__ int base_sh, tot_sh;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (blockDim.x + 31) >> 5;
  const unsigned bal = __ballot_sync(0xffffffffu, pred);
  if (lane == 0) wsum[warp] = __popc(bal);
  __syncthreads();
  if (threadIdx.x == 0) {
    int t = 0;
    for (int w = 0; w < nw; ++w) {
      const int c = wsum[w];
      wsum[w] = t;
      t += c;
    }
    tot_sh = t;
    base_sh = t ? atomicAdd(ctr, t) : 0;
  }
  __syncthreads();
  const int r = pred ? base_sh + wsum[warp] + __popc(bal & ((1u << lane) - 1u)) : -1;
  if (block_total) *block_total = tot_sh;
  __syncthreads();
  return r;
}

// Number of staged records to apply: n, or the count in device memory (clamped to n) when the
// records were staged with a device-side count.
__device__ __forceinline__ int64_t rec_count(int64_t n, const int32_t* n_dev) {
  if (!n_dev) return n;
  const int64_t c = *n_dev;
  return c < 0 ? 0 : (c < n ? c : n);
}

// Grid-stride loops below keep every warp iterating together (the index base is block-uniform),
// so warp-wide votes and shuffles inside the loop see all 32 lanes.
#define GRID_STRIDE(i, n)                                                                              \
  for (int64_t i##_base = (int64_t)blockIdx.x * blockDim.x, i = i##_base + threadIdx.x; i##_base < (n); \
       i##_base += (int64_t)gridDim.x * blockDim.x, i = i##_base + threadIdx.x)

// Sets a flag word that only ever goes from 0 to 1, reading it first (L2): once one warp has set
// it the others find it set and issue no atomic on the shared word.
__device__ __forceinline__ void set_once(int32_t* flag) {
  if (!__ldcg(flag)) atomicOr(flag, 1);
}

// Places for the lanes with `want` in a list counted by *ctr: one atomic per warp (warp-uniform
// call); returns the lane's place (meaningful where want).
__device__ __forceinline__ int warp_reserve(int32_t* ctr, bool want) {
  const unsigned m = __ballot_sync(0xffffffffu, want);
  if (!m) return 0;
  const int lane = threadIdx.x & 31, leader = __ffs(m) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(ctr, __popc(m));
  base = __shfl_sync(0xffffffffu, base, leader);
  return base + __popc(m & ((1u << lane) - 1u));
}

__global__ void k_rec_brick_keys(GridView g, const rec_t* __restrict__ rec, int64_t n, const int32_t* n_dev,
                                 uint32_t* __restrict__ keys) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  const int64_t ne = rec_count(n, n_dev);  // keys past the count are the sentinel
  GRID_STRIDE(i, n) {
    uint32_t key = 0xFFFFFFFFu;
    bool zero = false, bad = false;
    if (i < ne) {
      int4 r = unpack_rec(rec[i]);
      if (!rec_valid(g, r)) {
        bad = true;
      } else if (r.w == 1) {
        key = (uint32_t)((r.x >> 3) + g.BX * ((r.y >> 3) + g.BY * (r.z >> 3)));
      } else {
        zero = true;
      }
    }
    // drop a key equal to the previous lane's (records of one brick tend to be adjacent)
    uint32_t prev = __shfl_up_sync(0xffffffffu, key, 1);
    if (lane > 0 && prev == key) key = 0xFFFFFFFFu;
    if (i < n) keys[i] = key;
    if (__any_sync(0xffffffffu, zero) && lane == 0) set_once(&g.counters[C_HAS_ZERO]);
    if (__any_sync(0xffffffffu, bad) && lane == 0) set_error(g, kErrInvalidRecord);
  }
}

// Many records: bucket the brick keys of "set" records through one flag per brick of the grid; the
// compaction of the flags is the unique key list; the node flags follow from the compacted bricks.
// With `dbits` (global form), the records' bits are also OR-ed into a dense mask of every brick of
// the grid (64 B per brick), so that allocation can copy each new brick's mask whole instead of a second pass
// over the records.
// A thread takes kMarkRecs consecutive records: neighbours along an x-row mostly share a mask word, whose bits
// it gathers in registers and ORs in with one atomic when the word changes; a brick's flag is only ever set,
// without reading it first, at the first word of it.  The brick
// masks' atomics and the flags bound it: 0.036 ms for the 8.4 million wall voxels of a 1024 x 1024 x 256 tunnel scene
// (four records a thread 0.038; a record a thread, merged over the warp by shuffles: 0.048, bound by issue).
template <bool DBITS>
__device__ __forceinline__ void mark_records(const GridView& g, const rec_t* __restrict__ rec, int64_t n,
                                             int32_t* __restrict__ flag, unsigned long long* __restrict__ dbits) {
  constexpr int kMarkRecs = 8;
  constexpr rec_t kWord = ~((7ull << 21) | 7ull);  // the bits of a record that tell its mask word (and its value)
  const bool vec = (reinterpret_cast<uintptr_t>(rec) & 15) == 0;
  bool zero = false, bad = false;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x * kMarkRecs;
  for (int64_t i = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * kMarkRecs; i < n; i += stride) {
    const int m = (int)min((int64_t)kMarkRecs, n - i);
    rec_t r[kMarkRecs];
    if (vec && m == kMarkRecs) {
      const ulonglong2* src = reinterpret_cast<const ulonglong2*>(rec + i);
#pragma unroll
      for (int k = 0; k < kMarkRecs; k += 2) {
        const ulonglong2 v = __ldg(src + k / 2);
        r[k] = v.x;
        r[k + 1] = v.y;
      }
    } else {
#pragma unroll
      for (int k = 0; k < kMarkRecs; ++k) r[k] = k < m ? __ldg(rec + i + k) : 0ull;
    }
    rec_t cur = 0ull;  // a record of the word being gathered (a "set" record has its top bit set)
    unsigned long long bits = 0ull;
    uint32_t flagged = 0xFFFFFFFFu;
    auto put = [&]() {
      const int4 c = unpack_rec(cur);
      const uint32_t lb = (uint32_t)(c.x >> 3) + (uint32_t)g.BX * ((uint32_t)(c.y >> 3) + (uint32_t)g.BY * (uint32_t)(c.z >> 3));
      if (lb != flagged) flag[lb] = 1;
      flagged = lb;
      if (DBITS) atomicOr(dbits + (size_t)lb * 8 + (c.z & 7), bits);
    };
#pragma unroll
    for (int k = 0; k < kMarkRecs; ++k) {
      if (k >= m) break;
      const int4 c = unpack_rec(r[k]);
      if (!rec_valid(g, c)) {
        bad = true;
      } else if (c.w == 0) {
        zero = true;
      } else {
        if (cur && ((cur ^ r[k]) & kWord)) {
          put();
          bits = 0ull;
        }
        cur = r[k];
        bits |= 1ull << ((c.x & 7) + 8 * (c.y & 7));
      }
    }
    if (cur) put();
  }
  const int lane = threadIdx.x & 31;
  if (__any_sync(0xffffffffu, zero) && lane == 0) set_once(&g.counters[C_HAS_ZERO]);
  if (__any_sync(0xffffffffu, bad) && lane == 0) set_error(g, kErrInvalidRecord);
}

__global__ void k_mark_record_bricks(GridView g, const rec_t* __restrict__ rec, int64_t n_max, const int32_t* n_dev,
                                     int32_t* __restrict__ flag, unsigned long long* __restrict__ dbits) {
  pdl_enter();
  const int64_t n = rec_count(n_max, n_dev);
  if (dbits) mark_records<true>(g, rec, n, flag, dbits);
  else mark_records<false>(g, rec, n, flag, dbits);
}

// A node absent from the table and inserted by exactly one thread, at index idx: its key, then a
// hash slot claimed with the final word (read by later kernels: the kernel boundary orders both).
__device__ void insert_new_node(const GridView& g, unsigned long long key, int idx) {
  if (idx >= g.node_cap) {
    set_error(g, kErrNodeOverflow);
    return;
  }
  g.node_key[idx] = (long long)key;
  const unsigned long long word = (key << kIndexBits) | (uint32_t)idx;
  uint32_t h = hash_key(key) & g.hmask;
  bool placed = false;
  for (uint32_t probe = 0; probe <= g.hmask && !placed; ++probe) {
    placed = atomicCAS(&g.hslots[h], kEmptySlot, word) == kEmptySlot;
    h = (h + 1) & g.hmask;
  }
  if (!placed) set_error(g, kErrNodeOverflow);
}

// Nodes of the obstacle bricks, created before the bricks so that no brick allocation waits on a
// node insertion in progress: one thread per flagged node key absent from the table; indices come
// from one atomic per block, and each key (inserted by exactly one thread) claims an empty hash
// slot with its final word.  Later kernels read the nodes (the kernel boundary orders them).
__device__ __forceinline__ void create_flagged_nodes(const GridView& g, int32_t* __restrict__ nflag, int64_t nkeys) {
  GRID_STRIDE(k, nkeys) {
    bool need = false;
    if (k < nkeys && nflag[k]) {
      nflag[k] = 0;
      need = find_node(g, (unsigned long long)k) < 0;
    }
    const int idx = block_agg_add(&g.counters[C_NNODES], need, nullptr);
    if (need) insert_new_node(g, (unsigned long long)k, idx);
  }
}

__global__ void k_create_flagged_nodes(GridView g, int32_t* __restrict__ nflag, int64_t nkeys) {
  pdl_enter();
  create_flagged_nodes(g, nflag, nkeys);
}

// Node flags of the unique brick keys (radix path).
__global__ void k_flag_key_nodes(GridView g, const uint32_t* __restrict__ uniq, int64_t n, int32_t* __restrict__ nflag) {
  pdl_enter();
  const int64_t cnt = min((int64_t)g.counters[C_UNIQUE], n);
  for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < cnt; j += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t lb = uniq[j];
    const int bx = (int)(lb % (uint32_t)g.BX), rest = (int)(lb / (uint32_t)g.BX);
    nflag[node_key_of(g, bx, rest % g.BY, rest / g.BY)] = 1;
  }
}

// Compaction of the flagged bricks, one atomic per block for the list positions (a block's bricks
// stay in key order, blocks follow in completion order; one counter word takes about a thousand
// atomics instead of one per warp holding a flagged brick), with the flags of their node keys:
// consecutive bricks mostly share a node, so only the first flagged lane of each run of one node
// key in the warp sets it (without reading it first).
__global__ void k_compact_flag_index(GridView g, const int32_t* __restrict__ flag, int64_t n,
                                     uint32_t* __restrict__ out, int32_t* __restrict__ nflag) {
  pdl_enter();
  const int lane = threadIdx.x & 31;
  GRID_STRIDE(i, n) {
    int nk = -1;
    if (i < n && flag[i]) {
      const uint32_t lb = (uint32_t)i, rest = lb / (uint32_t)g.BX;
      nk = (int)node_key_of(g, (int)(lb - rest * (uint32_t)g.BX), (int)(rest % (uint32_t)g.BY),
                            (int)(rest / (uint32_t)g.BY));
    }
    const unsigned set = __ballot_sync(0xffffffffu, nk >= 0);
    const int pos = block_agg_add(&g.counters[C_UNIQUE], nk >= 0, nullptr);  // block-uniform call
    const unsigned below = set & ((1u << lane) - 1u);
    if (nk >= 0) out[pos] = (uint32_t)i;
    const int prev_lane = 31 - __clz(below);  // previous flagged lane, or -1
    const int nk_prev = __shfl_sync(0xffffffffu, nk, prev_lane < 0 ? lane : prev_lane);
    if (nk >= 0 && (prev_lane < 0 || nk_prev != nk)) nflag[nk] = 1;
  }
}

__global__ void k_head_flags(const uint32_t* __restrict__ keys, int64_t n, uint32_t limit, int32_t* __restrict__ flag) {
  pdl_enter();
  GRID_STRIDE(i, n) {
    if (i < n) {
      uint32_t k = keys[i];
      flag[i] = (k < limit && (i == 0 || keys[i - 1] != k)) ? 1 : 0;
    }
  }
}

__global__ void k_compact_keys(const uint32_t* __restrict__ keys, const int32_t* __restrict__ flag,
                               const int32_t* __restrict__ pos, int64_t n, uint32_t* __restrict__ out) {
  pdl_enter();
  GRID_STRIDE(i, n) {
    if (i < n && flag[i]) out[pos[i]] = keys[i];
  }
}

// Bricks of the unique keys: node found or inserted, slot reserved with one atomic per block.
__global__ void k_alloc_obstacle_bricks(GridView g, const uint32_t* __restrict__ uniq, int64_t n,
                                        const unsigned long long* __restrict__ dbits) {
  pdl_enter();
  const int64_t cnt = min((int64_t)g.counters[C_UNIQUE], n);
  GRID_STRIDE(j, cnt) {
    int bx = 0, by = 0, bz = 0, node = -1;
    int* e = nullptr;
    bool need = false;
    ulonglong2 mask[4];  // the records' bits, loaded while the node is looked up
    if (j < cnt) {
      const uint32_t lb = uniq[j];
      if (dbits) {
        const ulonglong2* src = reinterpret_cast<const ulonglong2*>(dbits + (size_t)lb * 8);
#pragma unroll
        for (int q = 0; q < 4; ++q) mask[q] = src[q];
      }
      bx = (int)(lb % (uint32_t)g.BX);
      int rest = (int)(lb / (uint32_t)g.BX);
      by = rest % g.BY;
      bz = rest / g.BY;
      node = get_or_create_node(g, node_key_of(g, bx, by, bz));
      if (node >= 0) {
        e = &g.child[(size_t)node * kNodeBricks + local_brick(bx, by, bz)];
        need = *e == kNoSlot;
      }
    }
    int total = 0;
    const int slot = block_agg_add(&g.counters[C_NBRICKS], need, &total);
    if (need) {
      if (slot >= g.cap) {
        set_error(g, kErrOverflow);
      } else {
        if (dbits) {  // a new brick takes the records' mask as it is (the dense mask path is untracked)
          init_brick_meta(g, slot, node, bx, by, bz);
          ulonglong2* dst = reinterpret_cast<ulonglong2*>(g.occ + (size_t)slot * 8);
#pragma unroll
          for (int q = 0; q < 4; ++q) dst[q] = mask[q];
        } else {
          init_brick(g, slot, node, bx, by, bz);
        }
        *e = slot;
      }
    } else if (dbits && j < cnt && e) {  // a stored brick ORs the records' mask in
      const int sl = *e;
      if (sl >= 0 && sl < g.cap) {
        ulonglong2* dst = reinterpret_cast<ulonglong2*>(g.occ + (size_t)sl * 8);
        ulonglong2 old[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) old[q] = dst[q];
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = make_ulonglong2(mask[q].x | old[q].x, mask[q].y | old[q].y);
      }
    }
    if (threadIdx.x == 0 && total) atomicAdd(&g.counters[C_NEW_BRICKS], total);
  }
}

// All records set voxels: OR the bits in.  Adjacent lanes that hit the same 64-bit word (records
// of one x-row usually sit next to each other) are merged by a segmented OR over the warp, and the
// last lane of each segment issues the atomic.
__global__ void k_apply_set_only(GridView g, const rec_t* __restrict__ rec, int64_t n_max, const int32_t* n_dev) {
  pdl_enter();
  if (g.counters[C_HAS_ZERO]) return;
  const int lane = threadIdx.x & 31;
  const int64_t n = rec_count(n_max, n_dev);
  GRID_STRIDE(i, n) {
    unsigned long long word = 0ull;  // address of the target word, 0 for none
    unsigned long long bits = 0ull;
    if (i < n) {
      int4 r = unpack_rec(rec[i]);
      if (rec_valid(g, r) && r.w == 1) {
        int s = find_brick(g, r.x >> 3, r.y >> 3, r.z >> 3);
        if (s >= 0) {
          word = (unsigned long long)(&g.occ[(size_t)s * 8 + (r.z & 7)]);
          bits = 1ull << ((r.x & 7) + 8 * (r.y & 7));
        }
      }
    }
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long wp = __shfl_up_sync(0xffffffffu, word, o);
      const unsigned long long bp = __shfl_up_sync(0xffffffffu, bits, o);
      if (lane >= o && wp == word) bits |= bp;
    }
    const unsigned long long wn = __shfl_down_sync(0xffffffffu, word, 1);
    if (word && (lane == 31 || wn != word)) atomicOr(reinterpret_cast<unsigned long long*>(word), bits);
  }
}

// Tracked ingest (incremental form), first kernel: each record's brick slot for the ordered
// kernels (rslot).  A "set" record whose brick is not stored yet creates the brick's interior node
// when it is missing (inline, as the marking kernel does) and claims the brick with a per-node bit
// (`nclaim`, the amask layout); the claiming thread allocates the brick (slots reserved a warp at a
// time; its fields are set with the other new bricks', init_new_fields) and publishes its slot in the child
// table.
// Records that lose the claim, or read the child table before the claimer publishes, look the
// brick up again in the next kernel (rslot -2).  The claimer's record keeps -3 - slot, so that the
// next kernel, when no record of this ingest tests the bit any more, clears it: `nclaim` is zero
// between updates.  Records of stored bricks need no brick work at all.
template <class US>
__global__ void k_rec_slots(US us) {
  pdl_enter();
  const UpdArgs A = us.get();
  const GridView& g = A.g;
  const int lane = threadIdx.x & 31;
  const int64_t n = rec_count(A.n, A.n_dev);
  const rec_t* __restrict__ rec = A.rec;
  GRID_STRIDE(i, n) {  // block-uniform rounds: the warp-wide steps below see all 32 lanes
    bool zero = false, bad = false, claim = false;
    int rs = -1;  // the record's brick slot (-2: looked up once allocated)
    int node = -1, bx = 0, by = 0, bz = 0;
    if (i < n) {
      int4 r = unpack_rec(rec[i]);
      if (!rec_valid(g, r)) {
        bad = true;
      } else if (r.w == 1) {
        bx = r.x >> 3;
        by = r.y >> 3;
        bz = r.z >> 3;
        node = get_or_create_node(g, node_key_of(g, bx, by, bz));
        rs = -2;
        if (node >= 0) {
          const int l = local_brick(bx, by, bz);
          const int sl = g.child[(size_t)node * kNodeBricks + l];
          if (sl >= 0) {
            rs = sl;
          } else {
            const uint32_t b = 1u << (l & 31);
            claim = (atomicOr(&g.nclaim[(size_t)node * 128 + (l >> 5)], b) & b) == 0u;
          }
        }
      } else {
        zero = true;
        // a cleared voxel matters only in a stored brick: one stored now, or one a "set" record of
        // the same ingest adds (looked up again once it is published)
        rs = find_brick(g, r.x >> 3, r.y >> 3, r.z >> 3);
        if (rs < 0) rs = -2;
      }
    }
    const int slot = warp_reserve(&g.counters[C_NBRICKS], claim);
    const bool ok = claim && slot < g.cap;
    if (claim && !ok) {
      set_error(g, kErrOverflow);  // more bricks than the capacity holds: give the claim back
      const int l = local_brick(bx, by, bz);
      atomicAnd(&g.nclaim[(size_t)node * 128 + (l >> 5)], ~(1u << (l & 31)));
    }
    if (ok) {
      init_brick(g, slot, node, bx, by, bz);
      g.child[(size_t)node * kNodeBricks + local_brick(bx, by, bz)] = slot;
      rs = -3 - slot;
    }
    const unsigned made = __ballot_sync(0xffffffffu, ok);
    if (lane == 0 && made) atomicAdd(&g.counters[C_NEW_BRICKS], __popc(made));
    if (i < n) A.rslot[i] = rs;
    if (__any_sync(0xffffffffu, zero) && lane == 0) set_once(&g.counters[C_HAS_ZERO]);
    if (__any_sync(0xffffffffu, bad) && lane == 0) set_error(g, kErrInvalidRecord);
  }
}

// Ordered path: the last record of each voxel decides its bit.  vlast holds, per voxel of the
// pool (slot * 512 + voxel in brick), the highest index of a record for it (-1 when none): the
// first kernel raises it with atomicMax, the second applies each voxel's winning record and puts
// the entry back to -1, so vlast is all -1 between ingests.  Both run only when some record
// clears a voxel, or when flips are tracked.

// voxel index of a record inside its brick
__device__ __forceinline__ int rec_in_brick(rec_t packed) {
  const int4 r = unpack_rec(packed);
  return (r.x & 7) + 8 * (r.y & 7) + 64 * (r.z & 7);
}

__device__ __forceinline__ int64_t rec_voxel(const GridView& g, rec_t packed) {
  const int4 r = unpack_rec(packed);
  if (!rec_valid(g, r)) return -1;
  const int s = find_brick(g, r.x >> 3, r.y >> 3, r.z >> 3);
  if (s < 0) return -1;
  return (int64_t)s * 512 + ((r.x & 7) + 8 * (r.y & 7) + 64 * (r.z & 7));
}

// Flips are counted; with TRACK (an update) the brick is appended once per epoch to the changed list, and each
// record's brick slot comes from rslot.
template <bool TRACK>
__device__ __forceinline__ void apply_last(const GridView& g, const rec_t* __restrict__ rec, int64_t n_max,
                                           const int32_t* n_dev, int32_t* __restrict__ vlast,
                                           int32_t* __restrict__ changed, const int32_t* __restrict__ rslot) {
  const int64_t n = rec_count(n_max, n_dev);
  const int epoch = g.counters[C_EPOCH];
  GRID_STRIDE(j, n) {
    bool flip = false, first = false;
    int slot = 0;
    if (j < n) {
      const rec_t packed = rec[j];
      int64_t key;
      if (TRACK) {
        const int sl = rslot[j];
        key = sl >= 0 ? (int64_t)sl * 512 + rec_in_brick(packed) : -1;
      } else {
        key = rec_voxel(g, packed);
      }
      if (key >= 0 && vlast[key] == (int)j) {
        vlast[key] = -1;
        const int s = (int)(key >> 9), v = (int)(key & 511);
        const unsigned long long bit = 1ull << (v & 63);
        unsigned long long* word = &g.occ[(size_t)s * 8 + (v >> 6)];
        const bool cur = (*word & bit) != 0ull;
        if (cur != ((packed >> 63) != 0ull)) {
          atomicXor(word, bit);
          flip = true;
          first = TRACK && atomicExch(&g.bepoch[s], epoch) != epoch;
          slot = s;
          if (TRACK && g.ut_bits) {
            // untruncated grid (brick s at bx + BX (by + BY bz)): the voxel's x row is dirty
            const int64_t row = (int64_t)(s / g.BX) * 64 + (v >> 3);
            atomicOr(&g.ut_bits[row >> 5], 1u << (row & 31));
          }
        }
      }
    }
    // the changed list: each brick once per epoch, a block's bricks with one atomic (as the flip
    // count): the counter words see one atomic per block, not one per warp
    if (TRACK) {
      const int p = block_agg_add(&g.counters[C_CHANGED], first, nullptr);
      if (first) changed[p] = slot;
    }
    block_agg_add(&g.counters[C_FLIPS], flip, nullptr);
  }
}

__global__ void k_rec_last(GridView g, const rec_t* __restrict__ rec, int64_t n_max, const int32_t* n_dev,
                           int32_t* __restrict__ vlast) {
  pdl_enter();
  if (!g.counters[C_HAS_ZERO]) return;
  const int64_t n = rec_count(n_max, n_dev);
  GRID_STRIDE(i, n) {
    if (i < n) {
      const int64_t key = rec_voxel(g, rec[i]);
      if (key >= 0) atomicMax(&vlast[key], (int)i);
    }
  }
}

__global__ void k_apply_last(GridView g, const rec_t* __restrict__ rec, int64_t n_max, const int32_t* n_dev,
                             int32_t* __restrict__ vlast) {
  pdl_enter();
  if (!g.counters[C_HAS_ZERO]) return;
  apply_last<false>(g, rec, n_max, n_dev, vlast, nullptr, nullptr);
}

// The tracked forms (incremental update): every record, flips tracked, each record's brick slot
// taken from the first ingest kernel (looked up here only for bricks allocated since).
template <class US>
__global__ void k_upd_rec_last(US us) {
  pdl_enter();
  const UpdArgs A = us.get();
  const GridView& g = A.g;
  const int64_t n = rec_count(A.n, A.n_dev);
  GRID_STRIDE(i, n) {
    if (i < n) {
      const rec_t packed = A.rec[i];
      int s = A.rslot[i];
      if (s <= -3) {
        // the record that allocated its brick: the claim bit goes back to zero
        s = -3 - s;
        const int4 c = g.bcoord[s];
        const int l = local_brick(c.x, c.y, c.z);
        atomicAnd(&g.nclaim[(size_t)c.w * 128 + (l >> 5)], ~(1u << (l & 31)));
        A.rslot[i] = s;
      } else if (s == -2) {
        const int4 r = unpack_rec(packed);
        s = find_brick(g, r.x >> 3, r.y >> 3, r.z >> 3);
        A.rslot[i] = s;
      }
      if (s >= 0) atomicMax(&A.vlast[(int64_t)s * 512 + rec_in_brick(packed)], (int)i);
    }
  }
}

template <class US>
__global__ void k_upd_apply_last(US us) {
  pdl_enter();
  const UpdArgs A = us.get();
  apply_last<true>(A.g, A.rec, A.n, A.n_dev, A.vlast, A.changed, A.rslot);
}

// ---- dense ingest ----
// Two streaming passes.  (1) Masks: one warp per brick row (below) writes each brick's eight mask
// words into a plane-major scratch, with one flag per brick and one per node key.  (2) After the
// flagged nodes are created, one thread per brick of the grid allocates the occupied bricks (slots
// reserved with one atomic per block) and copies their masks in.  The grid was reset just before,
// so every brick is new; brick fields are left for the global transform that always follows a
// dense ingest.

// Bit i set when byte i of w is nonzero: the high bit of (low seven bits + 0x7F) | byte marks a
// nonzero byte, and one multiply gathers the four marks (bits 7, 15, 23, 31 land on 28 .. 31
// without overlapping any other partial product).
__device__ __forceinline__ uint32_t nonzero4(uint32_t w) {
  const uint32_t t = (((w & 0x7F7F7F7Fu) + 0x7F7F7F7Fu) | w) & 0x80808080u;
  return (t * 0x00204081u) >> 28;
}

// The aligned word at address w of the bytes [lo, hi) (its bytes outside them read as zero).
__device__ __forceinline__ uint32_t load_word(uintptr_t w, uintptr_t lo, uintptr_t hi) {
  if (w >= lo && w + 4 <= hi) return __ldg(reinterpret_cast<const uint32_t*>(w));
  uint32_t v = 0u;
  for (int k = 0; k < 4; ++k)
    if (w + k >= lo && w + k < hi) v |= (uint32_t)*reinterpret_cast<const uint8_t*>(w + k) << (8 * k);
  return v;
}

// Up to 16 voxels (nvx) of each of nr <= 8 rows at any alignment: bit x of m[y] set where byte x of row y is
// nonzero.  Five aligned words and a funnel shift a row, four rows' loads together (a byte at a time
// took 50 us of a 100 x 90 x 70 map's ingest).  Not inlined: its registers would cost the aligned forms theirs.
__device__ __noinline__ void ragged_rows(const uint8_t* rows, int pitch, int nr, int nvx, uintptr_t lo, uintptr_t hi,
                                         uint32_t* m) {
  if (pitch < kBrick) {
    // rows narrower than a brick: all of them are one stretch of at most 56 bytes, read as such (1 and 5 voxels
    // x 1024 x 512 in 40 and 51 us; row by row 80 and 86, a byte at a time 45 and 84)
    const uintptr_t at = reinterpret_cast<uintptr_t>(rows), end = at + nr * pitch;
    unsigned long long bits = 0ull;
#pragma unroll
    for (int q = 0; q < 15; ++q) {
      const uintptr_t w = (at & ~(uintptr_t)3) + 4 * q;
      if (w < end) bits |= (unsigned long long)nonzero4(load_word(w, lo, hi)) << (4 * q);
    }
    bits >>= at & 3;
    for (int r = 0; r < nr; ++r) m[r] = (uint32_t)(bits >> (r * pitch)) & ((1u << pitch) - 1u);
    return;
  }
  for (int h = 0; h < nr; h += 4) {
    uint32_t t[4][5], sh[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const uintptr_t at = reinterpret_cast<uintptr_t>(rows + (size_t)(h + r) * pitch);
      sh[r] = 8u * (uint32_t)(at & 3u);
#pragma unroll
      for (int q = 0; q < 5; ++q) {
        const uintptr_t w = (at & ~(uintptr_t)3) + 4 * q;
        t[r][q] = h + r < nr && w < at + nvx ? load_word(w, lo, hi) : 0u;
      }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      uint32_t v = 0u;
#pragma unroll
      for (int q = 0; q < 4; ++q) v |= nonzero4(__funnelshift_r(t[r][q], t[r][q + 1], sh[r])) << (4 * q);
      if (h + r < nr) m[h + r] = v & ((1u << nvx) - 1u);
    }
  }
}

// Scratch of the dense ingest: masks (8 words per brick of the grid, plane-major: plane z of brick
// lb at dbits[z * bricks + lb]), brick flags, node-key flags.
// A single grid's pointers are its own; grid i of a batch adds off[3i], off[3i + 1], off[3i + 2].
struct DenseScratch {
  unsigned long long* dbits;
  int32_t* flag;
  int32_t* nflag;
  const int64_t* off;  // nullptr for a single grid
  __device__ __forceinline__ void at(int gi, unsigned long long*& d, int32_t*& f, int32_t*& nf) const {
    d = dbits;
    f = flag;
    nf = nflag;
    if (off) {
      d += off[3 * gi];
      f += off[3 * gi + 1];
      nf += off[3 * gi + 2];
    }
  }
};

// Pass 1: one warp per unit (a brick row: by, bz and up to kDenseX bricks along x; in small grids one of its
// eight planes).  A plane's eight input rows are one contiguous stretch; each lane loads 16 bytes (two
// bricks) of each row, the eight loads issued together, and assembles both bricks' mask word
// of that plane in registers -- no shared memory, no block barrier -- and stores it to the
// plane-major scratch (a warp's stores are one contiguous run); where it holds a bit the lane sets the
// brick's flag and its node's (both cleared before).  With fewer than kDenseRows rows a warp per row leaves
// the GPU idle while each works through eight planes in turn, so they are spread over eight warps (a
// 64^3 map's masks 2.5 us, was 6.5); with more, a warp per plane repeats the row's bookkeeping
// eight times with half the loads in flight (16 maps of 293 M voxels 140 us, a warp per row 65); a batch's
// grids share the GPU and always take whole rows.  Around the line (whole ingest, planes spread / whole rows):
// 625 rows 17.6 / 17.8 us, 1,024 22.1 / 18.3, 1,444 28.3 / 21.6; of ragged rows, whose loads take longer, 625
// 22.5 / 38.7, 1,024 28.7 / 39.3, 1,444 35.9 / 45.5, 2,601 67.6 / 60.4.
constexpr int64_t kDenseRows = 1024;
constexpr int kDenseX = 64;
__host__ __device__ inline int64_t dense_rows(const GridView& g) {
  return (int64_t)((g.BX + kDenseX - 1) / kDenseX) * g.BY * g.BZ;
}
inline int dense_planes(const GridView& g) { return dense_rows(g) < kDenseRows ? 1 : 8; }  // of a unit

template <class VS, class SRC>
__global__ void __launch_bounds__(256, 4) k_dense_masks(VS vs, SRC src, DenseScratch ds, int planes, bool zero_counters) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (zero_counters && bid == 0 && (int)threadIdx.x < C_NUM) g.counters[threadIdx.x] = 0;
  const uint8_t* __restrict__ grid = src.get(gi);
  unsigned long long* dbits;
  int32_t* flag;
  int32_t* nflag;
  ds.at(gi, dbits, flag, nflag);
  const int64_t nbr = (int64_t)g.BX * g.BY * g.BZ;
  const uint32_t nch = (uint32_t)(g.BX + kDenseX - 1) / kDenseX;
  const int split = planes == 1 ? 3 : 0;
  const uint64_t nunits = (uint64_t)dense_rows(g) << split;
  const int lane = threadIdx.x & 31;
  const bool v16 = (g.nx % 16) == 0 && (reinterpret_cast<uintptr_t>(grid) & 15u) == 0;
  const bool v8 = (g.nx % 8) == 0 && (reinterpret_cast<uintptr_t>(grid) & 7u) == 0;
  const uintptr_t lo_end = reinterpret_cast<uintptr_t>(grid), hi_end = lo_end + (size_t)g.nx * g.ny * g.nz;
  const uint32_t nw = (uint32_t)nblk * (blockDim.x >> 5);
  for (uint64_t unit = (uint32_t)bid * (blockDim.x >> 5) + (threadIdx.x >> 5); unit < nunits; unit += nw) {
    const int z0 = (int)unit & ((1 << split) - 1);
    const uint32_t u = (uint32_t)(unit >> split);
    const int ch = (int)(u % nch);
    const uint32_t rest = u / nch;
    const int by = (int)(rest % (uint32_t)g.BY), bz = (int)(rest / (uint32_t)g.BY);
    const int bx0 = ch * kDenseX, nbx = min(kDenseX, g.BX - bx0);
    const int j = 2 * lane;  // this lane: bricks j and j + 1 of the chunk
    if (j >= nbx) continue;  // lanes past the row's end (the warp has no collective below)
    const bool two = j + 1 < nbx;
    const int x0 = (bx0 + j) * 8;
    const int nrow = min(8, g.ny - by * 8), nplane = min(8, g.nz - bz * 8);
    const uint8_t* base = grid + ((size_t)bz * 8 * g.ny + (size_t)by * 8) * g.nx + x0;
    const size_t zstride = (size_t)g.ny * g.nx;
    const int64_t lb = (bx0 + j) + (int64_t)g.BX * (by + (int64_t)g.BY * bz);
    bool any0 = false, any1 = false;
#pragma unroll 2
    for (int z = z0; z < z0 + planes; ++z) {
      const uint8_t* pl = base + (size_t)z * zstride;
      const int nr = z < nplane ? nrow : 0;
      uint32_t m[8];  // row y: bits 0-7 brick j, bits 8-15 brick j + 1
      if (v16) {  // nx a multiple of 16: bricks come in whole pairs
        uint4 w[8];
#pragma unroll
        for (int y = 0; y < 8; ++y)
          w[y] = y < nr ? __ldg(reinterpret_cast<const uint4*>(pl + (size_t)y * g.nx)) : make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
        for (int y = 0; y < 8; ++y)
          m[y] = nonzero4(w[y].x) | (nonzero4(w[y].y) << 4) | (nonzero4(w[y].z) << 8) | (nonzero4(w[y].w) << 12);
      } else if (v8) {
        uint2 lo[8], hi[8];
#pragma unroll
        for (int y = 0; y < 8; ++y) {
          lo[y] = y < nr ? __ldg(reinterpret_cast<const uint2*>(pl + (size_t)y * g.nx)) : make_uint2(0u, 0u);
          hi[y] = y < nr && two ? __ldg(reinterpret_cast<const uint2*>(pl + (size_t)y * g.nx + 8)) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int y = 0; y < 8; ++y)
          m[y] = nonzero4(lo[y].x) | (nonzero4(lo[y].y) << 4) | (nonzero4(hi[y].x) << 8) | (nonzero4(hi[y].y) << 12);
      } else {
        const int nvx = min(two ? 16 : 8, g.nx - x0);
#pragma unroll
        for (int y = 0; y < 8; ++y) m[y] = 0u;
        ragged_rows(pl, g.nx, nr, nvx, lo_end, hi_end, m);
      }
      unsigned long long a = 0ull, b = 0ull;
#pragma unroll
      for (int y = 0; y < 8; ++y) {
        a |= (unsigned long long)(m[y] & 0xffu) << (8 * y);
        b |= (unsigned long long)(m[y] >> 8) << (8 * y);
      }
      unsigned long long* plane = dbits + (size_t)z * nbr;
      plane[lb] = a;
      if (two) plane[lb + 1] = b;
      any0 |= a != 0ull;
      any1 |= two && b != 0ull;
    }
    const int bx = bx0 + j;
    if (any0) {
      flag[lb] = 1;
      nflag[node_key_of(g, bx, by, bz)] = 1;
    }
    if (any1) {
      flag[lb + 1] = 1;
      nflag[node_key_of(g, bx + 1, by, bz)] = 1;
    }
  }
}

// Nodes of flagged keys, one thread per key (each key inserted by exactly one thread; indices come
// from one atomic per block): no insertion ever waits on another.
template <class VS>
__global__ void __launch_bounds__(256) k_dense_nodes(VS vs, DenseScratch ds) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  unsigned long long* dbits;
  int32_t* flag;
  int32_t* nflag;
  ds.at(gi, dbits, flag, nflag);
  const int64_t nkeys = (int64_t)g.NX * g.NY * g.NZ;
  for (int64_t base = (int64_t)bid * blockDim.x; base < nkeys; base += (int64_t)nblk * blockDim.x) {
    const int64_t k = base + threadIdx.x;
    bool need = false;
    if (k < nkeys && nflag[k]) {
      nflag[k] = 0;
      need = find_node(g, (unsigned long long)k) < 0;
    }
    const int idx = block_agg_add(&g.counters[C_NNODES], need, nullptr);
    if (need) insert_new_node(g, (unsigned long long)k, idx);
  }
}

template <class VS>
__global__ void __launch_bounds__(256) k_dense_alloc(VS vs, DenseScratch ds) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  unsigned long long* dbits;
  int32_t* flag;
  int32_t* nflag;
  ds.at(gi, dbits, flag, nflag);
  const int64_t nbr = (int64_t)g.BX * g.BY * g.BZ;
  for (int64_t base = (int64_t)bid * blockDim.x; base < nbr; base += (int64_t)nblk * blockDim.x) {
    const int64_t lb = base + threadIdx.x;
    int node = -1, bx = 0, by = 0, bz = 0;
    if (lb < nbr && flag[lb]) {
      const uint32_t l = (uint32_t)lb, r = l / (uint32_t)g.BX;  // bricks < 2^32
      bx = (int)(l - r * (uint32_t)g.BX);
      by = (int)(r % (uint32_t)g.BY);
      bz = (int)(r / (uint32_t)g.BY);
      node = find_node(g, node_key_of(g, bx, by, bz));
    }
    int total = 0;
    const int slot = block_agg_add(&g.counters[C_NBRICKS], node >= 0, &total);
    if (node >= 0) {
      if (slot >= g.cap) {
        set_error(g, kErrOverflow);
      } else {
        init_brick_meta(g, slot, node, bx, by, bz);
        ulonglong2* dst = reinterpret_cast<ulonglong2*>(g.occ + (size_t)slot * 8);
#pragma unroll
        for (int q = 0; q < 4; ++q) dst[q] = make_ulonglong2(dbits[(2 * q) * nbr + lb], dbits[(2 * q + 1) * nbr + lb]);
        g.child[(size_t)node * kNodeBricks + local_brick(bx, by, bz)] = slot;
      }
    }
    if (threadIdx.x == 0 && total) atomicAdd(&g.counters[C_NEW_BRICKS], total);
  }
}

// ---- activation ----
// Compute set = bricks within Chebyshev brick radius R of an obstacle brick.  Global form: per-node
// 4096-bit masks, obstacle bits first, then a separable dilation (x, then y, then z), each stage a
// pure gather over neighbouring nodes' rows (no atomics).  A mask word holds two 16-brick x-rows:
// word (y >> 1) + 8 z, bits 16 (y & 1) + x.

template <class VS>
__global__ void k_obstacle_flags(VS vs) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (vs.skip(g)) return;
  (void)gi;
  const int nb = min(g.counters[C_NBRICKS], g.cap);
  for (int s = bid * blockDim.x + threadIdx.x; s < nb; s += nblk * blockDim.x) {
    bool obst = brick_has_obstacle(g, s);
    uint32_t f = g.bflags[s];
    g.bflags[s] = obst ? (f | F_OBST) : (f & ~F_OBST);
    if (obst) {
      int4 c = g.bcoord[s];
      int l = local_brick(c.x, c.y, c.z);
      atomicOr(&g.mwork[(size_t)c.w * 384 + (l >> 5)], 1u << (l & 31));
    }
  }
}

__device__ __forceinline__ uint32_t row16(const uint32_t* m, int y, int z) {
  return (m[(y >> 1) + 8 * z] >> (16 * (y & 1))) & 0xFFFFu;
}

// One warp per node holding obstacle bricks: create the neighbouring nodes that hold a brick within
// R bricks (Chebyshev) of one of its obstacle bricks, the only nodes its dilation reaches.  With
// R <= 16 the neighbours are the 26 adjacent nodes: neighbour (dx, dy, dz) is needed when one
// obstacle brick lies within R bricks of the side shared with it along every axis with a nonzero
// offset.  Each lane classifies 8 of the node's 256 brick rows and the warp ORs the 27-bit set of
// directions they reach.  (R > 16: every node within ceil(R / 16) nodes.)
template <class VS>
__global__ void k_node_halo(VS vs) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (vs.skip(g)) return;
  (void)gi;
  const int nn = min(g.counters[C_NNODES], g.node_cap);
  const int lane = threadIdx.x & 31;
  const int NR = (g.R + 15) / 16, side = 2 * NR + 1;
  for (int node = (bid * blockDim.x + threadIdx.x) >> 5; node < nn; node += (nblk * blockDim.x) >> 5) {
    const uint32_t* om = g.mwork + (size_t)node * 384;
    uint32_t any = om[lane] | om[lane + 32] | om[lane + 64] | om[lane + 96];
    if (!__any_sync(0xffffffffu, any != 0u)) continue;
    int nxn, nyn, nzn;
    node_coords(g, (unsigned long long)g.node_key[node], nxn, nyn, nzn);
    uint32_t dirs = 0xFFFFFFFFu;  // directions o = (dx + 1) + 3 (dy + 1) + 9 (dz + 1) to create
    if (NR == 1) {
      const uint32_t lo = g.R >= 16 ? 0xFFFFu : ((1u << g.R) - 1u), hi = (lo << (16 - g.R)) & 0xFFFFu;
      dirs = 0u;
      for (int r = lane; r < 256; r += 32) {
        const int yy = r & 15, zz = r >> 4;
        const uint32_t row = row16(om, yy, zz);
        if (!row) continue;
        // per axis, bit k: offset k - 1 reachable from this row's obstacle bricks
        const uint32_t ax = ((row & lo) ? 1u : 0u) | 2u | ((row & hi) ? 4u : 0u);
        const uint32_t ay = (yy < g.R ? 1u : 0u) | 2u | (yy >= 16 - g.R ? 4u : 0u);
        const uint32_t az = (zz < g.R ? 1u : 0u) | 2u | (zz >= 16 - g.R ? 4u : 0u);
        for (int kz = 0; kz < 3; ++kz)
          for (int ky = 0; ky < 3; ++ky)
            for (int kx = 0; kx < 3; ++kx)
              if ((az >> kz) & (ay >> ky) & (ax >> kx) & 1u) dirs |= 1u << (kx + 3 * (ky + 3 * kz));
      }
      dirs = __reduce_or_sync(0xffffffffu, dirs);
    }
    for (int o = lane; o < side * side * side; o += 32) {
      const int dx = o % side - NR, dy = (o / side) % side - NR, dz = o / (side * side) - NR;
      const int x = nxn + dx, y = nyn + dy, z = nzn + dz;
      if (x < 0 || y < 0 || z < 0 || x >= g.NX || y >= g.NY || z >= g.NZ || (dx == 0 && dy == 0 && dz == 0)) continue;
      if (NR > 1 || ((dirs >> o) & 1u)) get_or_create_node(g, node_key_at(g, x, y, z));
    }
  }
}


__device__ __forceinline__ int node_at(const GridView& g, int x, int y, int z) {
  if (x < 0 || y < 0 || z < 0 || x >= g.NX || y >= g.NY || z >= g.NZ) return -1;
  return find_node(g, node_key_at(g, x, y, z));
}

// Stage 0 -> 1: dilate each x-row by R across the neighbouring nodes along x.
// Stage 1 -> 2: OR of the rows y - R .. y + R; stage 2 -> amask: rows z - R .. z + R, then clipped
// to the grid.  One thread per (node, mask word), i.e. two rows.
template <int AXIS, class VS>
__global__ void k_dilate_stage(VS vs) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (vs.skip(g)) return;
  (void)gi;
  const int nn = min(g.counters[C_NNODES], g.node_cap);
  const int R = g.R;
  const int src_off = AXIS * 128;  // obstacle bits, then stage 1, then stage 2
  for (int64_t i = (int64_t)bid * blockDim.x + threadIdx.x; i < (int64_t)nn * 128;
       i += (int64_t)nblk * blockDim.x) {
    const int node = (int)(i >> 7), w = (int)(i & 127);
    int nxn, nyn, nzn;
    node_coords(g, (unsigned long long)g.node_key[node], nxn, nyn, nzn);
    const int z = w >> 3;
    uint32_t out = 0u;
    for (int half = 0; half < 2; ++half) {
      const int y = 2 * (w & 7) + half;
      uint32_t r = 0u;
      if (AXIS == 0) {
        // absolute brick x of bit j of chunk c: 16 (nxn + c) + j
        const int NR = (R + 15) / 16;
        for (int c = -NR; c <= NR; ++c) {
          int nb = c == 0 ? node : node_at(g, nxn + c, nyn, nzn);
          if (nb < 0) continue;
          uint32_t v = row16(g.mwork + (size_t)nb * 384 + src_off, y, z);
          if (!v) continue;
          for (int x = 0; x < 16; ++x) {
            int lo = x - R - 16 * c, hi = x + R - 16 * c;  // chunk-local bit range
            if (hi < 0 || lo > 15) continue;
            lo = max(lo, 0);
            hi = min(hi, 15);
            uint32_t msk = ((hi - lo == 31) ? 0xFFFFFFFFu : ((1u << (hi - lo + 1)) - 1u)) << lo;
            if (v & msk) r |= 1u << x;
          }
        }
      } else if (AXIS == 1) {
        for (int d = -R; d <= R; ++d) {
          int yy = y + d;
          int q = (yy >= 0) ? (yy >> 4) : -((15 - yy) >> 4);
          int nb = q == 0 ? node : node_at(g, nxn, nyn + q, nzn);
          if (nb < 0) continue;
          r |= row16(g.mwork + (size_t)nb * 384 + src_off, yy - 16 * q, z);
        }
      } else {
        for (int d = -R; d <= R; ++d) {
          int zz = z + d;
          int q = (zz >= 0) ? (zz >> 4) : -((15 - zz) >> 4);
          int nb = q == 0 ? node : node_at(g, nxn, nyn, nzn + q);
          if (nb < 0) continue;
          r |= row16(g.mwork + (size_t)nb * 384 + src_off, y, zz - 16 * q);
        }
        // clip to the grid
        const int gy = nyn * 16 + y, gz = nzn * 16 + z;
        if (gy >= g.BY || gz >= g.BZ) r = 0u;
        const int xs = g.BX - nxn * 16;
        if (xs < 16) r &= (xs <= 0) ? 0u : ((1u << xs) - 1u);
      }
      out |= r << (16 * half);
    }
    if (AXIS < 2)
      g.mwork[(size_t)node * 384 + (AXIS + 1) * 128 + w] = out;
    else
      g.amask[(size_t)node * 128 + w] = out;
  }
}

// The whole dilation of one node in one block (R <= 16, so the neighbourhood is the 3 x 3 x 3 nodes
// around it): the obstacle rows of the 3 x 3 node columns along y and z are dilated along x
// (48-bit rows across the three nodes along x), then along y, then along z, in shared memory, and
// the node's own 16 x 16 rows are clipped to the grid and written.  Replaces the three separable
// stage launches.
template <class VS>
__global__ void __launch_bounds__(256) k_dilate_nodes(VS vs) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (vs.skip(g)) return;
  (void)gi;
  __shared__ int nbr[27];
  __shared__ uint16_t X[48][48];  // [z' + 16][y' + 16]: rows dilated along x
  __shared__ uint16_t Y[48][16];  // [z' + 16][y]: then along y
  const int nn = min(g.counters[C_NNODES], g.node_cap);
  const int R = g.R;
  for (int node = bid; node < nn; node += nblk) {
    int nxn, nyn, nzn;
    node_coords(g, (unsigned long long)g.node_key[node], nxn, nyn, nzn);
    if (threadIdx.x < 27) {
      const int t = threadIdx.x, dx = t % 3 - 1, dy = (t / 3) % 3 - 1, dz = t / 9 - 1;
      nbr[t] = (dx | dy | dz) == 0 ? node : node_at(g, nxn + dx, nyn + dy, nzn + dz);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < 48 * 48; r += blockDim.x) {
      const int zq = r / 48 - 16, yq = r % 48 - 16;
      const int dy = yq < 0 ? -1 : (yq >= 16 ? 1 : 0), dz = zq < 0 ? -1 : (zq >= 16 ? 1 : 0);
      const int y = yq - 16 * dy, z = zq - 16 * dz;
      unsigned long long w = 0ull;
#pragma unroll
      for (int dx = -1; dx <= 1; ++dx) {
        const int nb = nbr[(dx + 1) + 3 * ((dy + 1) + 3 * (dz + 1))];
        if (nb >= 0) w |= (unsigned long long)row16(g.mwork + (size_t)nb * 384, y, z) << (16 * (dx + 1));
      }
      unsigned long long d = w;
      for (int sft = 1; sft <= R; ++sft) d |= (w << sft) | (w >> sft);
      X[zq + 16][yq + 16] = (uint16_t)(d >> 16);
    }
    __syncthreads();
    for (int r = threadIdx.x; r < 48 * 16; r += blockDim.x) {
      const int zi = r / 16, y = r % 16;
      uint32_t o = 0u;
      for (int d = -R; d <= R; ++d) o |= X[zi][y + d + 16];
      Y[zi][y] = (uint16_t)o;
    }
    __syncthreads();
    if (threadIdx.x < 128) {
      const int w = threadIdx.x, z = w >> 3;
      uint32_t out = 0u;
      for (int half = 0; half < 2; ++half) {
        const int y = 2 * (w & 7) + half;
        uint32_t r = 0u;
        for (int d = -R; d <= R; ++d) r |= Y[z + d + 16][y];
        const int gy = nyn * 16 + y, gz = nzn * 16 + z;
        if (gy >= g.BY || gz >= g.BZ) r = 0u;
        const int xs = g.BX - nxn * 16;
        if (xs < 16) r &= (xs <= 0) ? 0u : ((1u << xs) - 1u);
        out |= r << (16 * half);
      }
      g.amask[(size_t)node * 128 + w] = out;
    }
    __syncthreads();
  }
}

// Places for `cnt` items of each lane in a list counted by *ctr: one atomic per warp (warp-uniform
// call); returns the lane's first place.  *total receives the warp's sum.
__device__ __forceinline__ int warp_reserve_count(int32_t* ctr, int cnt, int* total) {
  const int lane = threadIdx.x & 31;
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  *total = __shfl_sync(0xffffffffu, incl, 31);
  int base = 0;
  if (lane == 31 && *total) base = atomicAdd(ctr, *total);
  return __shfl_sync(0xffffffffu, base, 31) + incl - cnt;
}

// Storage for the bricks of a row segment whose compute-set bits (`bits` of amask word `word` of
// `node`; bit b is the brick at x = x16 + (b & 15) of row (y, z)) this thread set first, so that
// exactly one thread handles each: the ones without storage get slots (places reserved a warp at
// a time; warp-uniform call) and their metadata from the thread; their fields are set afterwards with all
// new bricks' (init_new_fields).
__device__ void alloc_new_bits(const GridView& g, int node, int word, uint32_t bits, int x16, int y, int z) {
  uint32_t need = 0u;
  if (node >= 0 && bits) {
    // the row's 16 child slots, loaded together
    const int half = bits > 0xFFFFu ? 16 : 0;
    const int4* row = reinterpret_cast<const int4*>(g.child + (size_t)node * kNodeBricks + word * 32 + half);
    int4 c[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) c[q] = row[q];
#pragma unroll
    for (int q = 0; q < 4; ++q)
      need |= ((uint32_t)(c[q].x == kNoSlot) | (uint32_t)(c[q].y == kNoSlot) << 1 | (uint32_t)(c[q].z == kNoSlot) << 2 |
               (uint32_t)(c[q].w == kNoSlot) << 3) << (4 * q + half);
    need &= bits;
  }
  const int cnt = __popc(need);
  int total = 0;
  const int base = warp_reserve_count(&g.counters[C_NBRICKS], cnt, &total);
  if ((threadIdx.x & 31) == 31 && total) atomicAdd(&g.counters[C_NEW_BRICKS], total);
  int k = 0;
  for (uint32_t b = need; b; b &= b - 1u, ++k) {
    const int bit = __ffs(b) - 1, slot = base + k;
    if (slot >= g.cap) {
      set_error(g, kErrOverflow);
      continue;
    }
    init_brick(g, slot, node, x16 + (bit & 15), y, z);
    g.child[(size_t)node * kNodeBricks + word * 32 + bit] = slot;
  }
}

// Allocate every marked brick without storage: a block per (node, 256-brick chunk), a brick per
// thread, one atomic per block for the slot range (block scan of the flags).  It is the last to run before
// the work lists and after the dilation, so it also puts the obstacle masks back to zero (they are zero
// whenever an activation begins) and, in the global form, the work lists' counters.
template <class VS>
__global__ void __launch_bounds__(256) k_alloc_marked(VS vs, bool zero_items) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (vs.skip(g)) return;
  (void)gi;
  const int nn = min(g.counters[C_NNODES], g.node_cap);
  if (zero_items && bid == 0 && threadIdx.x < 3) g.items_ctr[threadIdx.x] = 0;
  for (int b = bid; b < nn * 16; b += nblk) {
    const int node = b >> 4, l = (b & 15) * 256 + threadIdx.x;
    if (threadIdx.x < 8) g.mwork[(size_t)node * 384 + (b & 15) * 8 + threadIdx.x] = 0u;
    const bool need = ((g.amask[(size_t)node * 128 + (l >> 5)] >> (l & 31)) & 1u) &&
                      g.child[(size_t)node * kNodeBricks + l] == kNoSlot;
    int total = 0;
    const int slot = block_agg_add(&g.counters[C_NBRICKS], need, &total);
    if (threadIdx.x == 0 && total) atomicAdd(&g.counters[C_NEW_BRICKS], total);
    if (need) {
      if (slot >= g.cap) {
        set_error(g, kErrOverflow);
      } else {
        int nxn, nyn, nzn;
        node_coords(g, (unsigned long long)g.node_key[node], nxn, nyn, nzn);
        init_brick(g, slot, node, nxn * 16 + (l & 15), nyn * 16 + ((l >> 4) & 15), nzn * 16 + (l >> 8));
        g.child[(size_t)node * kNodeBricks + l] = slot;
      }
    }
  }
}

// ---- work items ----
// An update's dirty runs: per node 32 words for each axis (z, y and x runs; word 8 q + line / 32, q the run
// along the axis, line = o1 + 16 o2 over the two axes across it, as k_items_nodes numbers them), then the
// epoch of the node's last entry in the list of nodes with such bits, which follows the nodes' words.  The
// words are zero between updates: the kernel that queues the runs clears them.
__device__ __forceinline__ uint32_t* dirty_words(const GridView& g, int node, int axis, int q) {
  return g.mark + (size_t)node * kMarkWords + axis * 32 + q * 8;
}
__device__ __forceinline__ int32_t* dirty_nodes(const GridView& g) {
  return reinterpret_cast<int32_t*>(g.mark + (size_t)g.node_cap * kMarkWords);
}
// Bits into a word; the ones that were not there yet.  Read first: most of them were set by earlier marks,
// and the exchanges of all changed bricks around a word queue up on it (a lidar frame's marking 14 us on the
// critical path, 10 with the read).
__device__ __forceinline__ uint32_t or_bits(uint32_t* w, uint32_t bits) {
  return bits & ~__ldcg(w) ? bits & ~atomicOr(w, bits) : 0u;
}
// Node into the list once per epoch (a plain read first: most nodes are already there).
__device__ __forceinline__ void list_dirty_node(const GridView& g, int node, uint32_t epoch) {
  uint32_t* e = g.mark + (size_t)node * kMarkWords + 96;
  if (__ldcg(e) == epoch || atomicExch(e, epoch) == epoch) return;
  dirty_nodes(g)[atomicAdd(&g.counters[C_DIRTY_NODES], 1)] = node;
}

// Voxel gap between two bricks d apart along an axis: the nearest voxels of bricks 0 and d are
// 8 |d| - 7 apart (0 for the same brick).
__device__ __forceinline__ int brick_gap(int d) {
  d = abs(d);
  return d == 0 ? 0 : 8 * d - 7;
}
// largest |d| along an axis with brick_gap(d)^2 < rem (rem >= 1, below 2^24: the root is exact)
__device__ __forceinline__ int gap_reach(int rem) { return ((int)__fsqrt_rn((float)(rem - 1)) + 7) >> 3; }

// Bricks of changed brick c's cube (R bricks around it inside the grid) and its marking units: one per
// (z run, row), one per y run, one for the x runs.
struct DirtyCube {
  int x0, x1, y0, y1, z0, z1, nyr, nz, units;
  __device__ __forceinline__ DirtyCube(const GridView& g, const int4& c, int ry, int rz) {
    const int R = g.R;
    x0 = max(c.x - R, 0), x1 = min(c.x + R, g.BX - 1);
    y0 = max(c.y - R, 0), y1 = min(c.y + R, g.BY - 1);
    z0 = max(c.z - R, 0), z1 = min(c.z + R, g.BZ - 1);
    nyr = y1 - y0 + 1;
    nz = (z1 >> (__ffs(rz) - 1)) - (z0 >> (__ffs(rz) - 1)) + 1;  // runs are 4, 8 or 16
    units = nz * nyr + ((y1 >> (__ffs(ry) - 1)) - (y0 >> (__ffs(ry) - 1)) + 1) + 1;
  }
};

// Unit u of changed brick c: the bits of the runs along one axis in one row along x (along x itself: of c's
// x runs).  node(bx, by, bz): the node of a brick, -1 for none (then nothing is stored there).
template <class Node>
__device__ __forceinline__ void mark_dirty(const GridView& g, const int4& c, const DirtyCube& k, int u, int rx, int ry,
                                           int rz, Node node) {
  const int nzu = k.nz * k.nyr;
  if (u == k.units - 1) {  // x runs of c's row
    const int m = gap_reach(g.INF), xa = max(k.x0, c.x - m), xe = min(k.x1, c.x + m);
    const int line = (c.y & 15) + 16 * (c.z & 15);
    for (int x = xa & ~(rx - 1); x <= xe; x += rx) {
      const int n = node(x, c.y, c.z);
      if (n >= 0) atomicOr(dirty_words(g, n, 0, (x & 15) >> (__ffs(rx) - 1)) + (line >> 5), 1u << (line & 31));
    }
    return;
  }
  const bool z = u < nzu;
  const int run = z ? rz : ry, lo = z ? k.z0 : k.y0, hi = z ? k.z1 : k.y1, at = z ? c.z : c.y;
  const int r = (lo & ~(run - 1)) + (z ? u / k.nyr : u - nzu) * run;  // the run's first brick along the axis
  const int s = max(r, lo), e = min(r + run - 1, hi);
  const int by = z ? k.y0 + u % k.nyr : s, bz = z ? s : c.z;
  // its nearest brick's gap along the axis, and the row's gap across it (y runs: in c's layer)
  const int ga = brick_gap(at < s ? s - at : (at > e ? at - e : 0)), gr = z ? brick_gap(by - c.y) : 0;
  const int rem = g.INF - ga * ga - gr * gr;
  if (rem <= 0) return;
  const int m = gap_reach(rem), xe = min(k.x1, c.x + m), o2 = (z ? by : bz) & 15;
  for (int x = max(k.x0, c.x - m); x <= xe;) {  // node by node
    const int xl = min(xe, x | 15), n = node(x, by, bz);
    if (n >= 0)
      or_bits(dirty_words(g, n, z ? 2 : 1, (r & 15) >> (__ffs(run) - 1)) + (o2 >> 1),
              (((1u << (xl - x + 1)) - 1u) << (x & 15)) << (16 * (o2 & 1)));
    x = xl + 1;
  }
}

// The runs of a node along one axis: queued where they hold a stored brick (DIRTY: and their dirty bit is set,
// which is cleared here).  The block's 256 threads cover the 16 x 16 lines of the node across the axis, qrun is
// the run along it.  A thread reads its line's child entries, the run's and (NBQ > 0: 4 NBQ >= run + 2 R
// slots) its halo's of R bricks on both sides, which reach at most the neighbouring node each way
// (R <= 6 < 16); a block-wide scan compacts the runs, one atomic reserves their places, and each thread
// stores its slot list as vectors.  Bound by the chain of dependent reads: those of the node itself are
// issued before the neighbours are known and counted, the neighbours' while the places are reserved
// (19 us for the 300,000 runs of a 1024 x 1024 x 256 tunnel scene, 21 with a line along x read entry by entry; with
// the slots read again from the compacted queue, one per thread, that scene's call took 7 us more, a batch of
// 16 maps with its update 26 us more).
template <bool DIRTY, int NBQ>
__device__ __forceinline__ void node_runs(const GridView& g, int gi, int node, int axis, int qrun, int run, const Items& it) {
  __shared__ int wsum[8];
  __shared__ int base_sh;
  __shared__ int nbr_sh[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int R = NBQ ? g.R : 0;
  bool dirty = true;
  if (DIRTY) {
    uint32_t* w = dirty_words(g, node, axis, qrun) + warp;
    const uint32_t bits = *w;
    dirty = (bits >> lane & 1u) != 0u;
    if (!__syncthreads_or(dirty)) return;
    if (lane == 0 && bits) *w = 0u;
  }
  int q[3];
  node_coords(g, (unsigned long long)g.node_key[node], q[0], q[1], q[2]);
  const int a1 = axis == 0 ? 1 : 0, a2 = axis == 2 ? 1 : 2;
  const int r0 = qrun * run, nb = run + 2 * R;
  const int o1 = threadIdx.x & 15, o2 = threadIdx.x >> 4;
  const int across = (o1 << (4 * a1)) | (o2 << (4 * a2));
  // child entries along the line, c[j + sh] the one of brick r0 - R + j; first those of this node.  A line along
  // x is contiguous: read as vectors, from the last multiple of 4 bricks on (which no node boundary splits).
  constexpr int N = NBQ ? 4 * NBQ : 16;
  const int sh = NBQ && axis == 0 ? (r0 - R) & 3 : 0, x0 = r0 - R - sh;
  int c[N + 4];
#pragma unroll
  for (int j = 0; j < N + 4; ++j) c[j] = -1;
  auto quad = [&](int j, int n) {
    const int4 v = *reinterpret_cast<const int4*>(g.child + (size_t)n * kNodeBricks + (across | ((x0 + j) & 15)));
    c[j] = v.x, c[j + 1] = v.y, c[j + 2] = v.z, c[j + 3] = v.w;
  };
  if (NBQ && axis == 0) {
#pragma unroll
    for (int j = 0; j < N + 4; j += 4)
      if (dirty && j < nb + sh && (unsigned)(x0 + j) < 16u) quad(j, node);
  } else {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int x = r0 + j - R;
      if (dirty && j < nb && (unsigned)x < 16u) c[j] = g.child[(size_t)node * kNodeBricks + (across | (x << (4 * axis)))];
    }
  }
  if (NBQ && threadIdx.x >= 254) {
    int qq[3] = {q[0], q[1], q[2]};
    qq[axis] += threadIdx.x == 254 ? -1 : 1;
    int n2 = -1;
    if (qq[0] >= 0 && qq[1] >= 0 && qq[2] >= 0 && qq[0] < g.NX && qq[1] < g.NY && qq[2] < g.NZ)
      n2 = find_node(g, node_key_at(g, qq[0], qq[1], qq[2]));
    nbr_sh[threadIdx.x - 254] = n2;
  }
  bool any = false;
#pragma unroll
  for (int j = 0; j < N + 4; ++j) any |= j >= R + sh && j < R + sh + run && c[j] >= 0;
  const unsigned bal = __ballot_sync(0xffffffffu, any);
  if (lane == 0) wsum[warp] = __popc(bal);
  __syncthreads();
  if (threadIdx.x == 0) {
    int tot = 0;
    for (int w = 0; w < 8; ++w) {
      const int t = wsum[w];
      wsum[w] = tot;
      tot += t;
    }
    base_sh = tot ? atomicAdd(&g.items_ctr[axis], tot) : 0;
  }
  if (NBQ && any && axis == 0) {
#pragma unroll
    for (int j = 0; j < N + 4; j += 4) {
      const int x = x0 + j;
      if (j < nb + sh && (unsigned)x >= 16u) {
        const int src = nbr_sh[x < 0 ? 0 : 1];
        if (src >= 0) quad(j, src);
      }
    }
  } else if (NBQ && any) {
#pragma unroll
    for (int j = 0; j < N; ++j) {
      const int x = r0 + j - R;
      if (j < nb && (unsigned)x >= 16u) {
        const int src = nbr_sh[x < 0 ? 0 : 1];
        if (src >= 0) c[j] = g.child[(size_t)src * kNodeBricks + (across | ((x & 15) << (4 * axis)))];
      }
    }
  }
  __syncthreads();
  const int p = base_sh + wsum[warp] + __popc(bal & ((1u << lane) - 1u));
  if (any && p < g.item_cap) {
    int l0[3];
    l0[axis] = r0;
    l0[a1] = o1;
    l0[a2] = o2;
    it.run[axis][p] = pack_brick(q[0] * 16 + l0[0], q[1] * 16 + l0[1], q[2] * 16 + l0[2]);
    if (it.igrid[axis]) it.igrid[axis][p] = gi;
    int4* slots = reinterpret_cast<int4*>(it.slots[axis] + (size_t)p * kItemSlots);
    auto pool = [&](int j) {
      const int s = sh & 2 ? (sh & 1 ? c[j + 3] : c[j + 2]) : (sh & 1 ? c[j + 1] : c[j]);
      return s >= 0 ? s + g.slot_base : -1;
    };
#pragma unroll
    for (int v = 0; v < NBQ; ++v) slots[v] = make_int4(pool(4 * v), pool(4 * v + 1), pool(4 * v + 2), pool(4 * v + 3));
  }
  __syncthreads();  // wsum, base_sh and nbr_sh are free again
}

// The form of node_runs for runs of this length (without slot lists: the envelope form, any R).
template <bool DIRTY>
__device__ __forceinline__ void node_runs_of(const GridView& g, int gi, int node, int axis, int qrun, int run, const Items& it,
                                             bool with_slots) {
  const int nb = run + 2 * g.R;
  if (!with_slots) node_runs<DIRTY, 0>(g, gi, node, axis, qrun, run, it);
  else if (nb <= 12) node_runs<DIRTY, 3>(g, gi, node, axis, qrun, run, it);
  else if (nb <= 16) node_runs<DIRTY, 4>(g, gi, node, axis, qrun, run, it);
  else node_runs<DIRTY, 7>(g, gi, node, axis, qrun, run, it);
}

// Global form: every run that holds a stored brick, found node by node.  Block = (node, axis, run
// index along the axis).
template <class VS>
__global__ void __launch_bounds__(256) k_items_nodes(VS vs, int rx, int ry, int rz, Items it, bool with_slots) {
  pdl_enter();
  int bid, nblk, gi;
  const GridView g = vs.get(bid, nblk, gi);
  if (vs.skip(g)) return;
  const int nn = min(g.counters[C_NNODES], g.node_cap);
  for (int b = bid; b < nn * 12; b += nblk) {
    const int axis = (b % 12) / 4, qrun = b % 4;
    const int run = axis == 0 ? rx : (axis == 1 ? ry : rz);
    if (qrun >= 16 / run) continue;  // block-uniform
    node_runs_of<false>(g, gi, b / 12, axis, qrun, run, it, with_slots);
  }
}

// Fields of the bricks that the running update stored (slots from its start's count on) at dmax^2: a
// brick per warp, streaming.  Done here, by the whole GPU at once, rather than where each brick is
// allocated: the few blocks of the marking that meet the frontier of the stored bricks allocate hundreds each
// (a lidar frame's marking took 44 us on average with it, 20 without).
__device__ __forceinline__ void init_new_fields(const GridView& g, int block, int nblocks) {
  const int end = min(g.counters[C_NBRICKS], g.cap), nw = nblocks * (int)(blockDim.x >> 5);
  for (int slot = g.counters[C_NB_START] + block * (int)(blockDim.x >> 5) + (int)(threadIdx.x >> 5); slot < end; slot += nw)
    init_fields_warp(g, slot, threadIdx.x & 31);
}

// An update's work lists, from the dirty bits of its listed nodes (blockIdx.z 0), and beside them the fields of
// the bricks that it stored (1).  The global form's lists come from k_items_nodes, and its passes write every
// field.  A run is queued by one block, so no run is claimed and no slot list is built from a queue:
// claiming each run with an exchange while marking and reading slot lists back from the queue took 20 + 17 us
// of a lidar frame on average.
template <class US>
__global__ void __launch_bounds__(256) k_items_dirty(US us, int rx, int ry, int rz, Items it, bool with_slots) {
  pdl_enter();
  const UpdArgs A = us.get();
  const GridView& g = A.g;
  if (big_update(g)) return;
  if (blockIdx.z == 1) {
    init_new_fields(g, (int)blockIdx.x, (int)gridDim.x);
    return;
  }
  const int nn = min(g.counters[C_DIRTY_NODES], g.node_cap);
  for (int b = (int)blockIdx.x; b < nn * 12; b += (int)gridDim.x) {
    const int axis = (b % 12) / 4, qrun = b % 4;
    const int run = axis == 0 ? rx : (axis == 1 ? ry : rz);
    if (qrun >= 16 / run) continue;  // block-uniform
    node_runs_of<true>(g, (int)blockIdx.y, dirty_nodes(g)[b / 12], axis, qrun, run, it, with_slots);
  }
}

// Update statistics only (launched when they are asked for): the stored bricks each pass
// recomputes, i.e. the own entries (R .. R + run - 1) of every run's slot list that hold a slot,
// added to the counters of the run's grid (views == nullptr: every run is grid `one`'s).
// blockIdx.y = axis, a thread per run.
__global__ void k_count_run_bricks(const GridView* __restrict__ views, GridView one, const int32_t* __restrict__ items_ctr,
                                   int item_cap, int rx, int ry, int rz, Items it) {
  const int axis = (int)blockIdx.y;
  const int run = axis == 0 ? rx : (axis == 1 ? ry : rz);
  const int n = min(items_ctr[axis], item_cap);
  for (int item = (int)(blockIdx.x * blockDim.x + threadIdx.x); item < n; item += (int)(gridDim.x * blockDim.x)) {
    const int32_t* sl = it.slots[axis] + (size_t)item * kItemSlots + one.R;
    int own = 0;
    for (int j = 0; j < run; ++j) own += sl[j] >= 0;
    int32_t* ctr = views ? views[it.igrid[axis][item]].counters : one.counters;
    if (own) atomicAdd(&ctr[C_XB + axis], own);
  }
}

// ---- incremental ----
// For every changed brick c: refresh its obstacle flag; if it holds obstacles, mark its dilation
// (the bricks within R that must be stored); and mark its dirty runs.
// Dirty sets: D(v) depends only on obstacles closer than dmax (Eq. 1 with the truncation), so a
// flip in c can change D only in bricks whose nearest voxels lie closer than dmax to c's -- the
// ball of radius dmax around c at brick granularity, about half the cube of R bricks.  Such a brick
// needs its z pass if it is stored or about to be (every brick of the cube of an obstacle-holding
// c is: the dilation just marked it, and the allocation of the marked bricks runs before the
// passes).  The in-plane values g2 change only in c's z layer, within dmax in the plane (a disk):
// those bricks also need the in-plane pass; the x-line values g1 change only in c's x row: those
// bricks also need the x pass.
// Dirty runs are bits per node, OR-ed a row along x at a time (one unit of mark_dirty: for dmax 32 and runs
// of 4, 32 to 41 per changed brick; no value comes back, nothing is waited for), and queued node by node
// by k_items_dirty.  Runs are aligned to their length (4, 8 or 16) inside nodes, hence at multiples of it in
// grid coordinates.
// With at most two changed bricks per block, a block per changed brick: its first threads find
// (or, for an obstacle-holding c, create) the interior nodes c's cube spans (at most 4 per axis:
// 2R + 1 <= 47 bricks), then a thread per row (y, z) of the cube sets the row's x extent in the
// allocation masks, beside a thread per unit.  With more changed bricks
// per block (a batch's share of the launch, a large update), a thread per (changed brick, row) and
// then per (changed brick, unit), each with its own node lookups, keeps every thread
// of the GPU busy instead.
template <class US>
__global__ void __launch_bounds__(256, 6) k_changed_mark(US us, int rx, int ry, int rz) {
  pdl_enter();
  __shared__ int nodes[64];
  __shared__ int obst_sh;
  const UpdArgs A = us.get();
  const GridView& g = A.g;
  const int32_t* __restrict__ changed = A.changed;
  const int nc = min(g.counters[C_CHANGED], g.cap);
  const int R = g.R, side = 2 * R + 1;
  // an update that takes the global form leaves all this to the gated kernels of the side stream
  if (big_update(g)) {
    if (blockIdx.x == 0 && threadIdx.x == 0) g.counters[C_BIG] = 1;
    return;
  }
  const uint32_t epoch = (uint32_t)g.counters[C_EPOCH];
  if (nc > 2 * (int)gridDim.x) {
    // dilation: a thread per (changed brick, row), the rounds block-uniform
    const int rows = side * side, nseg = (side + 15) / 16 + 1;
    for (int64_t base = (int64_t)blockIdx.x * blockDim.x; base < (int64_t)nc * rows;
         base += (int64_t)gridDim.x * blockDim.x) {
      const int64_t i = base + threadIdx.x;
      int s = -1, r = 0;
      bool obst = false;
      if (i < (int64_t)nc * rows) {
        s = changed[i / rows];
        r = (int)(i % rows);
        obst = brick_has_obstacle(g, s);
        if (r == 0) {
          const uint32_t f = g.bflags[s];
          g.bflags[s] = obst ? (f | F_OBST) : (f & ~F_OBST);
        }
      }
      int4 c = make_int4(0, 0, 0, 0);
      if (obst) c = g.bcoord[s];
      const int y = c.y + r % side - R, z = c.z + r / side - R;
      const bool live = obst && (unsigned)y < (unsigned)g.BY && (unsigned)z < (unsigned)g.BZ;
      const int x0 = max(c.x - R, 0), x1 = min(c.x + R, g.BX - 1);
      const int ly = y & 15, lz = z & 15, word = (ly >> 1) + 8 * lz;
      int xa = x0;
      for (int k = 0; k < nseg; ++k) {  // the row's segments, one node each (same count on every lane)
        uint32_t added = 0u;
        int node = -1;
        const int x16 = xa & ~15;
        if (live && xa <= x1) {
          const int xe = min(x1, xa | 15);
          node = get_or_create_node(g, node_key_of(g, xa, y, z));
          if (node >= 0) {
            const uint32_t bitsx = ((1u << ((xe & 15) - (xa & 15) + 1)) - 1u) << (xa & 15);
            const uint32_t add = bitsx << (16 * (ly & 1));
            added = or_bits(&g.amask[(size_t)node * 128 + word], add);
          }
          xa = xe + 1;
        }
        alloc_new_bits(g, node, word, added, x16, y, z);
      }
    }
    // dirty runs: a thread per (changed brick, unit)
    const int umax = side * (side / rz + 2) + side / ry + 3;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)nc * umax;
         i += (int64_t)gridDim.x * blockDim.x) {
      const int s = changed[i / umax], u = (int)(i % umax);
      const int4 c = g.bcoord[s];
      const DirtyCube k(g, c, ry, rz);
      if (u >= k.units) continue;
      const bool obst = brick_has_obstacle(g, s);
      mark_dirty(g, c, k, u, rx, ry, rz, [&](int bx, int by, int bz) {
        const unsigned long long key = node_key_of(g, bx, by, bz);
        const int n = obst ? get_or_create_node(g, key) : find_node(g, key);
        if (n >= 0) list_dirty_node(g, n, epoch);
        return n;
      });
    }
    return;
  }
  for (int i = (int)blockIdx.x; i < nc; i += (int)gridDim.x) {
    const int s = changed[i];
    __syncthreads();  // the table of the block's previous brick is no longer read
    const int4 c = g.bcoord[s];
    const DirtyCube k(g, c, ry, rz);
    const int x0 = k.x0, x1 = k.x1, y0 = k.y0, y1 = k.y1, z0 = k.z0, z1 = k.z1;
    const int qx0 = x0 >> 4, qy0 = y0 >> 4, qz0 = z0 >> 4;
    const int nqx = (x1 >> 4) - qx0 + 1, nqy = (y1 >> 4) - qy0 + 1, nqz = (z1 >> 4) - qz0 + 1;
    const int nq = nqx * nqy * nqz;  // at most 4^3
    // at once: the brick's obstacle bit (lanes 0-7 of warp 0, a mask word each) and the lookups of
    // the nodes its cube spans (threads 32 .. 32 + nq - 1); nodes an obstacle brick's dilation
    // needs and that do not exist yet are created after the barrier
    if (threadIdx.x < 8) {
      const bool any = __any_sync(0xffu, g.occ[(size_t)s * 8 + threadIdx.x] != 0ull);
      if (threadIdx.x == 0) {
        const uint32_t f = g.bflags[s];
        g.bflags[s] = any ? (f | F_OBST) : (f & ~F_OBST);
        obst_sh = any;
      }
    } else if ((int)threadIdx.x >= 32 && (int)threadIdx.x < 32 + nq) {
      const int q = (int)threadIdx.x - 32;
      nodes[q] = find_node(g, node_key_at(g, qx0 + q % nqx, qy0 + (q / nqx) % nqy, qz0 + q / (nqx * nqy)));
    }
    __syncthreads();
    const bool obst = obst_sh != 0;  // block-uniform
    if (obst) {
      if ((int)threadIdx.x < nq && nodes[threadIdx.x] < 0) {
        const int q = (int)threadIdx.x;
        nodes[q] = get_or_create_node(g, node_key_at(g, qx0 + q % nqx, qy0 + (q / nqx) % nqy, qz0 + q / (nqx * nqy)));
      }
      __syncthreads();
    }
    if (obst) {
      // dilation: a row's x extent is split at node boundaries (the same segments on every lane);
      // the rounds are block-uniform so that new bricks' slots are reserved a warp at a time
      const int nyr = y1 - y0 + 1, rows = nyr * (z1 - z0 + 1);
      for (int rb = 0; rb < rows; rb += (int)blockDim.x) {
        const int r = rb + (int)threadIdx.x;
        const bool live = r < rows;
        const int y = y0 + (live ? r % nyr : 0), z = z0 + (live ? r / nyr : 0);
        const int ly = y & 15, lz = z & 15, word = (ly >> 1) + 8 * lz;
        const int nrow = nqx * (((y >> 4) - qy0) + nqy * ((z >> 4) - qz0));
        for (int xa = x0; xa <= x1;) {
          const int xe = min(x1, xa | 15);
          const int node = live ? nodes[nrow + (xa >> 4) - qx0] : -1;
          uint32_t added = 0u;
          if (node >= 0) {
            const uint32_t bitsx = ((1u << ((xe & 15) - (xa & 15) + 1)) - 1u) << (xa & 15);
            const uint32_t add = bitsx << (16 * (ly & 1));
            added = or_bits(&g.amask[(size_t)node * 128 + word], add);
          }
          alloc_new_bits(g, node, word, added, xa & ~15, y, z);
          xa = xe + 1;
        }
      }
    }
    // dirty runs: the units on other warps than the first rows of the dilation, and the nodes into the list
    if (threadIdx.x >= 192 && (int)threadIdx.x - 192 < nq && nodes[threadIdx.x - 192] >= 0)
      list_dirty_node(g, nodes[threadIdx.x - 192], epoch);
    for (int u = (int)((threadIdx.x + 160) & 255); u < k.units; u += 256)
      mark_dirty(g, c, k, u, rx, ry, rz, [&](int bx, int by, int bz) {
        return nodes[((bx >> 4) - qx0) + nqx * (((by >> 4) - qy0) + nqy * ((bz >> 4) - qz0))];
      });
  }
}

// The incremental update's kernels for one grid or all grids of a batch (k = gridDim.y).
template <class US>
cudaError_t update_ingest_kernels(US us, int k, int64_t n, cudaStream_t st) {
  const int div = k > 1 ? k : 1;
  auto bx = [&](int64_t work, int hi) {
    int64_t b = (work + kT - 1) / kT;
    const int64_t lim = k > 1 ? (hi / div > 16 ? hi / div : 16) : hi;
    return (unsigned)(b < 1 ? 1 : (b > lim ? lim : b));
  };
  const dim3 gr(bx(n, 152 * 16), k);
  VDB_LAUNCH_PDL(k_rec_slots<US>, gr, kT, 0, st, us);
  VDB_LAUNCH_PDL(k_upd_rec_last<US>, gr, kT, 0, st, us);
  VDB_LAUNCH_PDL(k_upd_apply_last<US>, gr, kT, 0, st, us);
  return cudaGetLastError();
}

template <class US, class GV>
cudaError_t update_mark_kernels(US us, GV gv, int k, int node_cap, int R, bool with_slots, const Tuning& t,
                                const Items& it, const Fork& fk, cudaStream_t st) {
  const unsigned div = k > 1 ? (unsigned)k : 1u;
  auto share = [&](unsigned single) { return k > 1 ? (single / div > 16 ? single / div : 16u) : single; };
  const unsigned nc = (unsigned)node_cap;
  cudaError_t e = cudaSuccess;
  cudaStream_t gs = st;
  if (fk.side) {
    e = cudaEventRecord(fk.fork, st);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(fk.side, fk.fork, 0);
    if (e != cudaSuccess) return e;
    gs = fk.side;
  }
  // global form, for the grids whose update takes it (each kernel decides for itself; the others'
  // blocks return at once, and the kernels stride over their work, so a launch of at most two
  // blocks per SM keeps that cheap), on the side stream from the end of the ingest on, beside the
  // incremental marking
  auto gated = [&](unsigned single) { return share(single < 304u ? single : 304u); };
  VDB_LAUNCH(k_obstacle_flags<GV>, dim3(gated(1024), k), kT, 0, gs, gv);
  VDB_LAUNCH_PDL(k_node_halo<GV>, dim3(gated(64), k), kT, 0, gs, gv);
  if (R <= 16) {
    VDB_LAUNCH_PDL(k_dilate_nodes<GV>, dim3(gated(nc < 1024 ? nc : 1024u), k), 256, 0, gs, gv);
  } else {
    VDB_LAUNCH_PDL((k_dilate_stage<0, GV>), dim3(gated(256), k), kT, 0, gs, gv);
    VDB_LAUNCH_PDL((k_dilate_stage<1, GV>), dim3(gated(256), k), kT, 0, gs, gv);
    VDB_LAUNCH_PDL((k_dilate_stage<2, GV>), dim3(gated(256), k), kT, 0, gs, gv);
  }
  VDB_LAUNCH_PDL(k_alloc_marked<GV>, dim3(gated(nc * 16 < 8192 ? nc * 16 : 8192u), k), kT, 0, gs, gv, false);
  VDB_LAUNCH_PDL(k_items_nodes<GV>, dim3(gated(nc * 12 < 8192 ? nc * 12 : 8192u), k), kT, 0, gs, gv, t.run[0], t.run[1],
             t.run[2], it, with_slots);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  if (fk.side) {
    e = cudaEventRecord(fk.join, fk.side);
    if (e != cudaSuccess) return e;
  }
  // incremental form, for the others: the changed bricks' flags, their dilation (with storage for
  // the bricks it adds) and their dirty runs
  VDB_LAUNCH_PDL(k_changed_mark<US>, dim3(share(2432), k), kT, 0, st, us, t.run[0], t.run[1], t.run[2]);
  return cudaGetLastError();
}

}  // namespace

cudaError_t ensure_scratch(Scratch& s, size_t bytes) {
  if (s.bytes >= bytes) return cudaSuccess;
  if (s.buf) cudaFree(s.buf);
  s.buf = nullptr;
  s.bytes = 0;
  size_t want = bytes + bytes / 4 + 4096;
  cudaError_t e = cudaMalloc(&s.buf, want);
  if (e != cudaSuccess) return e;
  s.bytes = want;
  return cudaSuccess;
}

cudaError_t launch_reset(const GridView& g, cudaStream_t st) {
  VDB_LAUNCH_PDL(k_reset_nodes<OneView>, 1024, kT, 0, st, OneView{g}, (int32_t*)nullptr, (int64_t)0);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return cudaMemsetAsync(g.counters, 0, sizeof(int32_t) * C_NUM, st);
}

static size_t align_up(size_t v) { return (v + 255) & ~(size_t)255; }

// Apply staged records.  Bricks of "set" records are found or created through a counting sort over
// one flag per brick of the grid (many records, or a grid that mostly has storage), or a stable radix sort of brick keys, a unique pass
// and a compaction (few records).  Bits: in the global form, when every record sets a voxel, the
// records' bits go to the bricks directly (many records: OR-ed into a dense scratch mask during the
// counting pass and copied whole at allocation; few records: OR-ed per record).  Whenever a record
// clears a voxel, each voxel's last record decides its bit through the per-voxel last-record table (largest
// record index per voxel, then applied and reset).  Updates (tracked) take launch_ingest_tracked.
//
// Few records take the flags too where a flag per brick of the grid is small beside its storage (at least a quarter
// of its bricks have some) and quick to clear and compact: the sort's 18 launches cost more than 4 M flags
// (66,000 records: 35 us on a 1024 x 1024 x 256 grid, 51 us on 4 M bricks; sorted 155 and 162; one record on 64^3 21 and 83).
// Their scratch is 16 bytes a brick of the grid however few they are, at most 64 MB beside 4 GB or more of bricks.
constexpr int64_t kFlagBricks = (int64_t)1 << 22;
static bool counting_ingest(const GridView& g, int64_t n) {
  const int64_t nbr_all = (int64_t)g.BX * g.BY * g.BZ;
  return n >= nbr_all / 4 || (nbr_all <= kFlagBricks && nbr_all <= 4 * (int64_t)g.cap);
}
static bool dense_bits_ingest(const GridView& g, int64_t n) {
  const int64_t nbr_all = (int64_t)g.BX * g.BY * g.BZ;
  // the dense mask is indexed by a 32-bit word number (8 words per brick)
  return n >= nbr_all / 4 && nbr_all * 8 < (int64_t)0xFFFFFFFFll;
}
static size_t ingest_scratch_bytes(const GridView& g, int64_t n) {
  const int64_t nbr_all = (int64_t)g.BX * g.BY * g.BZ;
  const bool counting = counting_ingest(g, n);
  const bool dense_bits = dense_bits_ingest(g, n);
  const int64_t m = counting && nbr_all > n ? nbr_all : n;  // brick flags only on the counting path
  const size_t nb4 = align_up((size_t)m * 4);
  const size_t nkeys_al = ((size_t)g.NX * g.NY * g.NZ + 63) & ~(size_t)63;
  const size_t flags = align_up(((size_t)m + nkeys_al) * 4);  // node flags, then brick flags
  const size_t dbytes = dense_bits ? align_up((size_t)nbr_all * 64) : 0;
  return 3 * nb4 + flags + align_up(radix_temp_bytes(n)) + align_up(scan_temp_bytes(m)) + dbytes;
}

// The per-voxel last-record table of the ordered path: cap * 512 words, all -1 between ingests.
static cudaError_t ensure_vlast(const GridView& g, Scratch& vl, cudaStream_t st) {
  const size_t want = (size_t)g.cap * 512 * sizeof(int32_t);
  if (vl.bytes >= want) return cudaSuccess;
  cudaError_t e = ensure_scratch(vl, want);
  if (e != cudaSuccess) return e;
  return cudaMemsetAsync(vl.buf, 0xFF, want, st);
}

cudaError_t reserve_ingest(const GridView& g, int64_t n, Scratch& scr, Scratch& vl, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  cudaError_t e = g.unbounded ? cudaSuccess : ensure_scratch(scr, ingest_scratch_bytes(g, n));
  if (e != cudaSuccess) return e;
  return ensure_vlast(g, vl, st);
}

cudaError_t launch_begin_update(const GridView& g, cudaStream_t st) {
  UpdArgs a{};
  a.g = g;
  VDB_LAUNCH_PDL(k_begin_update<UpdOne>, 1, 32, 0, st, UpdOne{a});
  return cudaGetLastError();
}

cudaError_t prepare_update_args(const GridView& g, Scratch& vl, UpdArgs& a, cudaStream_t st) {
  cudaError_t e = ensure_vlast(g, vl, st);
  if (e != cudaSuccess) return e;
  a.vlast = (int32_t*)vl.buf;
  return cudaSuccess;
}

// The tracked ingest: with `track` (an incremental update) each flipped voxel's brick joins the
// changed list once; unbounded grids take this path for the global form too (no brick-key sort).
static cudaError_t launch_ingest_tracked(const GridView& g, const rec_t* rec, int64_t n, const int32_t* n_dev,
                                         int32_t* changed, int32_t* rslot, Scratch& vl, cudaStream_t st) {
  UpdArgs a{};
  a.g = g;
  a.rec = rec;
  a.n = n;
  a.n_dev = n_dev;
  a.changed = changed;
  a.rslot = rslot;
  cudaError_t e = prepare_update_args(g, vl, a, st);
  if (e != cudaSuccess) return e;
  return update_ingest_kernels(UpdOne{a}, 1, n, st);
}

cudaError_t launch_ingest_records(const GridView& g, const rec_t* rec, int64_t n, const int32_t* n_dev, bool track,
                                  int32_t* changed, int32_t* rslot, Scratch& scr, Scratch& vl, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  if (track || g.unbounded) return launch_ingest_tracked(g, rec, n, n_dev, changed, rslot, vl, st);
  const int64_t nbr_all = (int64_t)g.BX * g.BY * g.BZ;
  const bool counting = counting_ingest(g, n);
  const bool dense_bits = dense_bits_ingest(g, n);
  const int64_t m = counting && nbr_all > n ? nbr_all : n;  // brick flags only on the counting path
  const size_t nb4 = align_up((size_t)m * 4);
  cudaError_t e = ensure_scratch(scr, ingest_scratch_bytes(g, n));
  if (e != cudaSuccess) return e;
  e = ensure_vlast(g, vl, st);
  if (e != cudaSuccess) return e;
  int32_t* vlast = (int32_t*)vl.buf;
  char* p = (char*)scr.buf;
  uint32_t* ka = (uint32_t*)p;
  p += nb4;
  uint32_t* kb = (uint32_t*)p;
  p += nb4;
  // one flag per node key (nodes are created before their bricks), then one per brick or record
  const int64_t nkeys = (int64_t)g.NX * g.NY * g.NZ;
  const int64_t nkeys_al = (nkeys + 63) & ~(int64_t)63;
  int32_t* nflag = (int32_t*)p;
  int32_t* flag = nflag + nkeys_al;
  p += align_up(((size_t)m + (size_t)nkeys_al) * 4);
  // the dense mask follows the flags, so that one memset clears both
  unsigned long long* dbits = dense_bits ? (unsigned long long*)p : nullptr;
  if (dbits) p += align_up((size_t)nbr_all * 64);
  int32_t* pos = (int32_t*)p;
  p += nb4;
  void* rtemp = p;
  p += align_up(radix_temp_bytes(n));
  void* stemp = p;

  const unsigned nbk = blocks_for(n);
  const uint64_t nbr = (uint64_t)nbr_all;
  if (counting) {
    // one flag per brick of the grid, then compaction
    const size_t clear = dbits ? (size_t)((char*)(dbits + nbr * 8) - (char*)nflag) : sizeof(int32_t) * ((size_t)nkeys_al + nbr);
    e = cudaMemsetAsync(nflag, 0, clear, st);
    if (e != cudaSuccess) return e;
    VDB_LAUNCH(k_mark_record_bricks, nbk, kT, 0, st, g, rec, n, n_dev, flag, dbits);
    VDB_LAUNCH_PDL(k_compact_flag_index, blocks_for((int64_t)nbr), kT, 0, st, g, flag, (int64_t)nbr, ka, nflag);
    VDB_LAUNCH_PDL(k_create_flagged_nodes, blocks_for(nkeys), kT, 0, st, g, nflag, nkeys);
    VDB_LAUNCH_PDL(k_alloc_obstacle_bricks, blocks_for((int64_t)nbr), kT, 0, st, g, ka, (int64_t)nbr, dbits);
    if (!dbits) VDB_LAUNCH_PDL(k_apply_set_only, nbk, kT, 0, st, g, rec, n, n_dev);
  } else {
    // LSD radix sort of the brick keys, unique, compaction
    VDB_LAUNCH(k_rec_brick_keys, nbk, kT, 0, st, g, rec, n, n_dev, ka);
    // the sentinel 0xFFFFFFFF sorts after every key below 2^bits
    bool in_b = false;
    e = radix_sort_u32(ka, kb, nullptr, nullptr, n, nullptr, bits_for(nbr), rtemp, st, &in_b);
    if (e != cudaSuccess) return e;
    uint32_t* sorted = in_b ? kb : ka;
    uint32_t* uniq = in_b ? ka : kb;
    VDB_LAUNCH(k_head_flags, nbk, kT, 0, st, sorted, n, (uint32_t)nbr, flag);
    e = exclusive_scan_i32(flag, pos, n, g.counters + C_UNIQUE, stemp, st);
    if (e != cudaSuccess) return e;
    VDB_LAUNCH(k_compact_keys, nbk, kT, 0, st, sorted, flag, pos, n, uniq);
    e = cudaMemsetAsync(nflag, 0, sizeof(int32_t) * (size_t)nkeys, st);
    if (e != cudaSuccess) return e;
    VDB_LAUNCH(k_flag_key_nodes, blocks_for(n), kT, 0, st, g, uniq, n, nflag);
    VDB_LAUNCH_PDL(k_create_flagged_nodes, blocks_for(nkeys), kT, 0, st, g, nflag, nkeys);
    VDB_LAUNCH_PDL(k_alloc_obstacle_bricks, blocks_for(n), kT, 0, st, g, uniq, n, nullptr);
    VDB_LAUNCH_PDL(k_apply_set_only, nbk, kT, 0, st, g, rec, n, n_dev);
  }
  // ordered path (its kernels return at once when no record clears a voxel)
  VDB_LAUNCH_PDL(k_rec_last, nbk, kT, 0, st, g, rec, n, n_dev, vlast);
  VDB_LAUNCH_PDL(k_apply_last, nbk, kT, 0, st, g, rec, n, n_dev, vlast);
  return cudaGetLastError();
}

size_t dense_scratch_bytes(const GridView& g) {
  const size_t nbr = (size_t)g.BX * g.BY * g.BZ, nkeys = (size_t)g.NX * g.NY * g.NZ;
  return align_up(nbr * 64) + align_up(nbr * 4) + align_up(nkeys * 4);
}

cudaError_t launch_ingest_dense(const GridView& g, const uint8_t* grid, Scratch& scr, cudaStream_t st) {
  const size_t nbr = (size_t)g.BX * g.BY * g.BZ, nkeys = (size_t)g.NX * g.NY * g.NZ;
  char* p = (char*)scr.buf;
  DenseScratch ds{(unsigned long long*)p, (int32_t*)(p + align_up(nbr * 64)),
                  (int32_t*)(p + align_up(nbr * 64) + align_up(nbr * 4)), nullptr};
  const OneView v{g};
  // the reset that a dense ingest starts with also clears the brick and node flags; the counters, which its blocks
  // read, are cleared by the next kernel
  VDB_LAUNCH_PDL(k_reset_nodes<OneView>, 1024, kT, 0, st, v, ds.flag, (int64_t)(align_up(nbr * 4) / 4 + nkeys));
  const int planes = dense_planes(g);
  VDB_LAUNCH_PDL((k_dense_masks<OneView, OneSrc>), blocks_for(dense_rows(g) * (8 / planes) * 32), kT, 0, st, v, OneSrc{grid}, ds,
                 planes, true);
  VDB_LAUNCH_PDL(k_dense_nodes<OneView>, batch_blocks(g, BK_DNODES), kT, 0, st, v, ds);
  VDB_LAUNCH_PDL(k_dense_alloc<OneView>, batch_blocks(g, BK_DALLOC), kT, 0, st, v, ds);
  return cudaGetLastError();
}

cudaError_t launch_activation_full(const GridView& g, cudaStream_t st) {
  const OneView v{g};
  VDB_LAUNCH_PDL(k_obstacle_flags<OneView>, 1024, kT, 0, st, v);
  VDB_LAUNCH_PDL(k_node_halo<OneView>, 64, kT, 0, st, v);
  if (g.R <= 16) {
    VDB_LAUNCH_PDL(k_dilate_nodes<OneView>, g.node_cap < 1024 ? g.node_cap : 1024, 256, 0, st, v);
  } else {
    VDB_LAUNCH_PDL((k_dilate_stage<0, OneView>), 256, kT, 0, st, v);
    VDB_LAUNCH_PDL((k_dilate_stage<1, OneView>), 256, kT, 0, st, v);
    VDB_LAUNCH_PDL((k_dilate_stage<2, OneView>), 256, kT, 0, st, v);
  }
  VDB_LAUNCH_PDL(k_alloc_marked<OneView>, g.node_cap * 16 < 8192 ? g.node_cap * 16 : 8192, kT, 0, st, v, true);
  return cudaGetLastError();
}

cudaError_t launch_build_items_full(const GridView& g, const Tuning& t, const Items& it, bool with_slots,
                                    cudaStream_t st) {
  VDB_LAUNCH_PDL(k_items_nodes<OneView>, g.node_cap * 12 < 8192 ? g.node_cap * 12 : 8192, kT, 0, st, OneView{g}, t.run[0],
             t.run[1], t.run[2], it, with_slots);
  return cudaGetLastError();
}

cudaError_t launch_items_dirty(const GridView& g, const Tuning& t, const Items& it, bool with_slots, cudaStream_t st) {
  UpdArgs a{};
  a.g = g;
  VDB_LAUNCH_PDL(k_items_dirty<UpdOne>, dim3(912, 1, 2), kT, 0, st, UpdOne{a}, t.run[0], t.run[1], t.run[2], it, with_slots);
  return cudaGetLastError();
}

cudaError_t launch_count_run_bricks(const GridView* views, const GridView& one, const int32_t* items_ctr, int item_cap,
                                   const Tuning& t, const Items& it, cudaStream_t st) {
  VDB_LAUNCH(k_count_run_bricks, dim3(152, 3), kT, 0, st, views, one, items_ctr, item_cap, t.run[0], t.run[1], t.run[2],
             it);
  return cudaGetLastError();
}

cudaError_t launch_items_dirty_batch(const UpdArgs* d_args, int k, const Tuning& t, const Items& it, cudaStream_t st) {
  if (k <= 0) return cudaSuccess;
  const unsigned share = 912 / k > 16 ? 912 / k : 16;
  VDB_LAUNCH_PDL(k_items_dirty<UpdBatch>, dim3(share, k, 2), kT, 0, st, UpdBatch{d_args}, t.run[0], t.run[1], t.run[2], it,
                 true);
  return cudaGetLastError();
}

// ---- batches ----
static int clamp_blocks(int64_t n, int hi) { return (int)(n < 1 ? 1 : (n > hi ? hi : n)); }

int batch_blocks(const GridView& g, int kind) {
  const int64_t t = kT;
  switch (kind) {
    case BK_RESET: return clamp_blocks(((int64_t)g.node_cap * (kNodeBricks / 4) + g.hmask + t) / t, 1024);  // int4 stores
    case BK_DENSE: {
      const int64_t units = dense_rows(g);  // a warp each
      return clamp_blocks((units * 32 + t - 1) / t, 152 * 16);
    }
    case BK_DNODES: return clamp_blocks(((int64_t)g.NX * g.NY * g.NZ + t - 1) / t, 1024);
    case BK_DALLOC: return clamp_blocks(((int64_t)g.BX * g.BY * g.BZ + t - 1) / t, 152 * 64);
    case BK_OBST: return clamp_blocks(((int64_t)g.cap + t - 1) / t, 1024);
    case BK_HALO: return clamp_blocks(((int64_t)g.node_cap * 32 + t - 1) / t, 64);
    case BK_DILATE: return clamp_blocks(g.node_cap, 1024);
    case BK_ALLOC: return clamp_blocks((int64_t)g.node_cap * 8, 8192);  // two 256-brick chunks per block
    case BK_ITEMS: return clamp_blocks((int64_t)g.node_cap * 12, 8192);
  }
  return 1;
}

cudaError_t launch_reset_batch(const GridView* views, const BatchShape& b, int32_t* counters_all, size_t n_counters,
                               cudaStream_t st) {
  if (b.k <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_reset_nodes<BatchViews>, b.total[BK_RESET], kT, 0, st, BatchViews{views, b.first[BK_RESET], b.k},
                 (int32_t*)nullptr, (int64_t)0);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return cudaMemsetAsync(counters_all, 0, sizeof(int32_t) * n_counters, st);
}

cudaError_t launch_ingest_dense_batch(const GridView* views, const BatchShape& b, const uint8_t* const* srcs,
                                      void* scratch, const int64_t* offsets, size_t flag_words, int32_t* flag0,
                                      cudaStream_t st) {
  if (b.k <= 0) return cudaSuccess;
  if (b.k > kBatchMax) return cudaErrorInvalidValue;
  BatchSrc src;
  for (int i = 0; i < kBatchMax; ++i) src.p[i] = i < b.k ? srcs[i] : nullptr;
  cudaError_t e = cudaMemsetAsync(flag0, 0, flag_words * 4, st);
  if (e != cudaSuccess) return e;
  char* p = (char*)scratch;
  DenseScratch ds{(unsigned long long*)p, (int32_t*)p, (int32_t*)p, offsets};
  VDB_LAUNCH((k_dense_masks<BatchViews, BatchSrc>), b.total[BK_DENSE], kT, 0, st,
             BatchViews{views, b.first[BK_DENSE], b.k}, src, ds, 8, false);
  VDB_LAUNCH_PDL(k_dense_nodes<BatchViews>, b.total[BK_DNODES], kT, 0, st, BatchViews{views, b.first[BK_DNODES], b.k}, ds);
  VDB_LAUNCH_PDL(k_dense_alloc<BatchViews>, b.total[BK_DALLOC], kT, 0, st, BatchViews{views, b.first[BK_DALLOC], b.k}, ds);
  return cudaGetLastError();
}

cudaError_t launch_activation_batch(const GridView* views, const BatchShape& b, cudaStream_t st) {
  if (b.k <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_obstacle_flags<BatchViews>, b.total[BK_OBST], kT, 0, st, BatchViews{views, b.first[BK_OBST], b.k});
  VDB_LAUNCH_PDL(k_node_halo<BatchViews>, b.total[BK_HALO], kT, 0, st, BatchViews{views, b.first[BK_HALO], b.k});
  const BatchViews dv{views, b.first[BK_DILATE], b.k};
  if (b.R <= 16) {
    VDB_LAUNCH_PDL(k_dilate_nodes<BatchViews>, b.total[BK_DILATE], 256, 0, st, dv);
  } else {
    VDB_LAUNCH((k_dilate_stage<0, BatchViews>), b.total[BK_DILATE], kT, 0, st, dv);
    VDB_LAUNCH((k_dilate_stage<1, BatchViews>), b.total[BK_DILATE], kT, 0, st, dv);
    VDB_LAUNCH((k_dilate_stage<2, BatchViews>), b.total[BK_DILATE], kT, 0, st, dv);
  }
  VDB_LAUNCH_PDL(k_alloc_marked<BatchViews>, b.total[BK_ALLOC], kT, 0, st, BatchViews{views, b.first[BK_ALLOC], b.k},
                 true);
  return cudaGetLastError();
}

cudaError_t launch_build_items_batch(const GridView* views, const BatchShape& b, const Tuning& t, const Items& it,
                                     cudaStream_t st) {
  if (b.k <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_items_nodes<BatchViews>, b.total[BK_ITEMS], kT, 0, st, BatchViews{views, b.first[BK_ITEMS], b.k},
             t.run[0], t.run[1], t.run[2], it, true);
  return cudaGetLastError();
}

// Incremental: records were already applied with flip tracking (changed list filled).
// (the item counters were cleared when the update began)
cudaError_t launch_incremental_mark(const GridView& g, const Tuning& t, const int32_t* changed, const Items& it,
                                    const Fork& fk, cudaStream_t st) {
  UpdArgs a{};
  a.g = g;
  a.changed = const_cast<int32_t*>(changed);
  return update_mark_kernels(UpdOne{a}, GatedOne{g}, 1, g.node_cap, g.R, windowed_form(g), t, it, fk, st);
}

// Batched update: begin + tracked ingest of every grid, then the marking (one launch per step).
cudaError_t launch_update_batch_ingest(const UpdArgs* d_args, const BatchUpdShape& s, const BatchCounts& counts,
                                       cudaStream_t st) {
  if (s.k <= 0) return cudaSuccess;
  VDB_LAUNCH_PDL(k_begin_batch_update, dim3(1, s.k), 32, 0, st, d_args, counts);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return update_ingest_kernels(UpdBatch{d_args}, s.k, s.max_n, st);
}

cudaError_t launch_update_batch_mark(const UpdArgs* d_args, const BatchUpdShape& s, const Tuning& t, const Items& it,
                                     const Fork& fk, cudaStream_t st) {
  if (s.k <= 0) return cudaSuccess;
  return update_mark_kernels(UpdBatch{d_args}, GatedBatch{d_args}, s.k, (int)s.max_node_cap, s.R, s.windowed, t, it, fk,
                             st);
}

}  // namespace vdbedt
