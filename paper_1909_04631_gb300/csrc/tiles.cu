// Steps a2-a3 by occupied tiles: the downsampling of hits and free samples to
// one exact centroid per (cell, label) without sorting the items.
//
// The items (hits and the samples of every beam) are cheap to compute from the
// transformed hits, so each pass below forms them again instead of storing
// them, and the sums of a cell are integers (x 2^-E with E fixed by the cell's
// tile of 8^3 cells), so they may be added in any order:
//   mark     a directory word per tile of the scans' frames, set by the first
//            item of the tile (with counts per 256 and per 65536 entries);
//   rank     occupied tiles numbered in directory order; each gets 512 cells;
//   masks    per cell a bit per label that occurs: a training point each;
//   counts   training points per tile and per 256 tiles;
//   offsets  per cell its first training point; sums cleared, keys noted;
//   add      every item adds x 2^-E to the three 64-bit sums of its training
//            point and 1 to its count, runs of neighbouring beams at once;
//   finish   the mean of every training point, rounded once.
// The training point of an item is offset[cell] + the number of lower labels in
// the cell's mask, which orders the points by (scan, tile, cell, label), the
// order of the sorted form, and gives the same bits.
// A member with a fraction in units of 2^E (a coordinate within about 2^-21 ds
// of a coordinate plane: a few hits of most ground scans) has the fraction noted
// in a short list.  Fractions below 2^-40, a full list, a mean below the FP32
// normal range or 2^18 members next to a plane leave the point to two more
// launches (idle otherwise), which gather the members of such points and take
// the sorted form's exact mean of a cell.
//
// Why: the sorted form moves every item through four or five radix passes
// (12 bytes in and out each) and a segment pass; here a run of neighbouring
// beams' items is three reductions and two dependent lookups into tables that
// stay in L2.  Ingest of a 64 x 2048 street scan (3.0M items, 690k points)
// 348 -> 239 us, of a 640 x 480 depth frame (9.3M items, 300k points) 822 -> 354,
// of a 9k-ray scan 153 -> 122, of 16 street scans in a batch 2600 -> 1490.
// What bounds it: the reductions (40 of the 85 us of `add` on the street scan)
// and the issue of forming each item three times; for sparse scans the cells of
// their tiles, for few beams the walk along the longest.  There, and for beams in
// no order, the sorted form is the faster one: TileGate draws the line.
#include <algorithm>
#include <cmath>

#include "exact_mean.cuh"
#include "point_common.cuh"

namespace sbki {
namespace {

constexpr int kCells = 1 << kLocalBits;  // cells of a tile
constexpr int kChunk = 256;              // directory entries per rank CTA, one per thread
constexpr int kSuper = 256;              // chunks per second-level count
// words from one second-level count to the next: a line each.  A sparse scan adds
// up to its number of items to a few of them, and atomics on one line take turns
// (side by side in two lines, marking 3.2M items of a 60 m scan took 91 us)
constexpr int kSuperStep = 32;
constexpr int kGroup = 256;              // tiles per count of training points
constexpr uint32_t kBadPoint = 1u << 31;   // info word: the sums do not give the point's mean
constexpr uint32_t kLowPoint = 1u << 30;   // info word: fractions of its members are in the list
constexpr uint32_t kRankMask = kLowPoint - 1u;
constexpr int kLowBits = 40;               // a noted fraction counts units of 2^(E - 40)
constexpr uint32_t kLowCap = 256;          // noted fractions at most
constexpr uint32_t kNoPoint = 0xffffffffu;
constexpr uint32_t kMaxMembers = 1u << 18;  // |sum| < n 2^(24 + kSegShift - 3) < 2^63 below this

struct LowPart {  // a member's fraction on one axis
  long long low;
  uint32_t p, ax;
};

// Buffers of the tile form, in the scratch of the sorted form (S = its item capacity).
struct TileBufs {
  uint32_t* dir;       // [entries] 0, 1 marked, then rank + 1; chunk and second-level counts behind (keys)
  uint32_t* chunks;    // [entries / kChunk + 1] occupied tiles per chunk
  uint32_t* supers;    // [chunks / kSuper + 1] counts, kSuperStep words apart
  uint32_t* groups;    // [tile_cap / kGroup + 1] training points per kGroup tiles
  uint2* cells;        // [tile_cap * kCells] (label mask, first training point) (sitems)
  int4* tiles;         // [tile_cap] each occupied tile: index per axis, scan (seg_start)
  uint32_t* counts;    // [tile_cap] training points per tile (seg_start)
  uint32_t* start;     // [flagged points] where the next gathered member goes (the rest of seg_start)
  unsigned long long* sum[3];  // [points] per axis (items: x, y; keys2: z)
  uint32_t* members;   // [points] (vals)
  uint32_t* info;      // [points] tile rank, kLowPoint; kBadPoint | the place among the flagged (vals2)
  uint32_t* key;       // [points] label | cell << 5 (flags)
  uint32_t* flagged;   // [flagged points] training point (slow)
  LowPart* low;        // [kLowCap] (hist)
  float4* gathered;    // [members of flagged points] (items, when the sums are done)
  uint32_t entries;
  uint32_t tile_cap;
};

struct TileArgs {
  Geom g;
  TileBufs b;
  const float4* world;
  const unsigned long long* cnt;  // hits << 40 | samples per point
  const ScanDesc* desc;
  int ns;
  float4* train;
  DevCounters* dc;
  bool alone;           // no sorted form behind: an item outside the frame is an error
  TileGate gate;
  uint32_t pack_limit;  // scans of fewer points have no cell of 2^19 members: counts ride on the sums
};

// The frame of one scan's tiles in the directory.
struct TileFrame {
  int o[3], e[3];
  uint32_t first;
};
__device__ __forceinline__ TileFrame frame_of(const ScanDesc& d) {
  TileFrame f;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    f.o[a] = d.org[a];
    f.e[a] = d.ext[a];
  }
  f.first = d.tile0;
  return f;
}

// One item: its directory entry (kNoPoint for none), cell and label.
struct Item {
  float x[3];
  int gc[3];  // downsampling cell per axis
  uint32_t entry, cell;  // cell | label << kLocalBits
  bool out;              // live, but outside the frame (no entry)
  __device__ __forceinline__ uint32_t local() const { return cell & (uint32_t)(kCells - 1); }
  __device__ __forceinline__ uint32_t label() const { return cell >> kLocalBits; }
};
__device__ __forceinline__ Item make_item(bool live, float x, float y, float z, uint32_t label, const Geom& g,
                                          const TileFrame& f) {
  Item it;
  it.x[0] = x;
  it.x[1] = y;
  it.x[2] = z;
  int t[3];
  bool in = true;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    it.gc[a] = floor_small(__fmul_rn(it.x[a], g.inv_ds));  // |cell| < 2^22 (the transform declines others)
    t[a] = (it.gc[a] >> kTileShift) - f.o[a];
    in = in && (uint32_t)t[a] < (uint32_t)f.e[a];
  }
  constexpr int m = kTileEdge - 1;
  it.cell = (uint32_t)(((it.gc[2] & m) << (2 * kTileShift)) | ((it.gc[1] & m) << kTileShift) | (it.gc[0] & m)) |
            label << kLocalBits;
  it.out = live && !in;
  it.entry = kNoPoint;
  if (live && in) it.entry = f.first + (uint32_t)((t[0] * f.e[1] + t[1]) * f.e[2] + t[2]);
  return it;
}

// A run of consecutive lanes whose items share a cell and label: `last` in its
// last lane, which looks the cell up and writes for all of them.
struct Run {
  bool last;
  uint32_t lasts;  // last lanes of the warp
  int first;       // first lane of this lane's run
  __device__ __forceinline__ explicit Run(const Item& it) {
    const int lane = threadIdx.x & 31;
    const uint32_t e = __shfl_down_sync(0xffffffffu, it.entry, 1), c = __shfl_down_sync(0xffffffffu, it.cell, 1);
    last = lane == 31 || e != it.entry || c != it.cell;
    lasts = __ballot_sync(0xffffffffu, last);
    const uint32_t below = lasts & ((1u << lane) - 1u);
    first = below ? 32 - __clz((int)below) : 0;
  }
};

// t / r to nearest for many 0 < t <= r: Markstein's quotient (P. Markstein,
// "Computation of elementary functions on the IBM RISC System/6000 processor",
// 1990): with y the correctly rounded reciprocal of r and q within an ulp of
// t / r, the remainder t - q r is exact and RN(q + (t - q r) y) = RN(t / r),
// unless r's mantissa is all ones.  One such step takes RN(t y) to within an
// ulp, the second gives the quotient.  Those r, and ones outside 2^-40..2^40
// (where the remainder could leave the normal range: t >= 2^-24 r here), divide.
struct Quotient {
  float r, y;
  bool plain;
  __device__ __forceinline__ explicit Quotient(float r_) : r(r_) {
    const uint32_t b = __float_as_uint(r);
    plain = (b & 0x7fffffu) == 0x7fffffu || !(r > 0x1p-40f && r < 0x1p40f);
    y = __frcp_rn(plain ? 1.0f : r);
  }
  __device__ __forceinline__ float operator()(float t) const {
    if (plain || t < 0x1p-24f * r) return __fdiv_rn(t, r);
    float q = __fmul_rn(t, y);
    q = __fmaf_rn(__fmaf_rn(-q, r, t), y, q);
    return __fmaf_rn(__fmaf_rn(-q, r, t), y, q);
  }
};

// Every item of the update through op.  A warp takes 32 consecutive points
// (beams), a lane each, so the samples at the same place along neighbouring
// beams, which mostly share a cell, meet in one warp: op.look sees the runs and
// only their last lanes touch memory; op.done ends the warp's share early.  kPhases warps share 32 beams, each
// taking two samples of every 2 kPhases (two chains of dependent loads in
// flight); the first also takes the hits.
constexpr int kPhases = 8;
template <class Op>
__device__ __forceinline__ void each_item(const TileArgs& a, Op& op) {
  __shared__ int64_t s_off[kMaxScans + 1];
  for (int t = threadIdx.x; t <= a.ns; t += blockDim.x) s_off[t] = a.desc[t].off;
  __syncthreads();
  const Geom& g = a.g;
  const int64_t n = s_off[a.ns];
  const int lane = threadIdx.x & 31;
  const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nwarps = ((int64_t)gridDim.x * blockDim.x) >> 5;
  TileFrame f = frame_of(a.desc[0]);
  float o[3] = {a.desc[0].o[0], a.desc[0].o[1], a.desc[0].o[2]};
  for (int64_t task = warp; task < (n + 31) / 32 * kPhases; task += nwarps) {
    const int64_t i = task / kPhases * 32 + lane;
    const uint32_t phase = (uint32_t)(task % kPhases);
    uint32_t nfree = 0;
    bool hit = false;
    float4 w = make_float4(0.f, 0.f, 0.f, 0.f);
    if (i < n) {
      if (a.ns > 1) {
        const ScanDesc& d = a.desc[scan_of(s_off, a.ns, i)];
        f = frame_of(d);
        o[0] = d.o[0];
        o[1] = d.o[1];
        o[2] = d.o[2];
      }
      const unsigned long long c = a.cnt[i];
      hit = (c >> 40) != 0ull;
      nfree = (uint32_t)(c & kFreeMask);
      w = a.world[i];
    }
    if (phase == 0) {
      const Item it = make_item(hit, w.x, w.y, w.z, (uint32_t)(int)w.w, g, f);
      op.apply(op.look(it, Run(it)));
    }
    const float sx = __fsub_rn(w.x, o[0]), sy = __fsub_rn(w.y, o[1]), sz = __fsub_rn(w.z, o[2]);
    const float rr = __fsqrt_rn(__fadd_rn(__fadd_rn(__fmul_rn(sx, sx), __fmul_rn(sy, sy)), __fmul_rn(sz, sz)));
    const uint32_t most = __reduce_max_sync(0xffffffffu, nfree);
    const Quotient by_r(rr);
    for (uint32_t j0 = 2 * phase + 1; j0 <= most; j0 += 2 * kPhases) {
      typename Op::Found found[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        const uint32_t j = j0 + u;
        const bool live = j <= nfree;
        const float k = by_r(__fsub_rn(rr, __fmul_rn((float)j, g.step)));
        const Item it = make_item(live, __fadd_rn(o[0], __fmul_rn(sx, k)), __fadd_rn(o[1], __fmul_rn(sy, k)),
                                  __fadd_rn(o[2], __fmul_rn(sz, k)), 0u, g, f);
        found[u] = op.look(it, Run(it));
      }
#pragma unroll
      for (int u = 0; u < 2; ++u) op.apply(found[u]);
      if (op.done()) return;  // warp-uniform
    }
  }
}

// whether the tile form takes this update: decided on the device when its tiles are marked
// (tile_rank_kernel; n_sort holds the answer for the sorted form)
__device__ __forceinline__ bool tiles_on(const TileArgs& a) { return a.dc->tiles_taken != 0u; }
__device__ __forceinline__ bool packed(const TileArgs& a) { return a.dc->max_points < a.pack_limit; }

// ---------------------------------------------------------------- mark, rank
// A warp adds its fresh tiles to the total in steps of kFlush and stops once the
// total is past the limit: a sparse scan, whose items mostly have a tile each, is
// declined after a small share of them.
constexpr uint32_t kFlush = 16;
struct MarkOp {
  struct Found {
    uint32_t entry, old;
  };
  const TileArgs& a;
  uint32_t limit;
  uint32_t fresh = 0;
  bool out = false;
  __device__ __forceinline__ bool done() {
    const uint32_t w = __reduce_add_sync(0xffffffffu, fresh);
    if (w < kFlush) return false;
    uint32_t before = 0;
    if ((threadIdx.x & 31) == 0) {
      before = *(volatile const uint32_t*)&a.dc->n_ttiles;
      if (before <= limit) before = atomicAdd(&a.dc->n_ttiles, w);
    }
    fresh = 0;
    return __shfl_sync(0xffffffffu, before, 0) + w > limit;
  }
  // A tile's word is mostly set already: a cached read first (it may be an old
  // 0), then one past the L1, so the tiles around the sensor do not serialise.
  __device__ __forceinline__ Found look(const Item& it, const Run& run) {
    Found f{it.entry, 1u};
    out = out || it.out;
    if (run.last && it.entry != kNoPoint) {
      f.old = a.b.dir[it.entry];
      if (f.old == 0u) f.old = *(volatile const uint32_t*)(a.b.dir + it.entry);
    }
    return f;
  }
  __device__ __forceinline__ void apply(const Found& f) {
    if (f.old == 0u && atomicExch(a.b.dir + f.entry, 1u) == 0u) {
      atomicAdd(a.b.chunks + f.entry / kChunk, 1u);
      atomicAdd(a.b.supers + f.entry / (kChunk * kSuper) * kSuperStep, 1u);
      ++fresh;
    }
  }
};
// The directory and its counts to zero, unless marking will not start.  Up to
// kClearAlways words a plain memset takes no longer than this launch.
constexpr int64_t kClearAlways = 1 << 18;
__global__ void __launch_bounds__(256) tile_clear_kernel(TileArgs a, uint32_t words) {
  __shared__ uint32_t s_limit;  // nothing of it changes in this launch
  if (threadIdx.x == 0) s_limit = a.dc->err || a.dc->n_ttiles ? 0u : a.gate.limit(*a.dc);
  __syncthreads();
  if (s_limit == 0u) return;
  uint4* const d = reinterpret_cast<uint4*>(a.b.dir);
  const uint32_t i0 = blockIdx.x * 256 + threadIdx.x;
  for (uint32_t i = i0; i < words / 4; i += gridDim.x * 256) d[i] = make_uint4(0u, 0u, 0u, 0u);
  if (i0 < (words & 3u)) a.b.dir[words / 4 * 4 + i0] = 0u;
}

__global__ void __launch_bounds__(256, 6) tile_mark_kernel(TileArgs a) {
  // other CTAs of this launch may set the error, decline or pass the limit, so one read decides for the whole CTA:
  // warps that went on without the others would miss each_item's scan offsets
  __shared__ uint32_t s_limit;  // 0: nothing to do
  if (threadIdx.x == 0) {
    s_limit = a.gate.limit(*a.dc);
    if (s_limit == 0u) atomicMax(&a.dc->n_ttiles, kTilesDeclined);  // not even one tile
    if (*(volatile const int*)&a.dc->err != 0 || *(volatile const uint32_t*)&a.dc->n_ttiles > s_limit) s_limit = 0u;
  }
  __syncthreads();
  const uint32_t limit = s_limit;
  if (limit == 0u) return;
  MarkOp op{a, limit};
  each_item(a, op);
  const uint32_t w = __reduce_add_sync(0xffffffffu, op.fresh);
  const bool out = __any_sync(0xffffffffu, op.out);
  if ((threadIdx.x & 31) == 0 && w) atomicAdd(&a.dc->n_ttiles, w);
  if ((threadIdx.x & 31) == 0 && out) {  // a pose that scales or shears can leave the frame of max_range
    if (a.alone) set_error(a.dc, SBKI_ERR_INVALID_ARG);
    else atomicMax(&a.dc->n_ttiles, kTilesDeclined);
  }
}

// The scan whose directory entries hold e, and e's tile per axis.
__device__ __forceinline__ int tile_of_entry(const TileArgs& a, uint32_t e, int t[3]) {
  int s = 0;
  while (s + 1 < a.ns && a.desc[s + 1].tile0 <= e) ++s;
  const TileFrame f = frame_of(a.desc[s]);
  uint32_t r = e - f.first;
  const uint32_t xy = r / (uint32_t)f.e[2];
  t[2] = (int)(r - xy * (uint32_t)f.e[2]) + f.o[2];
  const uint32_t x = xy / (uint32_t)f.e[1];
  t[1] = (int)(xy - x * (uint32_t)f.e[1]) + f.o[1];
  t[0] = (int)x + f.o[0];
  return s;
}

// Ranks in directory order: a CTA per chunk adds up the counts before it (whole
// second-level counts, then chunks), so no CTA waits on another; the cells of
// its tiles are cleared.  n_sort: the items left to the sorted form.
__global__ void __launch_bounds__(256) tile_rank_kernel(TileArgs a) {
  __shared__ uint32_t s_w[8];
  if (!a.gate.takes(*a.dc)) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    a.dc->tiles_taken = 1u;
    a.dc->n_sort = a.dc->n_scan = 0u;
  }
  const uint32_t nch = (a.b.entries + kChunk - 1) / kChunk;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t whole = 0u, next = threadIdx.x;  // this thread's share of the second-level counts, read once as c grows
  for (uint32_t c = blockIdx.x; c < nch; c += gridDim.x) {
    if (a.b.chunks[c] == 0u) continue;  // uniform over the CTA
    __syncthreads();
    for (; next < c / kSuper; next += 256) whole += a.b.supers[next * kSuperStep];
    uint32_t before = whole;
    for (uint32_t k = c / kSuper * kSuper + threadIdx.x; k < c; k += 256) before += a.b.chunks[k];
    before = __reduce_add_sync(0xffffffffu, before);
    if (lane == 0) s_w[warp] = before;
    __syncthreads();
    before = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) before += s_w[w];
    __syncthreads();
    const uint32_t e = c * kChunk + threadIdx.x;
    const bool occupied = e < a.b.entries && a.b.dir[e] != 0u;
    const unsigned mask = __ballot_sync(0xffffffffu, occupied);
    if (lane == 0) s_w[warp] = __popc(mask);
    __syncthreads();
    uint32_t r = before + __popc(mask & ((1u << lane) - 1u)), total = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      if (w < warp) r += s_w[w];
      total += s_w[w];
    }
    if (occupied) {
      a.b.dir[e] = r + 1u;
      int t[3];
      const int scan = tile_of_entry(a, e, t);
      a.b.tiles[r] = make_int4(t[0], t[1], t[2], scan);
    }
    // the chunk's tiles have consecutive ranks: one run of cells to clear
    uint4* z = reinterpret_cast<uint4*>(a.b.cells + (size_t)before * kCells);
    for (uint32_t k = threadIdx.x; k < total * (kCells / 2); k += 256) z[k] = make_uint4(0u, 0u, 0u, 0u);
  }
}

// ---------------------------------------------------------------- masks, offsets
struct MaskOp {
  struct Found {
    uint32_t rank, cell, bit, old;
  };
  const TileArgs& a;
  __device__ __forceinline__ Found look(const Item& it, const Run& run) const {
    Found f{0u, 0u, 0u, 0u};
    if (run.last && it.entry != kNoPoint) {
      f.rank = __ldg(a.b.dir + it.entry) - 1u;
      f.cell = it.local();
      f.bit = 1u << it.label();
      f.old = *(volatile const uint32_t*)&a.b.cells[(size_t)f.rank * kCells + f.cell].x;
    }
    return f;
  }
  __device__ __forceinline__ bool done() const { return false; }
  __device__ __forceinline__ void apply(const Found& f) {
    if ((f.old & f.bit) != f.bit) atomicOr(&a.b.cells[(size_t)f.rank * kCells + f.cell].x, f.bit);
  }
};
__global__ void __launch_bounds__(256, 6) tile_masks_kernel(TileArgs a) {
  if (!tiles_on(a)) return;
  MaskOp op{a};
  each_item(a, op);
}

// A warp per tile: its training points, the labels of its cells.
__global__ void __launch_bounds__(256) tile_counts_kernel(TileArgs a) {
  if (!tiles_on(a)) return;
  const uint32_t nt = a.dc->n_ttiles;
  const int lane = threadIdx.x & 31;
  for (uint32_t r = (blockIdx.x * 256 + threadIdx.x) >> 5; r < nt; r += gridDim.x * 8) {
    const uint4* cells = reinterpret_cast<const uint4*>(a.b.cells + (size_t)r * kCells);
    uint32_t k = 0;
#pragma unroll
    for (int q = 0; q < kCells / 64; ++q) {
      const uint4 c = cells[q * 32 + lane];
      k += __popc(c.x) + __popc(c.z);
    }
    k = __reduce_add_sync(0xffffffffu, k);
    if (lane == 0) {
      a.b.counts[r] = k;
      atomicAdd(a.b.groups + r / kGroup, k);
    }
  }
}

// A warp per tile, eight consecutive tiles per CTA: every cell's first training
// point; the tile's sums cleared.  Bound by memory (4 KB of cells a tile, mostly
// empty, and 36 bytes a point).  With 16 consecutive cells per lane (loads and
// stores of 16 bytes, 128 apart) it took 260 us for a batch of 16 scans, by rows 141.
__global__ void __launch_bounds__(256) tile_offsets_kernel(TileArgs a) {
  if (!tiles_on(a)) return;
  const uint32_t nt = a.dc->n_ttiles;
  __shared__ uint32_t s_w[8], s_c[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (uint32_t r0 = blockIdx.x * 8; r0 < nt; r0 += gridDim.x * 8) {  // uniform over the CTA
    // points before the CTA's eight tiles: whole groups, then tiles
    __syncthreads();
    uint32_t before = 0;
    for (uint32_t k = threadIdx.x; k < r0 / kGroup; k += 256) before += a.b.groups[k];
    for (uint32_t k = r0 / kGroup * kGroup + threadIdx.x; k < r0; k += 256) before += a.b.counts[k];
    before = __reduce_add_sync(0xffffffffu, before);
    const uint32_t r = r0 + warp;
    if (lane == 0) {
      s_w[warp] = before;
      s_c[warp] = r < nt ? a.b.counts[r] : 0u;
    }
    __syncthreads();
    uint32_t p = 0, p1 = 0;
#pragma unroll
    for (int w = 0; w < 8; ++w) {
      p += s_w[w];
      if (w < warp) p += s_c[w];
    }
    if (r >= nt) continue;
    p1 = p + s_c[warp];
    if (r == nt - 1 && lane == 0) a.dc->n_train = p1;
    for (uint32_t k = p + lane; k < p1; k += 32) {
      a.b.sum[0][k] = 0ull;
      a.b.sum[1][k] = 0ull;
      a.b.sum[2][k] = 0ull;
      a.b.members[k] = 0u;
      a.b.info[k] = r;
    }
    // rows of 64 cells, two consecutive cells per lane, so every load and store is whole lines; the counts of
    // two rows share a scan (a tile has at most 2^14 points)
    constexpr int kRows = kCells / 64;
    uint4* cells = reinterpret_cast<uint4*>(a.b.cells + (size_t)r * kCells);
    uint4 c[kRows];
#pragma unroll
    for (int q = 0; q < kRows; ++q) c[q] = cells[q * 32 + lane];
    uint32_t first = p;
#pragma unroll
    for (int q = 0; q < kRows; q += 2) {
      const uint32_t n0 = __popc(c[q].x) + __popc(c[q].z), n1 = __popc(c[q + 1].x) + __popc(c[q + 1].z);
      const uint32_t n = n0 | n1 << 16;
      if (!__any_sync(0xffffffffu, n)) continue;
      uint32_t inc = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t u = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += u;
      }
      const uint32_t all = __shfl_sync(0xffffffffu, inc, 31);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint4& w = c[q + h];
        if ((w.x | w.z) == 0u) continue;
        uint32_t at = h == 0 ? first + (inc & 0xffffu) - n0 : first + (all & 0xffffu) + (inc >> 16) - n1;
        const uint32_t cell = (uint32_t)((q + h) * 64 + 2 * lane) << 5;
        w.y = at;
        for (uint32_t m = w.x; m; m &= m - 1u) a.b.key[at++] = (uint32_t)(__ffs((int)m) - 1) | cell;
        w.w = at;
        for (uint32_t m = w.z; m; m &= m - 1u) a.b.key[at++] = (uint32_t)(__ffs((int)m) - 1) | (cell + 32u);
        cells[(q + h) * 32 + lane] = w;
      }
      first += (all & 0xffffu) + (all >> 16);
    }
  }
}

// ---------------------------------------------------------------- sums
__device__ __forceinline__ uint32_t point_of(const TileArgs& a, const Item& it) {
  const uint32_t rank = __ldg(a.b.dir + it.entry) - 1u;
  const uint2 c = __ldg(a.b.cells + (size_t)rank * kCells + it.local());
  return c.y + __popc(c.x & ((1u << it.label()) - 1u));
}
// The unit 2^E of a tile's sums on one axis.  Away from the coordinate plane
// (tile index t other than 0 and -1) every |x| of the tile is at least
// 8 m ds (1 - 2^-22), m = t or -t - 1, and with E 24 below the exponent of
// 8 m ds every x 2^-E is an integer below 2^26 (1 + 2^-22): 32 of them add up
// in 32 bits, and any number of them in 64.  Next to the plane the unit is the
// segment pass's (TileUnit); there the sums are taken from the corner of the
// cell, an integer near c ds 2^-E, and stay below 2^63 for kMaxMembers.
// Where no cell can have 2^19 members (packed), the count of members rides
// above bit 45 of the first such axis's sum of magnitudes (below 2^45 then), so
// a point takes three reductions instead of four.
constexpr int kCountShift = 45;
__device__ __forceinline__ int count_axis(bool p0, bool p1, bool p2) {  // p: plane; 3: the members' own word
  return !p0 ? 0 : (!p1 ? 1 : (!p2 ? 2 : 3));
}
struct AxisUnit {
  float scale;  // 2^-E, 0 outside the FP32 normal range
  int E;
  bool plane;
};
__device__ __forceinline__ AxisUnit axis_unit(int t, const Geom& g) {
  AxisUnit u;
  const int m = t < 0 ? -t - 1 : t;
  u.plane = m == 0;
  const float L = __fmul_rn((float)(u.plane ? kTileEdge + 2 : kTileEdge * m), g.ds);
  u.E = (int)(__float_as_uint(L) >> 23) - (u.plane ? 150 + kSegShift : 151);
  u.scale = u.E >= -126 && u.E <= 126 ? __uint_as_float((uint32_t)(127 - u.E) << 23) : 0.f;
  return u;
}
__device__ __forceinline__ long long corner_of(int c, float ds, float scale) {
  return (long long)c * __float2ll_rz(__fmul_rn(ds, scale));
}

// Sum of v over this lane's run, in the run's last lane: the difference of two
// prefix sums of the warp (exact in wrapping integers).
template <typename T>
__device__ __forceinline__ T run_sum(T v, const Run& run) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int s = 1; s < 32; s <<= 1) {
    const T o = __shfl_up_sync(0xffffffffu, v, s);
    if (lane >= s) v += o;
  }
  const T before = __shfl_sync(0xffffffffu, v, max(run.first - 1, 0));
  return run.first ? v - before : v;
}

// The fractions of a member of point p into the list (rare); false when one is
// finer than the list's unit or the list is full.
__device__ __noinline__ bool note_fractions(LowPart* list, uint32_t* count, uint32_t p, float fx, float fy, float fz) {
  for (uint32_t ax = 0; ax < 3; ++ax) {
    const float frac = ax == 0 ? fx : (ax == 1 ? fy : fz);
    if (frac == 0.f) continue;
    const float v = frac * (float)(1ull << kLowBits);  // exact; an integer unless the fraction is finer
    const long long low = __float2ll_rz(v);
    const uint32_t k = atomicAdd(count, 1u);
    if ((float)low != v || k >= kLowCap) return false;
    list[k] = {low, p, ax};
  }
  return true;
}

struct AddOp {
  struct Found {
    unsigned long long d[3];
    uint32_t p, n;
    bool bad, own;  // own: the count goes to the members' own word
  };
  const TileArgs& a;
  bool packed;
  __device__ __forceinline__ Found look(const Item& it, const Run& run) const {
    const int lane = threadIdx.x & 31;
    Found f;
    f.p = kNoPoint;
    if (run.last && it.entry != kNoPoint) f.p = point_of(a, it);
    // sums over the run, in its last lane
    const int at = lane - run.first;  // place in the run
    f.n = (uint32_t)at + 1u;
    const bool live = it.entry != kNoPoint;
    const bool runs = __any_sync(0xffffffffu, live && !run.last);  // some run has two lanes
    bool bad = false, plane[3];
    float frac[3];  // fraction of x 2^-E, or 0
#pragma unroll
    for (int ax = 0; ax < 3; ++ax) {
      const AxisUnit u = axis_unit(it.gc[ax] >> kTileShift, a.g);
      plane[ax] = u.plane;
      const float q = __fmul_rn(it.x[ax], u.scale);  // x 2^-E, exact when |q| >= 2^23
      const float aq = fabsf(q);
      bad = bad || u.scale == 0.f;
      frac[ax] = 0.0f;
      if (__any_sync(0xffffffffu, live && u.plane)) {
        bad = bad || aq >= 281474976710656.0f;
        frac[ax] = aq < 8388608.0f ? q - truncf(q) : 0.0f;
        const long long v = u.plane ? __float2ll_rz(q) - corner_of(it.gc[ax], a.g.ds, u.scale) : __float2ll_rz(aq);
        f.d[ax] = (unsigned long long)v;
        if (runs) f.d[ax] = run_sum(f.d[ax], run);
      } else {  // the tile fixes the sign: magnitudes, below 2^32 for the run
        bad = bad || aq >= 134217728.0f;
        uint32_t v = __float2uint_rz(aq);
        if (runs) v = run_sum(v, run);
        f.d[ax] = (unsigned long long)v;
      }
    }
    f.own = !packed;
    if (packed) {
      const int c = count_axis(plane[0], plane[1], plane[2]);
      const unsigned long long n = (unsigned long long)f.n << kCountShift;
      if (c == 0) f.d[0] += n;
      else if (c == 1) f.d[1] += n;
      else if (c == 2) f.d[2] += n;
      else f.own = true;
    }
    const bool low = live && (frac[0] != 0.f || frac[1] != 0.f || frac[2] != 0.f);
    if (__any_sync(0xffffffffu, low)) {
      const uint32_t p = __shfl_sync(0xffffffffu, f.p, lane + __ffs((int)(run.lasts >> lane)) - 1);
      if (low) {
        if (note_fractions(a.b.low, &a.dc->n_low, p, frac[0], frac[1], frac[2])) atomicOr(a.b.info + p, kLowPoint);
        else bad = true;
      }
    }
    const uint32_t bads = __ballot_sync(0xffffffffu, bad);
    f.bad = ((bads >> run.first) & (0xffffffffu >> (31 - at))) != 0u;
    return f;
  }
  __device__ __forceinline__ bool done() const { return false; }
  __device__ __forceinline__ void apply(const Found& f) {
    if (f.p == kNoPoint) return;
    atomicAdd(a.b.sum[0] + f.p, f.d[0]);
    atomicAdd(a.b.sum[1] + f.p, f.d[1]);
    atomicAdd(a.b.sum[2] + f.p, f.d[2]);
    if (f.own) atomicAdd(a.b.members + f.p, f.n);
    if (f.bad) atomicOr(a.b.info + f.p, kBadPoint);
  }
};
__global__ void __launch_bounds__(256) tile_add_kernel(TileArgs a) {
  if (!tiles_on(a)) return;
  AddOp op{a, packed(a)};
  each_item(a, op);
}

// label + 32 map of training point p
__device__ __forceinline__ float label_word_of(const TileArgs& a, uint32_t p, int scan) {
  return (float)((a.b.key[p] & 31u) + 32u * (uint32_t)a.desc[scan].map_id);
}

// A thread per training point: the mean of its members, rounded once.  (A warp
// per tile instead saves the tile lookups but leaves the chip waiting for the
// fullest tiles: 72 against 26 us for 690k points.)
__global__ void __launch_bounds__(256) tile_finish_kernel(TileArgs a) {
  if (!tiles_on(a)) return;
  const uint32_t P = a.dc->n_train;
  for (uint32_t p = blockIdx.x * 256 + threadIdx.x; p < P; p += gridDim.x * 256) {
    const uint32_t info = a.b.info[p], key = a.b.key[p];
    const int4 tile = a.b.tiles[info & kRankMask];
    const int t[3] = {tile.x, tile.y, tile.z}, scan = tile.w;
    const uint32_t cell = key >> 5;
    unsigned long long sum[3] = {a.b.sum[0][p], a.b.sum[1][p], a.b.sum[2][p]};
    const AxisUnit units[3] = {axis_unit(t[0], a.g), axis_unit(t[1], a.g), axis_unit(t[2], a.g)};
    const int c = packed(a) ? count_axis(units[0].plane, units[1].plane, units[2].plane) : 3;
    uint32_t n;
    if (c == 3) {
      n = a.b.members[p];
    } else {
      const unsigned long long w = c == 0 ? sum[0] : (c == 1 ? sum[1] : sum[2]);
      n = (uint32_t)(w >> kCountShift);
#pragma unroll
      for (int ax = 0; ax < 3; ++ax)
        if (ax == c) sum[ax] &= (1ull << kCountShift) - 1ull;
    }
    bool ok = !(info & kBadPoint);
    float out[3] = {0.f, 0.f, 0.f};
    if (ok) {
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const AxisUnit u = units[ax];
        const long long rel = !u.plane && t[ax] < 0 ? -(long long)sum[ax] : (long long)sum[ax];
        const int gc = t[ax] * kTileEdge + (int)((cell >> (ax * kTileShift)) & (kTileEdge - 1));
        const long long corner = u.plane ? corner_of(gc, a.g.ds, u.scale) : 0ll;
        if (u.plane && n >= kMaxMembers) ok = false;
        const bool low = u.plane && (info & kLowPoint);
        if (n < (1u << 15) && !low) {  // |sum| < n 2^48
          const long long T = rel + (long long)n * corner;
          if (T) {
            float f = 0.f;
            ok = round_mean64(T < 0 ? (unsigned long long)(-T) : (unsigned long long)T, n, u.E, f) && ok;
            out[ax] = T < 0 ? -f : f;
          }
        } else {
          const unsigned long long mag = corner < 0 ? (unsigned long long)(-corner) : (unsigned long long)corner;
          U128 T;  // n corner + rel in two's complement, in units of 2^-40 with fractions
          T.lo = mag * n;
          T.hi = __umul64hi(mag, (unsigned long long)n);
          if (corner < 0) {
            T.lo = ~T.lo + 1ull;
            T.hi = ~T.hi + (T.lo == 0ull ? 1ull : 0ull);
          }
          u128_add(T, (unsigned long long)rel, rel < 0 ? ~0ull : 0ull);
          if (low) {
            T.hi = (T.hi << kLowBits) | (T.lo >> (64 - kLowBits));
            T.lo <<= kLowBits;
            const uint32_t nl = min(a.dc->n_low, kLowCap);
            for (uint32_t k = 0; k < nl; ++k)
              if (a.b.low[k].p == p && a.b.low[k].ax == (uint32_t)ax)
                u128_add(T, (unsigned long long)a.b.low[k].low, a.b.low[k].low < 0 ? ~0ull : 0ull);
          }
          const bool neg = (long long)T.hi < 0;
          if (neg) {
            T.lo = ~T.lo + 1ull;
            T.hi = ~T.hi + (T.lo == 0ull ? 1ull : 0ull);
          }
          if (T.lo | T.hi) {
            float f = 0.f;
            ok = round_mean(T, n, low ? u.E - kLowBits : u.E, f) && ok;
            out[ax] = neg ? -f : f;
          }
        }
      }
    }
    if (ok) {
      a.train[p] = make_float4(out[0], out[1], out[2], label_word_of(a, p, scan));
    } else {
      const uint32_t w = atomicAdd(&a.dc->n_wide, 1u);
      a.b.flagged[w] = p;
      a.b.start[w] = atomicAdd(&a.dc->n_gather, n);
      a.b.members[p] = n;
      a.b.info[p] = kBadPoint | w;
      // the label word waits in the point's place (coordinates follow)
      a.train[p] = make_float4(0.f, 0.f, 0.f, label_word_of(a, p, scan));
    }
  }
}

// ---------------------------------------------------------------- flagged points
// Members of the flagged points, each point's together.
struct GatherOp {
  struct Found {
    float x[3];
    uint32_t w;
  };
  const TileArgs& a;
  __device__ __forceinline__ Found look(const Item& it, const Run&) const {
    Found f{{it.x[0], it.x[1], it.x[2]}, kNoPoint};
    if (it.entry != kNoPoint) {
      const uint32_t info = __ldg(a.b.info + point_of(a, it));
      if (info & kBadPoint) f.w = info & ~kBadPoint;
    }
    return f;
  }
  __device__ __forceinline__ bool done() const { return false; }
  __device__ __forceinline__ void apply(const Found& f) {
    if (f.w != kNoPoint)
      a.b.gathered[atomicAdd(a.b.start + f.w, 1u)] = make_float4(f.x[0], f.x[1], f.x[2], 0.f);
  }
};
__global__ void __launch_bounds__(256) flagged_gather_kernel(TileArgs a) {
  if (a.dc->n_wide == 0u || !tiles_on(a)) return;
  GatherOp op{a};
  each_item(a, op);
}

// A warp per flagged point: the exact mean of its members.
__global__ void __launch_bounds__(256) flagged_mean_kernel(TileArgs a) {
  if (!tiles_on(a)) return;
  const uint32_t nw = a.dc->n_wide;
  for (uint32_t w = (blockIdx.x * 256 + threadIdx.x) >> 5; w < nw; w += gridDim.x * 8) {
    const uint32_t p = a.b.flagged[w], end = a.b.start[w];
    float out[3] = {0.f, 0.f, 0.f};
    cell_mean_warp(a.b.gathered, end - a.b.members[p], end, a.g, out);
    if ((threadIdx.x & 31u) == 0) a.train[p] = make_float4(out[0], out[1], out[2], a.train[p].w);
  }
}

// CTAs of a pass over the items (kPhases warps per 32 points, 8 warps a CTA), persistent
unsigned item_blocks(const MapState& m, int64_t total_n) {
  return (unsigned)std::max<int64_t>(
      1, std::min<int64_t>(((total_n + 31) / 32 * kPhases + 7) / 8, (int64_t)m.sm_count * m.tune.ingest_ctas_per_sm));
}

TileArgs tile_args(const MapState& m, int ns, uint32_t entries, const KeyFrame& kf, bool alone) {
  const Scratch& s = m.s;
  TileArgs a;
  a.g = m.g;
  a.b.dir = reinterpret_cast<uint32_t*>(s.keys);
  a.b.chunks = a.b.dir + entries;
  a.b.supers = a.b.chunks + (entries / kChunk + 1);
  a.b.groups = a.b.supers + ((entries / kChunk + 1) / kSuper + 1) * kSuperStep;
  a.b.cells = reinterpret_cast<uint2*>(s.sitems);
  a.b.tile_cap = (uint32_t)tile_capacity(s.s_cap);
  a.b.tiles = reinterpret_cast<int4*>(s.seg_start);
  a.b.counts = s.seg_start + 4 * (size_t)a.b.tile_cap;
  a.b.start = a.b.counts + a.b.tile_cap;
  a.b.sum[0] = reinterpret_cast<unsigned long long*>(s.items);
  a.b.sum[1] = a.b.sum[0] + s.s_cap;
  a.b.sum[2] = s.keys2;
  a.b.members = s.vals;
  a.b.info = s.vals2;
  a.b.key = s.flags;
  a.b.flagged = s.slow;
  a.b.low = reinterpret_cast<LowPart*>(s.hist);
  a.b.gathered = s.items;
  a.b.entries = entries;
  a.world = s.world;
  a.cnt = s.cnt;
  a.desc = s.desc;
  a.ns = ns;
  a.train = s.train;
  a.dc = m.dc;
  a.alone = alone;
  a.gate = tile_gate(m, ns, kf);
  // a beam's samples lie `step` apart, so at most 1 + sqrt(3) ds / step of them are in one cell
  // (widened for FP32 positions); a point's members are hits (one a beam) or samples, never both
  const double per_beam = 1.0 + std::floor(1.74 * (double)m.g.ds / (double)m.g.step);
  a.pack_limit = (uint32_t)((double)(1 << (64 - kCountShift)) / per_beam);
  return a;
}

}  // namespace

// Directory words of `entries` tiles, counts included.
static int64_t directory_words(int64_t entries, int64_t tile_cap) {
  const int64_t chunks = entries / kChunk + 1;
  return entries + chunks + (chunks / kSuper + 1) * kSuperStep + (tile_cap / kGroup + 1);
}

// Occupied tiles that the scratch of S items has room for (8 bytes a cell in 16 S bytes).
int64_t tile_capacity(int64_t S) { return S / (kCells / 2); }

bool tile_frame_fits(const MapState& m, int ns, const KeyFrame& kf) {
  const int64_t e = (int64_t)kf.ext[0] * kf.ext[1] * kf.ext[2];
  // the directory lies in 8 S bytes; cells stay below 2^22 on every axis (voxels below 2^20)
  if (m.prm.res > 3.9 * (m.prm.ds_res > 0 ? m.prm.ds_res : m.prm.res)) return false;
  return e > 0 && e <= kTileFrameMax && directory_words(e * ns, tile_capacity(m.s.s_cap)) <= 2 * m.s.s_cap && tile_capacity(m.s.s_cap) > 0;
}

TileGate tile_gate(const MapState& m, int ns, const KeyFrame& kf) {
  const int64_t cap = tile_capacity(m.s.s_cap);
  TileGate t;
  t.tile_cap = (uint32_t)cap;
  // as many flagged points as items find room in seg_start, behind the tiles
  t.item_cap = (uint32_t)std::max<int64_t>(0, m.s.s_cap - 5 * cap - 1);
  t.entries = (uint32_t)((int64_t)kf.ext[0] * kf.ext[1] * kf.ext[2] * ns);
  return t;
}

cudaError_t launch_tile_mark(MapState& m, int ns, int64_t total_n, const KeyFrame& kf, bool alone) {
  const uint32_t entries = (uint32_t)((int64_t)kf.ext[0] * kf.ext[1] * kf.ext[2] * ns);
  const TileArgs a = tile_args(m, ns, entries, kf, alone);
  const int64_t words = directory_words(entries, a.b.tile_cap);
  if (words <= kClearAlways) {
    const cudaError_t e = cudaMemsetAsync(a.b.dir, 0, sizeof(uint32_t) * (size_t)words, m.stream);
    if (e != cudaSuccess) return e;
  } else {
    const unsigned blocks = (unsigned)std::min<int64_t>((words / 4 + 255) / 256 + 1, (int64_t)m.sm_count * 8);
    tile_clear_kernel<<<blocks, 256, 0, m.stream>>>(a, (uint32_t)words);
    m.launches += 1;
  }
  tile_mark_kernel<<<item_blocks(m, total_n), 256, 0, m.stream>>>(a);
  m.launches += 1;
  return cudaGetLastError();
}

cudaError_t launch_tiles(MapState& m, int ns, int64_t total_n, const KeyFrame& kf, int64_t nitems) {
  const uint32_t entries = (uint32_t)((int64_t)kf.ext[0] * kf.ext[1] * kf.ext[2] * ns);
  const TileArgs a = tile_args(m, ns, entries, kf, false);
  const unsigned blocks = item_blocks(m, total_n);
  const int64_t sms = m.sm_count;
  tile_rank_kernel<<<(unsigned)std::min<int64_t>(entries / kChunk + 1, 8 * sms), 256, 0, m.stream>>>(a);
  tile_masks_kernel<<<blocks, 256, 0, m.stream>>>(a);
  const int64_t tiles = std::min<int64_t>(a.b.tile_cap, nitems);
  const unsigned tblocks = (unsigned)std::max<int64_t>(1, std::min<int64_t>((tiles + 7) / 8, 8 * sms));
  tile_counts_kernel<<<tblocks, 256, 0, m.stream>>>(a);
  tile_offsets_kernel<<<tblocks, 256, 0, m.stream>>>(a);
  tile_add_kernel<<<blocks, 256, 0, m.stream>>>(a);
  tile_finish_kernel<<<(unsigned)std::max<int64_t>(1, std::min<int64_t>((nitems + 255) / 256, 8 * sms)), 256, 0, m.stream>>>(a);
  flagged_gather_kernel<<<blocks, 256, 0, m.stream>>>(a);
  flagged_mean_kernel<<<(unsigned)sms, 256, 0, m.stream>>>(a);
  m.launches += 8;
  return cudaGetLastError();
}

}  // namespace sbki
