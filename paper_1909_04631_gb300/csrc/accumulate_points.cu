// Step a5, point-major form: one warp per training point adds
// sigma0 f(|c_v - x_i| / l) (Eq. alpha_kernel, Eq. kernel) into every voxel
// centre within l, with one global floating-point reduction per pair.
//
// Candidate voxels come from a static table.  Split the voxel of a point into
// 8x8x8 parts by the point's sub-voxel position; for each part the table
// lists every offset (dx, dy, dz) (relative to the point's voxel) whose centre
// can lie within l of some position in that part, widened by 0.001 voxel on
// every side (so FP32 rounding of the position cannot pick too small a list).
// For l = 3 res a list has at most 136 entries (94 % of them at most 128, four
// sweeps of 32), against ~113 in support.
// Per point the warp
//   1. forms the compensated offsets E0 = c(v0) - x of the point's own voxel
//      centre (hi + lo per axis) and fills two per-warp lookup tables in
//      shared memory: X[dx] = (ex^2, x-part of the voxel address) and
//      YZ[dy, dz] = (ey^2 + ez^2, y/z-part of the voxel address), where an
//      address part holds the block-offset digit (base 3 per axis) in its low
//      byte and the in-block index above it, so the two parts add up to the
//      full address without carries; and the pointers to class y_i of the
//      (at most 27) blocks the ball can reach;
//   2. sweeps its part's list, 32 candidates at a time (fully unrolled for
//      the common list lengths): a list entry holds the byte offsets of its X
//      and YZ rows, so d^2 and the address are two shared-memory loads and two
//      adds; the FP32 test (re-decided in FP64 inside the relative band around
//      l^2), the kernel value and red.global.add.f32 into alpha.  Padding
//      entries point at an X row with d^2 = 1e30.
// Training points arrive sorted by their downsampling cell, so the warps in
// flight at any moment update a compact region of the map (L2 locality).
// Blocks allocated by this update are zero-filled before (fresh_fill_kernel).
#include <algorithm>
#include <type_traits>
#include <climits>
#include <cmath>
#include <vector>

#include "kernel_value.cuh"
#include "pair_rows.cuh"

namespace sbki {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kAxisMax = 15;             // offsets per axis: 2R + 1 <= 15
constexpr int kYZMax = kAxisMax * kAxisMax;

struct PtArgs {
  Geom g;
  const float4* train;
  const unsigned long long* hkeys;
  const int32_t* hvals;
  int64_t hash_cap;
  float* alpha;
  int32_t* pairs;
  const uint32_t* ctab;  // [kParts^3][tpad] (X byte offset | YZ byte offset << 8 | dy << 19 | dz << 23)
  const int32_t* clen;   // [kParts^3] entries of each list
  int tpad;              // entries per list (multiple of 32)
  int R;                 // offsets per axis span [-R, R]
  uint32_t recip_na;     // small_recip(2R + 1)
  int chunk;             // consecutive training points per warp at most (fast form)
  int32_t sink;          // spare pool block that absent neighbour blocks point at
  const uint16_t* ftab;  // fast form: [tables][kFastLists][list_pad] entries, then a list of padding entries
  const int32_t* flen;   // [tables][kFastLists] entries of each list
  int list_pad;          // entries per list (a multiple of 16, at most kFastPad)
  uint32_t pad_list;     // first entry of the list of padding entries
  float band;            // half-width of the re-decision band around l^2
  const uint32_t* ownslot;  // fast form: per training point the hash slot of its own block (touched-block pass)
  const uint32_t* nbrslot;  // fast form: [hash_cap][32] per own block the hash slots of its touched neighbours
  const int32_t* softidx;   // soft labels (fast form), or null: per training point its weight row, or -1
  const float* wsoft;       // weight rows [.][K+1]
  int tab_of[kMaxClasses];  // per-class supports (fast form): each class's list table, or -1 (not this form)
  float band_k[kMaxClasses];  // per-class supports: half band of each class
  DevCounters* dc;
};

struct WarpTables {
  float2 x[kAxisMax + 1];  // (e_x^2, address part as int bits); entry 2R+1 is the padding row
  float2 yz[kYZMax];
  float* blk[27];          // alpha + (pool * (K+1) + y_i) * B^3 (pool = the spare block when absent)
  int32_t* cnt[27];        // pair counts of the block (tracking only)
};

// One candidate per lane, branch-free except for the (rare, warp-uniform)
// FP64 re-decision: every lane evaluates the kernel and the reduction is
// predicated.  Every list entry (padding included) yields a block digit in
// 0..26, so the block-pointer load is always in range.  A neighbour block
// that is not in the map holds no voxel within l of any training point of
// this update (the touched-block pass applies the same membership test and
// allocated every block that does), so no in-support pair reaches it; its
// pointer names the spare block after the pool, so the reduction needs no
// null test.  s0 is the point's class scale sigma0 * sigma0_scale[y_i].
// Returns 1 for an in-support pair.
template <bool kTrack>
__device__ __forceinline__ uint32_t candidate(const PtArgs& a, const WarpTables& t, uint32_t ent, const int v0[3],
                                              const float4& p, float s0) {
  const Geom& g = a.g;
  const float2 ex = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(t.x) + (ent & 0xffu));
  const float2 eyz = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(t.yz) + ((ent >> 8) & 0x7ffu));
  const float d2 = __fadd_rn(ex.x, eyz.x);
  const int pk = __float_as_int(ex.y) + __float_as_int(eyz.y);
  bool in = d2 < g.l2_lo;
  const bool band = !in && d2 < g.l2_hi;
  if (__any_sync(0xffffffffu, band)) {
    if (band)
      in = in_support64_call(v0[0] + (int)((ent & 0xffu) >> 3) - a.R, v0[1] + (int)((ent >> 19) & 15u) - a.R,
                             v0[2] + (int)((ent >> 23) & 15u) - a.R, p.x, p.y, p.z, g.res64, g.l2_64);
  }
  if (g.assoc) in = in && ((kFaceDigits >> (pk & 0xff)) & 1u);  // extended block: own block and face neighbours
  float* base = t.blk[pk & 0xff];
  const float d = d2 * rsqrtf(fmaxf(d2, 1e-30f));
  const float u = fmaxf(__fmaf_rn(-d, g.inv_l, 1.0f), 0.0f);
  const float w = u * u;
  red_add_if(in, base + (pk >> 8), s0 * (w * w * u * kernel_q(w)));
  if (kTrack) red_add_if(in, t.cnt[pk & 0xff] + (pk >> 8), 1);
  return in ? 1u : 0u;
}

// kNit > 0: lists of exactly kNit x 32 entries, unrolled; 0: any length
template <bool kTrack, int kNit>
__global__ void __launch_bounds__(kThreads, 4) accumulate_points_kernel(PtArgs a) {
  __shared__ WarpTables s_tab[kWarps];
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const uint32_t gw = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const uint32_t nw = (gridDim.x * blockDim.x) >> 5;
  const int R = a.R, na = 2 * R + 1;
  WarpTables& t = s_tab[wid];
  uint32_t npairs = 0;
  if (a.dc->err != 0) return;
  const uint32_t P = a.dc->n_train;
  if (lane == 0) t.x[na] = make_float2(kFar, __int_as_float(0));
  float4 pnext = gw < P ? a.train[gw] : make_float4(0.f, 0.f, 0.f, 0.f);
  for (uint32_t i = gw; i < P; i += nw) {
    const float4 p = pnext;
    if (i + nw < P) pnext = a.train[i + nw];  // in flight while this point is processed
    const int lm = label_of(p.w);  // label + 32 * map
    const int label = lm & ((1 << kLabelBits) - 1), map = lm >> kLabelBits;
    const float s0 = g.sigma0_k[label];  // class label's kernel scale
    const PointFrame f = point_frame(p.x, p.y, p.z, R, g);
    const uint32_t* tab = a.ctab + f.part * a.tpad;
    const int len = __ldg(a.clen + f.part);
    // X rows
    if (lane < na) {
      const float e = centre_offset_at(lane - R, f.hi[0], f.lo[0], g);
      t.x[lane] = make_float2(__fmul_rn(e, e), __int_as_float(xpart(f, lane, R, g)));
    }
    // Y rows in lanes 0..15, Z rows in lanes 16..31, combined into YZ rows by shuffles
    float sq1 = 0.f;
    int pk1 = 0;
    {
      const int ax = 1 + (lane >> 4), j = min(lane & 15, na - 1);
      const float e = centre_offset_at(j - R, f.hi[ax], f.lo[ax], g);
      const int v = f.v0[ax] + j - R, m = g.B - 1;
      sq1 = __fmul_rn(e, e);
      pk1 = ax == 1 ? (3 * ((v >> g.B_shift) - f.blo[1])) | ((v & m) << (g.B_shift + 8))
                    : (9 * ((v >> g.B_shift) - f.blo[2])) | ((v & m) << (2 * g.B_shift + 8));
    }
    for (int q0 = 0; q0 < na * na; q0 += 32) {  // uniform trip count: full-warp shuffles
      const int q = min(q0 + lane, na * na - 1);
      const int jy = (int)small_div((uint32_t)q, a.recip_na), jz = q - jy * na;
      const float sy = __shfl_sync(0xffffffffu, sq1, jy), sz = __shfl_sync(0xffffffffu, sq1, 16 + jz);
      const int py = __shfl_sync(0xffffffffu, pk1, jy), pz = __shfl_sync(0xffffffffu, pk1, 16 + jz);
      if (q0 + lane < na * na) t.yz[q] = make_float2(__fadd_rn(sy, sz), __int_as_float(py + pz));
    }
    // blocks the ball can reach: digit (bx, by, bz) in base 3
    if (lane < 27) {
      const int32_t pool = digit_pool(f, lane, map, a.hkeys, a.hvals, a.hash_cap);
      t.blk[lane] = a.alpha + ((size_t)(pool >= 0 ? pool : a.sink) * g.K1 + label) * g.B3;
      if (kTrack) t.cnt[lane] = a.pairs + (size_t)(pool >= 0 ? pool : a.sink) * g.B3;
    }
    __syncwarp();
    if (kNit > 0) {
      uint32_t ent[kNit > 0 ? kNit : 1];
#pragma unroll
      for (int it = 0; it < kNit; ++it) ent[it] = it * 32 < len ? __ldg(tab + it * 32 + lane) : 0u;
#pragma unroll
      for (int it = 0; it < kNit; ++it)
        if (it * 32 < len) npairs += candidate<kTrack>(a, t, ent[it], f.v0, p, s0);  // warp-uniform
    } else {
      for (int k = lane; k - lane < len; k += 32) npairs += candidate<kTrack>(a, t, __ldg(tab + k), f.v0, p, s0);
    }
    __syncwarp();  // the tables are rewritten for the next point
  }
  for (int o = 16; o > 0; o >>= 1) npairs += __shfl_down_sync(0xffffffffu, npairs, o);
  if (lane == 0) atomicAdd(&a.dc->pairs, (unsigned long long)npairs);
}

// The same update for 2R + 1 <= 7 (l below 3.5 voxels): half a warp per point,
// two voxels adjacent in x per lane.
//
// A warp takes a chunk of consecutive training points (sorted by tile, so
// mostly one block) from a work queue and forms their rows in groups of
// kGroup, four lanes per point (two for x, one each for y and z), into the
// point's 256-byte slot in shared memory:
//   X  four pairs of voxels from the even voxel at or below v0 - R on: the two
//      squared offsets and an address part (16 bytes a pair);
//   Y  per offset -R..R (squared offset, address part), and a padding row;
//   Z  the same; its parts carry the point's class row, label * B^3;
//   the point's list, class and block.
// An address part holds the block digit of its axis (4 dx, 12 dy, 36 dz, each
// in 0..2: a byte offset into the block table) in its top byte and the voxel's
// in-block index below it, so the three parts of a pair add up to
// (4 digit) << 24 | (label B^3 + in-block index).  A pair lies in one block
// (block edges are even).
//
// The point's sub-voxel part (kFastParts per axis) picks the list of pairs that
// can hold a voxel within l (70 to 88 for l = 3 res, x fastest, so the lanes of
// one voxel row reach the same 32 bytes).  A point in the upper half of its
// voxel along y or z writes its rows in reverse order and takes the mirrored
// list; along x, where the pairs' alignment breaks the symmetry, an odd v0 - R
// is the mirror image of an even one.  That leaves kFastLists lists of 16-bit
// entries, 24 KB for l = 3 res, which each CTA keeps in shared memory.  A list entry
// names the pair's X, Y and Z rows so that each row address is one or two
// operations on the slot's 256-byte aligned address.
// The block table holds, per digit, the first alpha element of the block (the
// pool slot times (K+1) B^3) minus the digit's top byte, so table entry +
// summed parts is the alpha element; it changes only when the half warp's
// point is in another block.  Both voxels' kernels are evaluated in packed
// FP32; a voxel past l gets u = 0 (a saturating FMA), hence adds zero, and a
// pair with a voxel within l is one 8-byte vector reduction.  Membership is the
// sign of d^2 - l^2, re-decided in FP64 where |d^2 - l^2| is inside the band.
//
// Why so: one voxel per lane (lists of up to 160, a warp per point) takes three
// row loads, a base load and a scalar reduction per voxel, and was bound by the
// L1 data pipe at 58 wavefronts a point; whole columns of voxels per lane
// evaluate 7 voxels per lane and round where 3.5 are within l, and were bound
// by issue (325 instructions a point, 236 us for 690k points).  Here the rows'
// loads serve two voxels: 29 shared-load wavefronts a point.  Stage times,
// one voxel per lane -> this form: 188k points of a small region 85 -> 70 us,
// 690k of a 64 x 2048 street scan 202 -> 198, softmax labels 479 -> 422,
// per-class l (the widest no longer left to the weighted form) 267 -> 192.
// Of the 178 us alone (147M warp instructions, issue 70 %, L1 data pipe 67 %)
// the row set-up takes 45, the reductions 26.
struct __align__(256) FastWarp {
  unsigned char slot[kGroup][kSlotBytes];
  uint32_t btab[2][64];                 // per half warp: alpha element base per block digit (27 used)
};
struct __align__(256) FastWarpTrack : FastWarp {
  uint32_t ptab[2][64];                 // the same for the pair counts
};
template <typename Base>
struct __align__(256) FastWarpSoft : Base {
  float cw[kGroup][kMaxClasses];        // soft labels: per point sigma0 s_k w^k by class
  uint32_t cmask[kGroup];               // its classes with a weight
  int soft[kGroup];                     // 1: the point has a weight row
};

// one reduction of 8 aligned bytes where p != 0 (each element is added atomically)
__device__ __forceinline__ void red_add2_if(uint32_t p, float* addr, float2 v) {
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %0, 0;\n\t@q red.global.add.v2.f32 [%1], {%2, %3};\n\t}" ::"r"(p),
               "l"(addr), "f"(v.x), "f"(v.y)
               : "memory");
}

// Soft labels (kSoft, reading K15): a point with a weight row forms its rows
// for class 0 with s0 = 1, and each of its in-support pairs adds
// f(d/l) sigma0 s_k w^k into every class k with a nonzero weight; a point
// without one (free samples) is a hard class-0 point.
// Per-class supports (kLk, reading K16): a point's list comes from the table
// of its class's support l_k, its membership test and kernel use l_k; points
// of a class without a table are left to the weighted form.
template <bool kTrack, bool kFace, bool kSoft = false, bool kLk = false>
__global__ void __launch_bounds__(kThreads, 4) accumulate_points_fast_kernel(PtArgs a) {
  using Plain = typename std::conditional<kTrack, FastWarpTrack, FastWarp>::type;
  using Warp = typename std::conditional<kSoft, FastWarpSoft<Plain>, Plain>::type;
  __shared__ Warp s_w[kWarps];
  extern __shared__ __align__(16) uint16_t s_lists[];  // common support: the lists and the padding list
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  Warp& W = s_w[wid];
  const int R = a.R;
  if (a.dc->err != 0) return;
  if ((smem_addr(&W) & 255u) != 0u) {  // the byte permutes need 256-byte aligned slots and tables
    if (lane == 0) set_error(a.dc, SBKI_ERR_CUDA);
    return;
  }
  // the padding rows, written once; a half without a point reads X row 0, Z row 0 and the
  // padding row of its slot, so the slots start at zero (finite, block digit 0)
  for (int e = lane; e < kGroup * kSlotBytes / 4; e += 32) reinterpret_cast<float*>(W.slot)[e] = 0.0f;
  __syncwarp();
  if (lane < kGroup) *reinterpret_cast<float*>(W.slot[lane] + kYRows + 8 * kFastAxis) = kFar;
  __syncwarp();
  if (!kLk) {
    const int n16 = list_entries(1, a.list_pad) / 8;
    for (int e = threadIdx.x; e < n16; e += kThreads)
      reinterpret_cast<uint4*>(s_lists)[e] = __ldg(reinterpret_cast<const uint4*>(a.ftab) + e);
    __syncthreads();
  }
  const uint32_t lists = smem_addr(s_lists);
  const uint32_t P = a.dc->n_train;
  const int half = lane >> 4, hl = lane & 15;
  const uint32_t slot0 = smem_addr(&W.slot[0][0]) + (uint32_t)half * kSlotBytes;
  const uint32_t btab0 = smem_addr(&W.btab[0][0]);
  // this lane's point of a group, and its role there: 0, 1 the halves of X, 2 Y, 3 Z
  const int gl = lane >> 2, role = lane & 3, ax = max(role - 1, 0);
  const uint32_t K1B3 = (uint32_t)(g.K1 * g.B3);
  uint32_t cown = 0xffffffffu;  // own block the half's table belongs to
  uint32_t npairs = 0;
  // Chunk: about three per warp, at most a.chunk.  Longer ones refill the block
  // table less often, shorter ones balance the warps (and the queue's one
  // address takes about 1 ns per claim): 16 / 32 / 48 points took 76 / 87 / 97 us
  // for 188k points and 228 / 206 / 197 us for 690k.
  const uint32_t warps = gridDim.x * kWarps;
  const uint32_t chunk = min((uint32_t)a.chunk, max(P / (3u * warps) / kGroup, 2u) * kGroup);
  uint32_t c = blockIdx.x * kWarps + (uint32_t)wid;  // the first chunk needs no claim
  while (c * chunk < P) {
    uint32_t cn = 0;  // next chunk, fetched while this one is processed
    if (lane == 0) cn = warps + atomicAdd(&a.dc->acc_next, 1u);
    const uint32_t c1 = min(P, c * chunk + chunk);
    for (uint32_t g0 = c * chunk; g0 < c1; g0 += kGroup) {
      const uint32_t gn = min(c1 - g0, (uint32_t)kGroup);  // warp-uniform
      // 1. rows of every point of the group
      int pt = 0, lw = 0, srow = -1;
      uint32_t own = 0u;
      if (gl < (int)gn) {
        const float4 p = a.train[g0 + gl];
        own = __ldg(a.ownslot + g0 + gl);
        if (kSoft) srow = __ldg(a.softidx + g0 + gl);
        const AxisFrame f = axis_frame(ax == 0 ? p.x : (ax == 1 ? p.y : p.z), g);
        lw = label_of(p.w);
        if (kSoft && srow >= 0) lw &= ~((1 << kLabelBits) - 1);  // class rows come per class in the sweep
        const uint32_t cls = (uint32_t)((lw & ((1 << kLabelBits) - 1)) * g.B3);
        pt = form_rows<true>(W.slot[gl], gl, role, f, cls, R, g);
      }
      const int pty = __shfl_sync(0xffffffffu, pt, lane | 2), ptz = __shfl_sync(0xffffffffu, pt, lane | 3);
      if (role == 0 && gl < (int)gn) {
        const int label = lw & ((1 << kLabelBits) - 1);
        const int tb = kLk ? a.tab_of[label] : 0;  // the table of the point's class support, or none
        const int list = tb * kFastLists + pt + kFastParts * (pty + kFastParts / 2 * ptz);
        const uint32_t rounds = tb >= 0 ? (uint32_t)(__ldg(a.flen + list) + 15) >> 4 : 0u;
        *reinterpret_cast<uint4*>(W.slot[gl] + kScalars) =
            make_uint4(tb >= 0 ? (uint32_t)(list * a.list_pad) : a.pad_list, (uint32_t)lw | (rounds << 16),
                       __float_as_uint((kSoft && srow >= 0) ? 1.0f : g.sigma0_k[label]), own);
      }
      if constexpr (kSoft) {  // class factors sigma0 s_k w^k of the group's soft points
        for (uint32_t k = 0; k < gn; ++k) {
          const int row = __shfl_sync(0xffffffffu, srow, 4 * k);
          float ck = 0.0f;
          if (row >= 0 && lane < g.K1) ck = g.sigma0_k[lane] * __ldg(a.wsoft + (size_t)row * g.K1 + lane);
          const unsigned cm = __ballot_sync(0xffffffffu, ck != 0.0f);
          if (lane < g.K1) W.cw[k][lane] = ck;
          if (lane == 0) {
            W.cmask[k] = cm;
            W.soft[k] = row >= 0 ? 1 : 0;
          }
        }
      }
      __syncwarp();
      // 2. block tables.  Points come sorted by tile, so most groups lie in one block: then both
      //    halves read one table, refilled when the block changes
      auto fill_digit = [&](int t, uint32_t slot_of_own, int d) {
        // a digit no point of this block touched holds a stale slot; no
        // in-support pair uses it (every reduction is predicated on membership)
        const uint32_t hs = a.nbrslot[(size_t)slot_of_own * 32 + d] & (uint32_t)(a.hash_cap - 1);
        const int32_t pool = a.hvals[hs];
        const uint32_t pb = (uint32_t)(pool >= 0 ? pool : a.sink);
        W.btab[t][d] = pb * K1B3 - ((4u * (uint32_t)d) << 24);
        if constexpr (kTrack) W.ptab[t][d] = pb * (uint32_t)g.B3 - ((4u * (uint32_t)d) << 24);
      };
      const uint32_t own0 = __shfl_sync(0xffffffffu, own, 0);
      const bool one = __all_sync(0xffffffffu, own == own0 || gl >= (int)gn);  // warp-uniform
      if (one && own0 != __shfl_sync(0xffffffffu, cown, 0)) {
        if (half == 0) cown = own0;
        if (lane < 27) fill_digit(0, own0, lane);
        __syncwarp();
      }
      const uint32_t btab = one ? btab0 : btab0 + (uint32_t)half * (uint32_t)sizeof(W.btab[0]);
      // 3. two points at a time, one per half warp
      for (uint32_t k0 = 0; k0 < gn; k0 += 2) {
        const uint32_t slot = slot0 + k0 * kSlotBytes, k = k0 + (uint32_t)half;
        const bool have = k < gn;
        const uint4 sv = lds_u4(slot + kScalars);
        // this lane's entries of the point's list, one per round
        const uint32_t list = (have ? sv.x : a.pad_list) + (uint32_t)hl;
        auto entry = [&](uint32_t r) {
          return kLk ? (uint32_t)__ldg(a.ftab + list + 16 * r) : lds_u16(lists + 2 * list + 32 * r);
        };
        if (!one) {  // warp-uniform: a half's point may be in another block than its table
          const bool moved = have && sv.w != cown;
          if (__any_sync(0xffffffffu, moved)) {
            if (moved) {
              cown = sv.w;
              for (int d = hl; d < 27; d += 16) fill_digit(half, cown, d);
            }
            __syncwarp();
          }
        }
        const uint32_t mine = have ? (sv.y >> 16) & 0xffu : 0u;  // rounds of this half's point
        const uint32_t rounds = max(mine, __shfl_xor_sync(0xffffffffu, mine, 16));
        const int label = (int)(sv.y & ((1u << kLabelBits) - 1u));
        const float s0 = __uint_as_float(sv.z);
        const float l2 = kLk ? __fmul_rn(0.5f, __fadd_rn(g.l2k_lo[label], g.l2k_hi[label])) : g.l2;
        const float band = kLk ? a.band_k[label] : a.band;
        const float ninv = kLk ? -g.inv_lk[label] : -g.inv_l;
        const float2 nl2 = make_float2(-l2, -l2), s02 = make_float2(s0, s0);
        uint32_t bits = 0u;  // one per voxel seen, 1 within l
        // one pair per lane: its d^2 and address, its membership into `bits`
        struct Pair {
          float2 d2, t;
          uint32_t pk;
        };
        auto rows_of = [&](uint32_t e) {
          Pair p;
          const uint32_t xa = slot | ((e >> 2) & 0x30u);
          const float2 rx = lds_f2(xa), ry = lds_f2((slot | (e & 0x38u)) + kYRows),
                       rz = lds_f2(__byte_perm(e, slot, 0x7651));
          const float rd = __fadd_rn(ry.x, rz.x);
          p.d2 = __fadd2_rn(make_float2(rd, rd), rx);
          p.pk = lds_u32(xa + 8) + __float_as_uint(ry.y) + __float_as_uint(rz.y);
          p.t = __fadd2_rn(p.d2, nl2);
          return p;
        };
        auto near = [](const Pair& p) { return fminf(fabsf(p.t.x), fabsf(p.t.y)); };
        auto member = [&](const Pair& p) {
          return __funnelshift_l(__float_as_uint(p.t.y), __float_as_uint(p.t.x) >> 31, 1);
        };
        // FP64 decisions of the voxels inside the band; one found outside gets a d^2 past l^2
        auto redecide = [&](uint32_t e, Pair& p, uint32_t& in) {
          const double l264 = kLk ? g.l2k_64[label] : g.l2_64;
          if (fabsf(p.t.x) <= band) {
            const bool i = band_decide(e, 0, a.train, g0 + k, R, g, l264);
            in = (in & ~2u) | (i ? 2u : 0u);
            if (!i) p.d2.x = 4.0f * l2;
          }
          if (fabsf(p.t.y) <= band) {
            const bool i = band_decide(e, 1, a.train, g0 + k, R, g, l264);
            in = (in & ~1u) | (i ? 1u : 0u);
            if (!i) p.d2.y = 4.0f * l2;
          }
        };
        // kernels f = u^5 Q(u^2), u = 1 - d / l (0 past l), times sigma0 s_k, added where `in` (bit 1: the
        // first voxel, bit 0: the second) is not 0
        auto add_pair = [&](const Pair& p, uint32_t in) {
          if (kFace && !((kFaceDigits >> (p.pk >> 26)) & 1u)) in = 0u;  // own block and face neighbours only
          const float2 u = make_float2(__saturatef(__fmaf_rn(sqrt_approx(p.d2.x), ninv, 1.0f)),
                                       __saturatef(__fmaf_rn(sqrt_approx(p.d2.y), ninv, 1.0f)));
          const float2 w = __fmul2_rn(u, u);
          const float2 v = __fmul2_rn(__fmul2_rn(__fmul2_rn(w, w), __fmul2_rn(u, s02)), kernel_q2(w));
          float* dst = a.alpha + (lds_u32(__byte_perm(p.pk, btab, 0x7653)) + p.pk);
          bool spread = false;
          if constexpr (kSoft) {
            if (W.soft[k & (kGroup - 1)]) {  // uniform over the half: every class with a weight
              for (unsigned cl = in ? W.cmask[k & (kGroup - 1)] : 0u; cl; cl &= cl - 1u) {
                const int kc = __ffs((int)cl) - 1;
                const float ck = W.cw[k & (kGroup - 1)][kc];
                red_add2_if(1u, dst + (uint32_t)kc * (uint32_t)g.B3, __fmul2_rn(v, make_float2(ck, ck)));
              }
              spread = true;
            }
          }
          red_add2_if(spread ? 0u : in, dst, v);
          if constexpr (kTrack) {
            int32_t* pc = a.pairs + (lds_u32(__byte_perm(p.pk, btab + (uint32_t)sizeof(W.btab), 0x7653)) + p.pk -
                                     (uint32_t)(label * g.B3));
            red_add_if(in & 2u, pc, 1);
            red_add_if(in & 1u, pc + 1, 1);
          }
          return in;
        };
        // rounds in twos (independent chains, one vote), then the odd one
        uint32_t r = 0;
        for (; r + 2 <= rounds; r += 2) {  // warp-uniform
          const uint32_t ea = entry(r), eb = entry(r + 1);
          Pair pa = rows_of(ea), pb = rows_of(eb);
          uint32_t ina = member(pa), inb = member(pb);
          if (__any_sync(0xffffffffu, fminf(near(pa), near(pb)) <= band)) {
            redecide(ea, pa, ina);
            redecide(eb, pb, inb);
          }
          ina = add_pair(pa, ina);
          inb = add_pair(pb, inb);
          bits = (bits << 4) | (ina << 2) | inb;
        }
        if (r < rounds) {
          const uint32_t ea = entry(r);
          Pair pa = rows_of(ea);
          uint32_t ina = member(pa);
          if (__any_sync(0xffffffffu, near(pa) <= band)) redecide(ea, pa, ina);
          bits = (bits << 2) | add_pair(pa, ina);
        }
        npairs += (uint32_t)__popc(bits);
      }
      __syncwarp();  // the slots are rewritten by the next group
    }
    c = __shfl_sync(0xffffffffu, cn, 0);
  }
  for (int o = 16; o > 0; o >>= 1) npairs += __shfl_down_sync(0xffffffffu, npairs, o);
  if (lane == 0) atomicAdd(&a.dc->pairs, (unsigned long long)npairs);
}

// Blocks created by this update start at zero (and so do their pair counts).
__global__ void fresh_fill_kernel(const uint32_t* fresh, const int32_t* hvals, float* alpha, int32_t* pairs, int K1B3,
                                  int B3, DevCounters* dc) {
  if (dc->err != 0) return;
  if (blockIdx.x == 0 && threadIdx.x == 0) dc->acc_next = 0;  // work queue of the accumulation launched next
  const uint32_t n_new = dc->n_new;
  for (uint32_t f = blockIdx.x; f < n_new; f += gridDim.x) {
    const int32_t pl = hvals[fresh[f]];
    float4* dst = reinterpret_cast<float4*>(alpha + (size_t)pl * K1B3);
    for (int e = threadIdx.x; e < K1B3 / 4; e += blockDim.x) dst[e] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (pairs)
      for (int e = threadIdx.x; e < B3; e += blockDim.x) pairs[(size_t)pl * B3 + e] = 0;
  }
}

// min over phi in [lo, hi] of |d + 1/2 - phi| (voxel units)
double min_axis_distance(int d, double lo, double hi) {
  const double c = d + 0.5;
  if (c >= lo && c <= hi) return 0.0;
  return std::min(std::fabs(c - lo), std::fabs(c - hi));
}

// Candidate offsets of each of parts^3 sub-voxel parts: every (dx, dy, dz) whose
// voxel centre can lie within l of some position in the part, the part widened
// by delta = 1e-3 voxel on every side (far above the FP32 error of the sub-voxel
// position, ~1e-6 voxel), so a point's list always holds its ball.  Offsets are
// packed as (dx + R) | (dy + R) << 4 | (dz + R) << 8; returns R.
int candidate_lists(double lr, int parts, std::vector<std::vector<int32_t>>& lists) {
  const double delta = 1e-3;
  const int R = (int)std::ceil(lr + 0.5 + delta);
  const int n = parts * parts * parts;
  lists.assign(n, {});
  for (int t = 0; t < n; ++t) {
    const int pt[3] = {t % parts, (t / parts) % parts, t / (parts * parts)};
    for (int dz = -R; dz <= R; ++dz)
      for (int dy = -R; dy <= R; ++dy)
        for (int dx = -R; dx <= R; ++dx) {
          const int d[3] = {dx, dy, dz};
          double m2 = 0.0;
          for (int a = 0; a < 3; ++a) {
            const double md =
                min_axis_distance(d[a], (double)pt[a] / parts - delta, (double)(pt[a] + 1) / parts + delta);
            m2 += md * md;
          }
          if (m2 < lr * lr * (1.0 + 1e-5)) lists[t].push_back((dx + R) | ((dy + R) << 4) | ((dz + R) << 8));
        }
  }
  return R;
}

// Pairs of voxels adjacent in x of an even v0 - R, per sub-voxel part
// (kFastParts along x, the lower half of them along y and z): pair jx holds the
// offsets -R + 2 jx and the one after it; a list takes every pair with a voxel
// whose centre can lie within l of a position in the part, widened as above.
// Entries are packed as jx | (dy + R) << 4 | (dz + R) << 8, x fastest.
void pair_lists(double lr, int R, std::vector<std::vector<int32_t>>& lists) {
  const double delta = 1e-3;
  const int n = kFastParts;
  auto dist = [&](int d, int part) {
    return min_axis_distance(d, (double)part / n - delta, (double)(part + 1) / n + delta);
  };
  lists.assign(kFastLists, {});
  for (int t = 0; t < kFastLists; ++t) {
    const int px = t % n, py = (t / n) % (n / 2), pz = t / (n * (n / 2));
    for (int dz = -R; dz <= R; ++dz)
      for (int dy = -R; dy <= R; ++dy)
        for (int jx = 0; jx < 4; ++jx) {
          const int dx = -R + 2 * jx;
          const double mx = std::min(dist(dx, px), dist(dx + 1, px)), my = dist(dy, py), mz = dist(dz, pz);
          if (mx * mx + my * my + mz * mz < lr * lr * (1.0 + 1e-5))
            lists[t].push_back(jx | ((dy + R) << 4) | ((dz + R) << 8));
        }
  }
}

// the largest offset whose voxel centre can lie within l of a position in the voxel
int largest_offset(double lr) {
  int R = 0;
  for (int d = 0; d <= 15; ++d)
    if (min_axis_distance(d, -1e-3, 1.001) < lr * (1.0 + 1e-5) || min_axis_distance(-d, -1e-3, 1.001) < lr * (1.0 + 1e-5))
      R = d;
  return R;
}

template <typename T>
cudaError_t upload_lists(const std::vector<T>& flat, const std::vector<int32_t>& len, T** tab, int32_t** lens) {
  cudaError_t e = cudaMalloc(tab, sizeof(T) * flat.size());
  if (e != cudaSuccess) return e;
  e = cudaMalloc(lens, sizeof(int32_t) * len.size());
  if (e != cudaSuccess) return e;
  e = cudaMemcpy(*lens, len.data(), sizeof(int32_t) * len.size(), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return e;
  return cudaMemcpy(*tab, flat.data(), sizeof(T) * flat.size(), cudaMemcpyHostToDevice);
}

}  // namespace

// Candidate lists (host, once per map): kParts^3 lists of voxels in the general
// form and, for supports of at most 7 offsets per axis, kFastLists lists of pairs
// of voxels per distinct class support in the fast form.
cudaError_t build_candidate_tables(MapState& m) {
  const double lr = m.prm.length_scale / m.prm.res;
  std::vector<std::vector<int32_t>> lists;
  const int R = candidate_lists(lr, kParts, lists);
  const int kLists = (int)lists.size();
  size_t longest = 0;
  int maxd = 0;  // offsets actually used
  for (auto& L : lists) {
    longest = std::max(longest, L.size());
    for (int32_t e : L)
      for (int a = 0; a < 3; ++a) maxd = std::max(maxd, std::abs(((e >> (4 * a)) & 15) - R));
  }
  // re-pack with the tight R (the lookups hold 2R + 1 <= 15 entries per axis):
  // X row jx at byte offset 8 jx, YZ row (jy, jz) at byte offset 8 (jy (2R+1) + jz);
  // padding entries point at X row 2R + 1 (d^2 = 1e30) and YZ row 0
  const int Rt = maxd, na = 2 * Rt + 1;
  if (na > kAxisMax) return cudaErrorInvalidValue;
  const int tpad = (int)((longest + 31) / 32 * 32);
  std::vector<uint32_t> flat((size_t)kLists * tpad, (uint32_t)(8 * na));
  std::vector<int32_t> len(kLists);
  for (int t = 0; t < kLists; ++t) len[t] = (int32_t)lists[t].size();
  for (int t = 0; t < kLists; ++t)
    for (size_t k = 0; k < lists[t].size(); ++k) {
      const int32_t e = lists[t][k];
      const uint32_t jx = (uint32_t)((e & 15) - R + Rt), jy = (uint32_t)(((e >> 4) & 15) - R + Rt),
                     jz = (uint32_t)(((e >> 8) & 15) - R + Rt);
      flat[(size_t)t * tpad + k] = (8u * jx) | ((8u * (jy * na + jz)) << 8) | (jy << 19) | (jz << 23);
    }
  cudaError_t e = upload_lists(flat, len, &m.ctab, &m.clen);
  if (e != cudaSuccess) return e;
  m.ctab_pad = tpad;
  m.ctab_R = Rt;
  // The fast form: one table of kFastLists lists per distinct class support
  // l_k = l l_scale[k] (one table for the common l) of at most 7 offsets per
  // axis.  The accumulation also needs every l_k above half the voxel diagonal:
  // a point's own voxel, hence its own block, is then always touched.
  const int K1 = m.prm.num_classes + 1;
  std::vector<double> lrs;  // distinct supports (voxel units) that qualify
  int rmax = 0;
  bool own_touched = true;
  m.ftab_classes = 0;
  for (int k = 0; k < 32; ++k) m.ftab_of[k] = -1;
  for (int k = 0; k < K1; ++k) {
    const double lrk = m.prm.length_scale * m.prm.l_scale[k] / m.prm.res;
    own_touched = own_touched && lrk > 0.8661;
    const int Rk = largest_offset(lrk);
    if (2 * Rk + 1 > kFastAxis) continue;
    rmax = std::max(rmax, Rk);
    size_t t = 0;
    while (t < lrs.size() && lrs[t] != lrk) ++t;
    if (t == lrs.size()) lrs.push_back(lrk);
    m.ftab_of[k] = (int)t;
    m.ftab_classes |= 1u << k;
  }
  if (m.ftab_classes == 0) return cudaSuccess;
  std::vector<std::vector<std::vector<int32_t>>> pairs(lrs.size());
  size_t most = 0;
  for (size_t t = 0; t < lrs.size(); ++t) {
    pair_lists(lrs[t], rmax, pairs[t]);
    for (auto& L : pairs[t]) most = std::max(most, L.size());
  }
  const size_t pad = (most + 15) / 16 * 16;
  if (pad > (size_t)kFastPad) return cudaErrorInvalidValue;
  std::vector<uint16_t> ff((size_t)list_entries((int)lrs.size(), (int)pad), (uint16_t)kPadEntry);
  std::vector<int32_t> fl(lrs.size() * kFastLists);
  for (size_t t = 0; t < lrs.size(); ++t)
    for (size_t q = 0; q < (size_t)kFastLists; ++q) {
      const auto& L = pairs[t][q];
      fl[t * kFastLists + q] = (int32_t)L.size();
      for (size_t k = 0; k < L.size(); ++k)
        ff[(t * kFastLists + q) * pad + k] =
            (uint16_t)(((L[k] & 15) << 6) | (8 * ((L[k] >> 4) & 15)) | ((kZRows + 8u * (uint32_t)((L[k] >> 8) & 15)) << 8));
    }
  e = upload_lists(ff, fl, &m.ftab, &m.flen);
  if (e != cudaSuccess) return e;
  m.ftab_pad = (int)pad;
  m.ftab_pad_list = (uint32_t)(lrs.size() * kFastLists * pad);
  m.ftab_R = rmax;
  m.ftab_own_touched = own_touched;
  return cudaSuccess;
}

namespace {

// ctas_per_sm: 0 = as many as fit
template <typename Kernel>
cudaError_t launch_persistent(Kernel kern, const PtArgs& a, int sm_count, int ctas_per_sm, cudaStream_t st,
                              size_t smem = 0) {
  int per_sm = 0;
  cudaError_t e = cudaSuccess;
  if (smem) e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kern, kThreads, smem);
  if (e != cudaSuccess) return e;
  if (ctas_per_sm > 0) per_sm = std::min(per_sm, ctas_per_sm);
  kern<<<std::max(1, per_sm) * sm_count, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

template <bool kTrack>
cudaError_t launch_fast(const PtArgs& a, int sm_count, int ctas_per_sm, cudaStream_t st) {
  if (a.g.lscaled)  // per-class supports: the exact association and hard labels only
    return launch_persistent(accumulate_points_fast_kernel<kTrack, false, false, true>, a, sm_count, ctas_per_sm,
                             st);
  const size_t lists = sizeof(uint16_t) * (size_t)list_entries(1, a.list_pad);
  if (a.softidx)  // soft labels take the exact association only
    return launch_persistent(accumulate_points_fast_kernel<kTrack, false, true>, a, sm_count, ctas_per_sm, st, lists);
  if (a.g.assoc)
    return launch_persistent(accumulate_points_fast_kernel<kTrack, true>, a, sm_count, ctas_per_sm, st, lists);
  return launch_persistent(accumulate_points_fast_kernel<kTrack, false>, a, sm_count, ctas_per_sm, st, lists);
}

template <bool kTrack>
cudaError_t launch_general(const PtArgs& a, int sm_count, int ctas_per_sm, cudaStream_t st) {
  switch (a.tpad / 32) {  // unrolled sweeps for the common list lengths
    case 2: return launch_persistent(accumulate_points_kernel<kTrack, 2>, a, sm_count, ctas_per_sm, st);
    case 3: return launch_persistent(accumulate_points_kernel<kTrack, 3>, a, sm_count, ctas_per_sm, st);
    case 4: return launch_persistent(accumulate_points_kernel<kTrack, 4>, a, sm_count, ctas_per_sm, st);
    case 5: return launch_persistent(accumulate_points_kernel<kTrack, 5>, a, sm_count, ctas_per_sm, st);
    case 6: return launch_persistent(accumulate_points_kernel<kTrack, 6>, a, sm_count, ctas_per_sm, st);
    default: return launch_persistent(accumulate_points_kernel<kTrack, 0>, a, sm_count, ctas_per_sm, st);
  }
}

}  // namespace

cudaError_t launch_fresh_fill(MapState& m) {
  fresh_fill_kernel<<<m.sm_count * 4, 256, 0, m.stream>>>(m.s.fresh, m.hvals, m.alpha, m.pairs, m.g.K1 * m.g.B3,
                                                          m.g.B3, m.dc);
  m.launches += 1;
  return cudaGetLastError();
}

// the fast form needs its tables (with per-class supports, every class's l_k
// above half the voxel diagonal, so that the touched-block pass may record
// every point's own block) and addresses alpha and the pair counts with
// 32-bit element indices
bool fast_form_ready(const MapState& m) {
  return m.ftab != nullptr && m.nbrslot != nullptr && m.ftab_own_touched &&
         (uint64_t)(m.pool_blocks + 1) * (uint64_t)(m.g.K1 * m.g.B3) <= (1ull << 32);
}

cudaError_t launch_accumulate_points(MapState& m) {
  fresh_fill_kernel<<<m.sm_count * 4, 256, 0, m.stream>>>(m.s.fresh, m.hvals, m.alpha, m.pairs, m.g.K1 * m.g.B3,
                                                          m.g.B3, m.dc);
  PtArgs a;
  a.g = m.g;
  a.train = m.s.train;
  a.hkeys = m.hkeys;
  a.hvals = m.hvals;
  a.hash_cap = m.hash_cap;
  a.alpha = m.alpha;
  a.pairs = m.pairs;
  a.ctab = m.ctab;
  a.clen = m.clen;
  a.tpad = m.ctab_pad;
  a.R = m.ctab_R;
  a.recip_na = ((1u << 20) + (uint32_t)(2 * m.ctab_R + 1) - 1u) / (uint32_t)(2 * m.ctab_R + 1);
  // the tuning counts pairs of points; whole groups of kGroup points; the kernel takes fewer where there are few points
  a.chunk = (2 * std::max(1, std::min(64, m.tune.accumulate_chunk)) + kGroup - 1) / kGroup * kGroup;
  // soft labels: a point with a weight row costs up to K+1 times the reductions, so smaller
  // chunks balance the work queue better (16 against 60 points: 413 against 477 us per street scan)
  if (m.soft) a.chunk = std::min(a.chunk, 16);
  a.sink = (int32_t)m.pool_blocks;
  a.ftab = m.ftab;
  a.flen = m.flen;
  a.list_pad = m.ftab_pad;
  a.pad_list = m.ftab_pad_list;
  // the re-decision band [l2_lo, l2_hi] as a half-width, widened by the roundings of its ends
  a.band = 1.0625f * std::max(m.g.l2_hi - m.g.l2, m.g.l2 - m.g.l2_lo);
  for (int k = 0; k < kMaxClasses; ++k) a.band_k[k] = 1.0625f * 0.5f * (m.g.l2k_hi[k] - m.g.l2k_lo[k]);
  a.ownslot = m.s.ownslot;
  a.nbrslot = m.nbrslot;
  a.softidx = m.soft ? m.s.softidx : nullptr;
  a.wsoft = m.soft ? m.s.wsoft : nullptr;
  for (int k = 0; k < kMaxClasses; ++k) a.tab_of[k] = m.ftab_of[k];
  a.dc = m.dc;
  m.launches += 2;
  const int cps = m.tune.accumulate_ctas_per_sm;
  const bool fast = fast_form_ready(m);
  // soft labels and per-class supports without the fast form: the caller takes the weighted form instead
  if ((m.soft || m.g.lscaled) && !fast) return cudaErrorInvalidValue;
  if (fast) a.R = m.ftab_R;
  if (fast)
    return m.pairs ? launch_fast<true>(a, m.sm_count, cps, m.stream) : launch_fast<false>(a, m.sm_count, cps, m.stream);
  return m.pairs ? launch_general<true>(a, m.sm_count, cps, m.stream)
                 : launch_general<false>(a, m.sm_count, cps, m.stream);
}

}  // namespace sbki
