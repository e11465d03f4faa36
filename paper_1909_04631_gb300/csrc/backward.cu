// Differentiable form of the S-BKI update.
//
// Forward: alpha_v^k = alpha_0 + sum_{i: y_i = k, d_iv < l} sigma0 f(d_iv / l)
// (Eq. alpha_kernel with Eq. kernel, d_iv = |c_v - x_i|).  Given an upstream
// gradient G_v^k = dL/dalpha_v^k, held per voxel in a pool-shaped buffer
// (same block slots and layout as alpha), the backward pass visits every
// in-support pair once more, recomputing the kernel instead of storing pairs:
//   dL/dsigma0 += G f(r)
//   dL/dl      += G sigma0 f'(r) (-d / l^2)
//   dL/dx_i    += G sigma0 f'(r) (x_i - c_v) / (l d)
// with r = d/l, f' = df/dr = -u^4 D(u^2), u = 1 - r (kernel_poly.cuh); the
// x_i term is written with the unit vector (x_i - c_v)/d, which stays bounded
// as d -> 0 (f'(0) = 0).  With per-class kernel scales (class k's kernel is
// sigma0 s_k f) every term of a class-k point carries s_k, applied once per
// point, and dL/ds_k = sigma0 sum_{pairs of class-k points} G f.
//
// The held-out log-likelihood of the differentiable form scores held-out
// labelled points at the voxel containing them:
//   LL = sum_h log(alpha_{v(h)}^{y_h} / sum_k alpha_{v(h)}^k),
//   dLL/dalpha_v^k = sum_{h in v} ([k = y_h] / alpha_v^{y_h} - 1 / sum_j alpha_v^j)
// (the Dirichlet mean of Eq. (variance) as the predictive probability).
//
// Enumeration of pairs is the one of the point-major accumulation (same
// candidate lists, same FP32 test with the FP64 re-decision band), so the
// backward pass sees exactly the pairs the forward pass added.
#include <algorithm>
#include <climits>

#include "kernel_value.cuh"
#include "pair_rows.cuh"

namespace sbki {
namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
constexpr int kAxisMax = 15;
constexpr int kYZMax = kAxisMax * kAxisMax;

// ---------------------------------------------------------------- held-out log-likelihood
struct LLArgs {
  Geom g;
  float alpha0;
  const unsigned long long* hkeys;
  const int32_t* hvals;
  int64_t hash_cap;
  const float* alpha;
  float* grad;  // nullable: accumulate dLL/dalpha
  const float* xyz;
  const int32_t* labels;
  int64_t h;
  double* ll;  // device accumulator
  int map;
  DevCounters* dc;
};

__global__ void __launch_bounds__(256) heldout_kernel(LLArgs a) {
  const Geom& g = a.g;
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  double term = 0.0;
  if (i < a.h) {
    const int y = a.labels[i];
    if (y < 0 || y >= g.K1) {
      set_error(a.dc, SBKI_ERR_LABEL_RANGE);
    } else {
      int v[3];
      bool inside = true;
#pragma unroll
      for (int ax = 0; ax < 3; ++ax) {
        const float s = __fmul_rn(a.xyz[3 * i + ax], g.inv_res);
        inside = inside && fabsf(s) < (float)(kKeyLimit - 64);
        v[ax] = inside ? (int)floorf(s) : 0;
      }
      int32_t pool = -1;
      int local = 0;
      if (inside) {
        pool = find_pool_slot(a.hkeys, a.hvals, a.hash_cap,
                              pack_block(v[0] >> g.B_shift, v[1] >> g.B_shift, v[2] >> g.B_shift, a.map));
        const int m = g.B - 1;
        local = (((v[2] & m) << g.B_shift) + (v[1] & m)) * g.B + (v[0] & m);
      }
      const float* inc = pool >= 0 ? a.alpha + (size_t)pool * g.K1 * g.B3 + local : nullptr;
      double S = 0.0;
      for (int k = 0; k < g.K1; ++k) S += (double)(a.alpha0 + (inc ? inc[(size_t)k * g.B3] : 0.f));
      const double ay = (double)(a.alpha0 + (inc ? inc[(size_t)y * g.B3] : 0.f));
      term = log(ay) - log(S);
      if (a.grad && pool >= 0) {
        float* gb = a.grad + (size_t)pool * g.K1 * g.B3 + local;
        const float mS = (float)(-1.0 / S);
        for (int k = 0; k < g.K1; ++k) red_add_if(true, gb + (size_t)k * g.B3, mS);
        red_add_if(true, gb + (size_t)y * g.B3, (float)(1.0 / ay));
      }
    }
  }
  for (int o = 16; o > 0; o >>= 1) term += __shfl_down_sync(0xffffffffu, term, o);
  if ((threadIdx.x & 31) == 0 && term != 0.0) atomicAdd(a.ll, term);
}

// ---------------------------------------------------------------- upstream gradient at voxel keys
__global__ void __launch_bounds__(256) grad_scatter_kernel(Geom g, const unsigned long long* hkeys,
                                                           const int32_t* hvals, int64_t hash_cap,
                                                           const int64_t* keys, const float* grad, int64_t count,
                                                           int map, float* gpool, unsigned long long* missed) {
  const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (q >= count) return;
  const int64_t kx = keys[3 * q], ky = keys[3 * q + 1], kz = keys[3 * q + 2];
  const int64_t lim = kKeyLimit;
  int32_t pool = -1;
  if (kx > -lim && kx < lim && ky > -lim && ky < lim && kz > -lim && kz < lim)
    pool = find_pool_slot(hkeys, hvals, hash_cap,
                          pack_block((int32_t)(kx >> g.B_shift), (int32_t)(ky >> g.B_shift), (int32_t)(kz >> g.B_shift),
                                     map));
  if (pool < 0) {
    atomicAdd(missed, 1ull);
    return;
  }
  const int m = g.B - 1;
  const int local = ((((int)kz & m) << g.B_shift) + ((int)ky & m)) * g.B + ((int)kx & m);
  float* gb = gpool + (size_t)pool * g.K1 * g.B3 + local;
  for (int k = 0; k < g.K1; ++k) red_add_if(true, gb + (size_t)k * g.B3, grad[q * g.K1 + k]);
}

// ---------------------------------------------------------------- backward through Eq. (kernel)
struct BwdArgs {
  Geom g;
  const float4* xyzl;  // training set (x, y, z, label)
  int64_t p;
  const unsigned long long* hkeys;
  const int32_t* hvals;
  int64_t hash_cap;
  const float* gpool;  // dL/dalpha, [pool][K1][B3]
  const uint32_t* ctab;
  const int32_t* clen;
  int tpad, R;
  uint32_t recip_na;
  double* acc;         // [2]: sum s G f, sum s G u^4 D d (s: the point's class scale)
  double* acc_class;   // nullable [32]: per class of the point, sum G f
  float* grad_xyz;     // nullable [p][3]: (sigma0 / l) sum G u^4 D (c_v - x)/d
  float xyz_scale;     // sigma0 / l
  const uint16_t* ftab;  // pair form: lists (as the fast accumulation's)
  const int32_t* flen;
  int list_pad, fR;
  uint32_t pad_list;
  float band;          // half-width of the re-decision band around l^2
  DevCounters* dc;
};

struct BwdTables {
  float4 x[kAxisMax + 1];  // (e_x^2, address part, e_x, 0); entry 2R+1 is the padding row
  float4 yz[kYZMax];       // (e_y^2 + e_z^2, address part, e_y, e_z)
  const float* blk[27];    // gpool + (pool (K+1) + y_i) B^3, or null
};

// Adds the warp's sum of one point's lane terms v into the warp's class row
// (lane 0 writes; every lane of the warp calls it).
__device__ __forceinline__ void add_class_sum(double* row, int label, float v, int lane) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if (lane == 0 && label < 32) row[label] += (double)v;
}

__global__ void __launch_bounds__(kThreads, 3) backward_kernel(BwdArgs a) {
  __shared__ BwdTables s_tab[kWarps];
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  const int64_t gw = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  const int R = a.R, na = 2 * R + 1;
  BwdTables& t = s_tab[wid];
  __shared__ double s_cls[kWarps][32];  // per warp: sum G f by class (only with acc_class)
  if (a.dc->err != 0) return;
  if (lane == 0) t.x[na] = make_float4(kFar, __int_as_float(0), 0.f, 0.f);
  s_cls[wid][lane] = 0.0;
  double acc_f = 0.0, acc_l = 0.0;
  for (int64_t i = gw; i < a.p; i += nw) {
    const float4 p = a.xyzl[i];
    const int lm = label_of(p.w);  // label + 32 * map
    const int label = lm & ((1 << kLabelBits) - 1), map = lm >> kLabelBits;
    const PointFrame f = point_frame(p.x, p.y, p.z, R, g);
    const uint32_t* tab = a.ctab + f.part * a.tpad;
    if (lane < na) {
      const float e = centre_offset_at(lane - R, f.hi[0], f.lo[0], g);
      t.x[lane] = make_float4(__fmul_rn(e, e), __int_as_float(xpart(f, lane, R, g)), e, 0.f);
    }
    for (int q = lane; q < na * na; q += 32) {
      const int jy = (int)small_div((uint32_t)q, a.recip_na), jz = q - jy * na;
      const float ey = centre_offset_at(jy - R, f.hi[1], f.lo[1], g);
      const float ez = centre_offset_at(jz - R, f.hi[2], f.lo[2], g);
      t.yz[q] = make_float4(__fadd_rn(__fmul_rn(ey, ey), __fmul_rn(ez, ez)), __int_as_float(yzpart(f, jy, jz, R, g)),
                            ey, ez);
    }
    if (lane < 27) {
      const int32_t pool = (label < g.K1 && map < kMaxMaps) ? digit_pool(f, lane, map, a.hkeys, a.hvals, a.hash_cap)
                                                            : -1;
      t.blk[lane] = pool >= 0 ? a.gpool + ((size_t)pool * g.K1 + label) * g.B3 : nullptr;
    }
    __syncwarp();
    float sf = 0.f, sl = 0.f, sx = 0.f, sy = 0.f, sz = 0.f;
    const int len = __ldg(a.clen + f.part);
    for (int k = lane; k - lane < len; k += 32) {  // warp-uniform trip count
      const uint32_t ent = __ldg(tab + k);
      const float4 ex = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(t.x) + 2u * (ent & 0xffu));
      const float4 eyz =
          *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(t.yz) + 2u * ((ent >> 8) & 0x7ffu));
      const float d2 = __fadd_rn(ex.x, eyz.x);
      const int pk = __float_as_int(ex.y) + __float_as_int(eyz.y);
      bool in = d2 < g.l2_lo;
      const bool band = !in && d2 < g.l2_hi;
      if (__any_sync(0xffffffffu, band)) {
        if (band)
          in = in_support64_call(f.v0[0] + entry_jx(ent) - R, f.v0[1] + entry_jy(ent) - R,
                                 f.v0[2] + entry_jz(ent) - R, p.x, p.y, p.z, g.res64, g.l2_64);
      }
      const float* base = t.blk[pk & 0xff];
      if (in && base != nullptr) {
        const float G = __ldg(base + (pk >> 8));
        const float inv_d = rsqrtf(fmaxf(d2, 1e-30f));
        const float d = d2 * inv_d;
        const float u = fmaxf(__fmaf_rn(-d, g.inv_l, 1.0f), 0.0f);
        const float w = u * u;
        const float u4 = w * w;
        const float s = G * u4 * kernel_dq(w);  // -G df/dr
        sf = __fmaf_rn(G * u4 * u, kernel_q(w), sf);
        sl = __fmaf_rn(s, d, sl);
        // e = c_v - x and dr/dx = -e/(l d), so dk/dx = sigma0 u^4 D e / (l d)
        const float c = s * inv_d;
        sx = __fmaf_rn(c, ex.z, sx);
        sy = __fmaf_rn(c, eyz.z, sy);
        sz = __fmaf_rn(c, eyz.w, sz);
      }
    }
    const float s = label < g.K1 ? g.scale_k[label] : 0.f;  // the class's kernel scale
    acc_f += (double)s * (double)sf;
    acc_l += (double)s * (double)sl;
    if (a.acc_class) add_class_sum(s_cls[wid], label, sf, lane);
    if (a.grad_xyz) {
      for (int o = 16; o > 0; o >>= 1) {
        sx += __shfl_down_sync(0xffffffffu, sx, o);
        sy += __shfl_down_sync(0xffffffffu, sy, o);
        sz += __shfl_down_sync(0xffffffffu, sz, o);
      }
      if (lane == 0) {
        a.grad_xyz[3 * i] = sx * (s * a.xyz_scale);
        a.grad_xyz[3 * i + 1] = sy * (s * a.xyz_scale);
        a.grad_xyz[3 * i + 2] = sz * (s * a.xyz_scale);
      }
    }
    __syncwarp();  // the tables are rewritten for the next point
  }
  for (int o = 16; o > 0; o >>= 1) {
    acc_f += __shfl_down_sync(0xffffffffu, acc_f, o);
    acc_l += __shfl_down_sync(0xffffffffu, acc_l, o);
  }
  if (lane == 0) {
    atomicAdd(&a.acc[0], acc_f);
    atomicAdd(&a.acc[1], acc_l);
  }
  if (a.acc_class) {
    __syncwarp();
    if (s_cls[wid][lane] != 0.0) atomicAdd(&a.acc_class[lane], s_cls[wid][lane]);
  }
}

// The same pass in the pair form of the fast accumulation (pair_rows.cuh: half
// a warp per point, two voxels adjacent in x per lane; the rows hold the offsets
// themselves here), for supports of at most 7 offsets per axis.  A pair reads
// its two values of G in one 8-byte load; kernel, slope and the sums are packed
// FP32.  FP64 runs at 1/64 of the FP32 rate on this chip, so a lane sums the
// points of a few chunks as unevaluated FP32 pairs (error-free sums and
// products, 2^-44 relative over its 32 points) and then adds them to an FP64
// sum of its own in shared memory (in registers: 921 us instead of 905 below):
// neither the range nor the error depends on the length of the set.
//
// Bound by instruction issue, as the accumulation's sweep is.  2.0M points,
// 223M pairs: one voxel per lane with FP64 sums per point took 1378 us, this
// form takes 905.  The largest part of the difference are the FP64 sums: two
// fused multiply-adds per point and lane hold the SM's FP64 units for ~900 us.
constexpr int kBwdChunk = 16;  // consecutive training points per warp
constexpr int kBwdFold = 4;    // chunks whose sums are held in FP32 pairs

struct __align__(256) BwdWarp {
  unsigned char slot[kGroup][kSlotBytes];
  uint32_t btab[2][64];  // per half warp: G element base per block digit (27 used)
};

__device__ __forceinline__ float rsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// Running sums of two quantities as unevaluated pairs hi + lo.
struct PairSum {
  float2 hi, lo;
  __device__ __forceinline__ void add(float2 v, float s) {  // += s v, exactly up to the pair's 2^-48
    const float2 s2 = make_float2(s, s), p = __fmul2_rn(v, s2);
    const float2 e = __ffma2_rn(v, s2, make_float2(-p.x, -p.y));
    const float2 t = __fadd2_rn(hi, p);
    const float2 b = __fadd2_rn(t, make_float2(-hi.x, -hi.y));
    const float2 d = __fadd2_rn(hi, __fadd2_rn(b, make_float2(-t.x, -t.y)));  // hi - (t - b)
    const float2 f = __fadd2_rn(p, make_float2(-b.x, -b.y));
    lo = __fadd2_rn(lo, __fadd2_rn(e, __fadd2_rn(d, f)));
    hi = t;
  }
  __device__ __forceinline__ void clear() { hi = lo = make_float2(0.f, 0.f); }
  // The sum of both, and back to zero; an infinite term leaves lo without meaning.
  __device__ __forceinline__ double take() {
    const float rest = (isfinite(hi.x) ? lo.x : 0.f) + (isfinite(hi.y) ? lo.y : 0.f);
    const double s = (double)hi.x + (double)hi.y + (double)rest;
    clear();
    return s;
  }
};

template <bool kClass>
__global__ void __launch_bounds__(kThreads, 3) backward_pairs_kernel(BwdArgs a) {
  __shared__ BwdWarp s_w[kWarps];
  __shared__ double s_cls[kClass ? kWarps : 1][32];  // per warp: sum G f by class
  __shared__ double s_sum[kWarps][2][32];            // per lane: sum s G f, sum s G u^4 D d
  extern __shared__ __align__(16) uint16_t s_lists[];
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  BwdWarp& W = s_w[wid];
  const int R = a.fR;
  if (a.dc->err != 0) return;
  if ((smem_addr(&W) & 255u) != 0u) {  // the byte permutes need 256-byte aligned slots and tables
    if (lane == 0) set_error(a.dc, SBKI_ERR_CUDA);
    return;
  }
  // a half without a point reads X row 0, Z row 0 and the padding row of its slot
  for (int e = lane; e < kGroup * kSlotBytes / 4; e += 32) reinterpret_cast<float*>(W.slot)[e] = 0.0f;
  __syncwarp();
  if (lane < kGroup) *reinterpret_cast<float*>(W.slot[lane] + kYRows + 8 * kFastAxis) = kFarOffset;
  if (kClass) s_cls[wid][lane] = 0.0;
  const int n16 = list_entries(1, a.list_pad) / 8;
  for (int e = threadIdx.x; e < n16; e += kThreads)
    reinterpret_cast<uint4*>(s_lists)[e] = __ldg(reinterpret_cast<const uint4*>(a.ftab) + e);
  __syncthreads();
  const uint32_t lists = smem_addr(s_lists);
  const int half = lane >> 4, hl = lane & 15;
  const uint32_t slot0 = smem_addr(&W.slot[0][0]) + (uint32_t)half * kSlotBytes;
  const uint32_t btab = smem_addr(&W.btab[half][0]);
  const int gl = lane >> 2, role = lane & 3, ax = max(role - 1, 0);
  const uint32_t K1B3 = (uint32_t)(g.K1 * g.B3);
  unsigned long long cblk = kEmpty;  // block the half's table belongs to
  uint32_t present = 0u;             // its digits that are in the map
  PairSum acc_f, acc_l;              // sum s G f, sum s G u^4 D d, by column
  acc_f.clear();
  acc_l.clear();
  s_sum[wid][0][lane] = s_sum[wid][1][lane] = 0.0;
  int chunks = 0;
  const int64_t gw = (int64_t)blockIdx.x * kWarps + wid, nw = (int64_t)gridDim.x * kWarps;
  for (int64_t c = gw; c * kBwdChunk < a.p; c += nw) {
    const int64_t c1 = min(a.p, c * kBwdChunk + kBwdChunk);
    for (int64_t g0 = c * kBwdChunk; g0 < c1; g0 += kGroup) {
      const int gn = (int)min(c1 - g0, (int64_t)kGroup);  // warp-uniform
      // rows of every point of the group, four lanes per point
      int pt = 0, lw = 0, b0 = 0;
      if (gl < gn) {
        const float4 p = a.xyzl[g0 + gl];
        const float x = ax == 0 ? p.x : (ax == 1 ? p.y : p.z);
        // A coordinate that is not finite or past floor_small's range reaches no voxel of a map.  Every candidate is
        // multiplied out below, masked or not, so such a point's rows must not hold it (0 * inf is NaN): they are
        // formed at 0 and the point has no list.
        const bool inside = fabsf(__fmul_rn(x, g.inv_res)) < 4194304.0f;
        const AxisFrame f = axis_frame(inside ? x : 0.f, g);
        lw = label_of(p.w);
        pt = form_rows<false>(W.slot[gl], gl, role, f, (uint32_t)((lw & ((1 << kLabelBits) - 1)) * g.B3), R, g);
        if (!inside) pt = kFastLists;
        b0 = f.v0 >> g.B_shift;
      }
      const int pty = __shfl_sync(0xffffffffu, pt, lane | 2), ptz = __shfl_sync(0xffffffffu, pt, lane | 3);
      const int by = __shfl_sync(0xffffffffu, b0, lane | 2), bz = __shfl_sync(0xffffffffu, b0, lane | 3);
      if (role == 0 && gl < gn) {
        const int list = pt + kFastParts * (pty + kFastParts / 2 * ptz);
        const int label = lw & ((1 << kLabelBits) - 1), map = lw >> kLabelBits;
        // others have no G
        const bool known = label < g.K1 && map < kMaxMaps && list < kFastLists;
        const unsigned long long key = known ? pack_block(b0, by, bz, map) : kEmpty;
        uint32_t* sc = reinterpret_cast<uint32_t*>(W.slot[gl] + kScalars);
        sc[0] = known ? (uint32_t)(list * a.list_pad) : a.pad_list;
        sc[1] = (uint32_t)(label & 31) | (known ? (uint32_t)(__ldg(a.flen + list) + 15) >> 4 : 0u) << 16;
        sc[2] = (uint32_t)key;
        sc[3] = (uint32_t)(key >> 32);
      }
      __syncwarp();
      // two points at a time, one per half warp
      for (int k0 = 0; k0 < gn; k0 += 2) {
        const uint32_t slot = slot0 + (uint32_t)k0 * kSlotBytes;
        const int k = k0 + half;
        const bool have = k < gn;
        const uint4 sv = lds_u4(slot + kScalars);
        const unsigned long long key = (unsigned long long)sv.w << 32 | sv.z;
        const bool moved = have && key != kEmpty && key != cblk;
        if (__any_sync(0xffffffffu, moved)) {  // a half's table belongs to another block
          uint32_t in = 0u;
          if (moved) {
            cblk = key;
            int bx, byy, bzz;
            unpack_block(key, bx, byy, bzz);
            const int map = map_of_block(key);
            for (int d = hl; d < 27; d += 16) {
              const int32_t pool = find_pool_slot(a.hkeys, a.hvals, a.hash_cap,
                                                  pack_block(bx - 1 + d % 3, byy - 1 + (d / 3) % 3, bzz - 1 + d / 9, map));
              in |= pool >= 0 ? 1u << d : 0u;
              W.btab[half][d] = (pool >= 0 ? (uint32_t)pool : 0u) * K1B3 - ((4u * (uint32_t)d) << 24);
            }
          }
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) in |= __shfl_xor_sync(0xffffffffu, in, o);
          if (moved) present = in;
          __syncwarp();
        }
        const uint32_t mine = have ? (sv.y >> 16) & 0xffu : 0u;  // rounds of this half's point
        const uint32_t rounds = max(mine, __shfl_xor_sync(0xffffffffu, mine, 16));
        const uint32_t list = lists + 2u * ((mine ? sv.x : a.pad_list) + (uint32_t)hl);
        const float2 nl2 = make_float2(-g.l2, -g.l2);
        float2 sf = make_float2(0.f, 0.f), sl = sf;  // sum G f, sum G u^4 D d of this lane's two columns
        float2 gx = sf, gy = sf, gz = sf;
        for (uint32_t r = 0; r < rounds; ++r) {  // warp-uniform
          const uint32_t e = lds_u16(list + 32u * r);
          const uint32_t xa = slot | ((e >> 2) & 0x30u);
          const float2 ex = lds_f2(xa), ry = lds_f2((slot | (e & 0x38u)) + kYRows),
                       rz = lds_f2(__byte_perm(e, slot, 0x7651));
          const float rd = __fadd_rn(__fmul_rn(ry.x, ry.x), __fmul_rn(rz.x, rz.x));
          const float2 d2 = __fadd2_rn(make_float2(rd, rd), __fmul2_rn(ex, ex));
          const uint32_t pk = lds_u32(xa + 8) + __float_as_uint(ry.y) + __float_as_uint(rz.y);
          const float2 t = __fadd2_rn(d2, nl2);
          bool ina = t.x < 0.f, inb = t.y < 0.f;
          if (__any_sync(0xffffffffu, fminf(fabsf(t.x), fabsf(t.y)) <= a.band)) {
            if (fabsf(t.x) <= a.band) ina = band_decide(e, 0, a.xyzl, (uint32_t)(g0 + k), R, g, g.l2_64);
            if (fabsf(t.y) <= a.band) inb = band_decide(e, 1, a.xyzl, (uint32_t)(g0 + k), R, g, g.l2_64);
          }
          const uint32_t dig = pk >> 26;
          float2 G = make_float2(0.f, 0.f);
          if ((ina || inb) && ((present >> dig) & 1u))
            G = __ldg(reinterpret_cast<const float2*>(a.gpool + (lds_u32(__byte_perm(pk, btab, 0x7653)) + pk)));
          if (!ina) G.x = 0.f;
          if (!inb) G.y = 0.f;
          const float2 id = make_float2(rsqrt_approx(fmaxf(d2.x, 1e-30f)), rsqrt_approx(fmaxf(d2.y, 1e-30f)));
          const float2 d = __fmul2_rn(d2, id);
          const float2 u = make_float2(__saturatef(__fmaf_rn(-d.x, g.inv_l, 1.0f)),
                                       __saturatef(__fmaf_rn(-d.y, g.inv_l, 1.0f)));
          const float2 w = __fmul2_rn(u, u);
          const float2 Gu4 = __fmul2_rn(G, __fmul2_rn(w, w));
          const float2 s = __fmul2_rn(Gu4, kernel_dq2(w));  // -G df/dr
          sf = __ffma2_rn(__fmul2_rn(Gu4, u), kernel_q2(w), sf);
          sl = __ffma2_rn(s, d, sl);
          const float2 c2 = __fmul2_rn(s, id);
          // e = c_v - x and dr/dx = -e/(l d), so dk/dx = sigma0 u^4 D e / (l d)
          gx = __ffma2_rn(c2, ex, gx);
          gy = __ffma2_rn(c2, make_float2(ry.x, ry.x), gy);
          gz = __ffma2_rn(c2, make_float2(rz.x, rz.x), gz);
        }
        const int label = (int)(sv.y & 31u);
        const float s = mine ? g.scale_k[label] : 0.f;  // the class's kernel scale
        acc_f.add(sf, s);
        acc_l.add(sl, s);
        if (kClass) {
          float v = mine ? sf.x + sf.y : 0.f;
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
          const float v1 = __shfl_sync(0xffffffffu, v, 16);
          const int l1 = __shfl_sync(0xffffffffu, label, 16);
          if (lane == 0) {
            s_cls[wid][label] += (double)v;
            s_cls[wid][l1] += (double)v1;
          }
        }
        if (a.grad_xyz) {
          // joined over the half's lanes; lanes 0, 1, 2 of a half write x, y, z
          float sx = gx.x + gx.y, sy = gy.x + gy.y, sz = gz.x + gz.y;
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) {
            sx += __shfl_xor_sync(0xffffffffu, sx, o);
            sy += __shfl_xor_sync(0xffffffffu, sy, o);
            sz += __shfl_xor_sync(0xffffffffu, sz, o);
          }
          if (have && hl < 3) a.grad_xyz[3 * (g0 + k) + hl] = (hl == 0 ? sx : (hl == 1 ? sy : sz)) * (s * a.xyz_scale);
        }
      }
      __syncwarp();  // the slots are rewritten by the next group
    }
    if (++chunks % kBwdFold == 0) {  // warp-uniform
      s_sum[wid][0][lane] += acc_f.take();
      s_sum[wid][1][lane] += acc_l.take();
    }
  }
  double af = s_sum[wid][0][lane] + acc_f.take(), al = s_sum[wid][1][lane] + acc_l.take();
  for (int o = 16; o > 0; o >>= 1) {
    af += __shfl_down_sync(0xffffffffu, af, o);
    al += __shfl_down_sync(0xffffffffu, al, o);
  }
  if (lane == 0) {
    atomicAdd(&a.acc[0], af);
    atomicAdd(&a.acc[1], al);
  }
  if (kClass) {
    __syncwarp();
    if (s_cls[wid][lane] != 0.0) atomicAdd(&a.acc_class[lane], s_cls[wid][lane]);
  }
}

template <bool kClass>
cudaError_t launch_backward_pairs(const BwdArgs& a, int sm_count, cudaStream_t st) {
  const size_t smem = sizeof(uint16_t) * (size_t)list_entries(1, a.list_pad);
  int per_sm = 0;
  cudaError_t e = cudaFuncSetAttribute(backward_pairs_kernel<kClass>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, backward_pairs_kernel<kClass>, kThreads, smem);
  if (e != cudaSuccess) return e;
  const int64_t want = (a.p + (int64_t)kWarps * kBwdChunk - 1) / ((int64_t)kWarps * kBwdChunk);
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)std::max(1, per_sm) * sm_count));
  backward_pairs_kernel<kClass><<<grid, kThreads, smem, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_heldout(const MapState& m, const float* xyz, const int32_t* labels, int64_t h, float* grad,
                           double* ll_dev) {
  if (h <= 0) return cudaSuccess;
  LLArgs a;
  a.g = m.g;
  a.alpha0 = (float)m.prm.alpha0;
  a.hkeys = m.hkeys;
  a.hvals = m.hvals;
  a.hash_cap = m.hash_cap;
  a.alpha = m.alpha;
  a.grad = grad;
  a.xyz = xyz;
  a.labels = labels;
  a.h = h;
  a.ll = ll_dev;
  a.map = m.active_map;
  a.dc = m.dc;
  heldout_kernel<<<(unsigned)((h + 255) / 256), 256, 0, m.stream>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_grad_scatter(const MapState& m, const int64_t* keys, const float* grad, int64_t count, float* gpool,
                                unsigned long long* missed_dev) {
  if (count <= 0) return cudaSuccess;
  grad_scatter_kernel<<<(unsigned)((count + 255) / 256), 256, 0, m.stream>>>(m.g, m.hkeys, m.hvals, m.hash_cap, keys,
                                                                             grad, count, m.active_map, gpool,
                                                                             missed_dev);
  return cudaGetLastError();
}

cudaError_t launch_backward(const MapState& m, const float4* xyzl, int64_t p, const float* gpool, double* acc_dev,
                            float* grad_xyz, double* acc_class) {
  if (p <= 0) return cudaSuccess;
  BwdArgs a;
  a.g = m.g;
  a.xyzl = xyzl;
  a.p = p;
  a.hkeys = m.hkeys;
  a.hvals = m.hvals;
  a.hash_cap = m.hash_cap;
  a.gpool = gpool;
  a.ctab = m.ctab;
  a.clen = m.clen;
  a.tpad = m.ctab_pad;
  a.R = m.ctab_R;
  a.recip_na = ((1u << 20) + (uint32_t)(2 * m.ctab_R + 1) - 1u) / (uint32_t)(2 * m.ctab_R + 1);
  a.acc = acc_dev;
  a.grad_xyz = grad_xyz;
  a.acc_class = acc_class;
  a.xyz_scale = (float)(m.prm.sigma0 / m.prm.length_scale);
  a.dc = m.dc;
  // the pair form has its lists and addresses G with 32-bit element indices (and points for the re-decision)
  if (m.ftab && (uint64_t)m.pool_blocks * (uint64_t)(m.g.K1 * m.g.B3) <= (1ull << 32) && p <= 0xffffffffll) {
    a.ftab = m.ftab;
    a.flen = m.flen;
    a.list_pad = m.ftab_pad;
    a.pad_list = m.ftab_pad_list;
    a.fR = m.ftab_R;
    a.band = 1.0625f * std::max(m.g.l2_hi - m.g.l2, m.g.l2 - m.g.l2_lo);
    return acc_class ? launch_backward_pairs<true>(a, m.sm_count, m.stream)
                     : launch_backward_pairs<false>(a, m.sm_count, m.stream);
  }
  int per_sm = 0;
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, backward_kernel, kThreads, 0);
  if (e != cudaSuccess) return e;
  const int64_t want = (p + kWarps - 1) / kWarps;
  const int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (int64_t)std::max(1, per_sm) * m.sm_count));
  backward_kernel<<<grid, kThreads, 0, m.stream>>>(a);
  return cudaGetLastError();
}

}  // namespace sbki
