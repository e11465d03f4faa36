// sbki_query_points: Eq. (alpha_kernel) at arbitrary points of space (Sec. IV:
// the continuous model can be queried at any resolution, not only at voxel
// centres), from a given training set:
//     alpha^k(x*) = alpha_0 + sum over training points i with |x* - x_i| < l
//                   and y_i = k of sigma0 s_k f(|x* - x_i| / l).
// The accumulation turned around: the training points are binned into cells of
// edge just above l (so every point within l of a query lies in the 3 x 3 x 3
// cells around the query's cell).  A hash holds the occupied cells; the points
// are counted into it, the cells get consecutive runs in no particular order,
// and the points are brought to their runs by a stable sort on the run's start
// (log2 of the number of points bits instead of the cell key's 63; stable, so
// every call sums in the same order).  Then one warp per query looks the 27
// cells up, drops those farther than l, walks the candidates of the rest as one
// list and sums the kernel per class.
// Membership is decided in FP32 from the exact FP32 offsets' squares and
// re-decided in FP64 inside the relative band around l^2, as in the map update,
// so it is the plain FP64 definition's.
//
// A street scan's training set and 200000 queries (23M pairs): 1310 us a call
// before, 535 now.  The query kernel, bound by instruction issue, takes 217 us;
// with the runs taken one after the other, a lane's run ended by a serial scan
// of the keys and shared atomics per class it took 591.  Sorting the cell keys
// took 126 us; counting, starts and the shorter sort take 85.
#include <algorithm>
#include <cmath>
#include <cstdio>

#include "kernel_value.cuh"
#include "point_common.cuh"

namespace sbki {
namespace {

constexpr int kQThreads = 256;
constexpr int kQWarps = kQThreads / 32;
constexpr int kCellBits = 21;  // per axis in a packed cell key (offset 2^20)

__device__ __forceinline__ unsigned long long cell_key(float x, float y, float z, float inv_c) {
  const unsigned long long off = 1ull << (kCellBits - 1);
  const unsigned long long m = (1ull << kCellBits) - 1;
  const long long cx = (long long)floorf(x * inv_c), cy = (long long)floorf(y * inv_c), cz = (long long)floorf(z * inv_c);
  return ((((unsigned long long)(cx + (long long)off)) & m) << (2 * kCellBits)) |
         ((((unsigned long long)(cy + (long long)off)) & m) << kCellBits) | (((unsigned long long)(cz + (long long)off)) & m);
}

__device__ __forceinline__ uint32_t cell_hash(unsigned long long k, uint32_t mask) {
  k ^= k >> 31;
  k *= 0x9e3779b97f4a7c15ull;
  k ^= k >> 29;
  return (uint32_t)k & mask;
}

// One slot of the hash, read in one 16-byte load; all ones when empty.
struct __align__(16) Cell {
  unsigned long long key;
  uint32_t start;  // first point of the cell's run
  uint32_t last;   // points in the run, less one (counted up from all ones)
};

// Counts the points into their cells and notes each point's slot.  The lanes of
// a warp that share a cell share its insertion and its atomic.
__global__ void __launch_bounds__(kQThreads) cell_count_kernel(const float4* __restrict__ train, int64_t p, float inv_c,
                                                               Cell* __restrict__ cells, uint32_t mask,
                                                               uint32_t* __restrict__ slot, DevCounters* dc) {
  const int lane = threadIdx.x & 31;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i0 = (int64_t)blockIdx.x * blockDim.x + (threadIdx.x & ~31); i0 < p; i0 += stride) {
    const int64_t i = i0 + lane;
    unsigned long long k = kEmpty;
    if (i < p) {
      const float4 t = train[i];
      k = cell_key(t.x, t.y, t.z, inv_c);
    }
    const uint32_t peers = __match_any_sync(0xffffffffu, k);
    const int leader = __ffs((int)peers) - 1;
    uint32_t h = 0;
    if (k != kEmpty && lane == leader) {
      h = cell_hash(k, mask);
      for (uint32_t probe = 0;; ++probe, h = (h + 1u) & mask) {
        unsigned long long at = cells[h].key;
        if (at == kEmpty) at = atomicCAS(&cells[h].key, kEmpty, k);
        if (at == kEmpty || at == k) {
          atomicAdd(&cells[h].last, (uint32_t)__popc(peers));
          break;
        }
        if (probe == mask) {
          set_error(dc, SBKI_ERR_CAPACITY);
          break;
        }
      }
    }
    h = __shfl_sync(0xffffffffu, h, leader);
    if (i < p) slot[i] = h;
  }
}

// Consecutive runs for the occupied cells, in any order: one atomic per CTA.
__global__ void __launch_bounds__(kQThreads) cell_starts_kernel(Cell* __restrict__ cells, uint32_t mask, uint32_t* total) {
  __shared__ uint32_t s_sum[kQWarps], s_base;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int64_t h0 = (int64_t)blockIdx.x * kQThreads; h0 <= (int64_t)mask; h0 += (int64_t)gridDim.x * kQThreads) {
    const int64_t h = h0 + threadIdx.x;  // the capacity is a multiple of the CTA
    const uint32_t n = cells[h].last + 1u;
    uint32_t inc = n;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) s_sum[wid] = inc;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t sum = 0;
      for (int w = 0; w < kQWarps; ++w) {
        const uint32_t v = s_sum[w];
        s_sum[w] = sum;
        sum += v;
      }
      s_base = sum ? atomicAdd(total, sum) : 0u;
    }
    __syncthreads();
    if (n) cells[h].start = s_base + s_sum[wid] + inc - n;
    __syncthreads();
  }
}

// sort keys of the points: where the run of the point's cell starts
__global__ void __launch_bounds__(kQThreads) run_keys_kernel(const Cell* __restrict__ cells, const uint32_t* __restrict__ slot,
                                                             int64_t p, unsigned long long* __restrict__ keys,
                                                             uint32_t* __restrict__ idx) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x) {
    keys[i] = cells[slot[i]].start;
    idx[i] = (uint32_t)i;
  }
}

__global__ void __launch_bounds__(kQThreads) run_fill_kernel(const float4* __restrict__ train, int64_t p,
                                                             const uint32_t* __restrict__ idx, float4* __restrict__ runs,
                                                             const DevCounters* dc) {
  if (dc->err != 0) return;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < p; i += (int64_t)gridDim.x * blockDim.x)
    runs[i] = train[idx[i]];
}

struct QueryArgs {
  Geom g;
  float inv_c;
  const float4* runs;  // [p] (x, y, z, label as float), cell by cell
  const Cell* cells;
  uint32_t mask;
  const float* pts;    // [q,3]
  int64_t q;
  float* alpha;        // [q,K+1]
  float alpha0;
  DevCounters* dc;
};

// How far (in cell edges) coordinate t, in its cell at fraction f, lies from the neighbour cell at offset o.
__device__ __forceinline__ float cell_gap(float f, int o) { return o == 0 ? 0.0f : (o < 0 ? f : 1.0f - f); }

// One warp per query point.  Lane c < 27 finds cell c's run; the runs that are
// not empty and not out of reach form one list, so its 32-point rounds are full
// whatever the runs' lengths (a surface leaves a few points per cell).  Every
// lane adds into columns of its own in shared memory (row: class): FP32 shared
// atomics on one class take turns, and the points around a query mostly share
// one.  The classes met are joined by shuffles at the end.
__global__ void __launch_bounds__(kQThreads, 6) query_points_kernel(QueryArgs a) {
  extern __shared__ float s_mem[];  // per warp: K1 rows of 32 sums, one row of run offsets
  const Geom& g = a.g;
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  if (a.dc->err != 0) return;
  float* sums = s_mem + (size_t)wid * (g.K1 + 1) * 32 + lane;
  uint32_t* runof = reinterpret_cast<uint32_t*>(s_mem + (size_t)wid * (g.K1 + 1) * 32 + 32 * g.K1);
  for (int k = 0; k < g.K1; ++k) sums[32 * k] = 0.0f;
  const int ox = lane % 3 - 1, oy = (lane / 3) % 3 - 1, oz = lane / 9 - 1;
  const uint32_t below = (2u << lane) - 1u;  // this lane and those before it
  const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
  for (int64_t qi = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; qi < a.q; qi += nw) {
    const float qx = a.pts[3 * qi], qy = a.pts[3 * qi + 1], qz = a.pts[3 * qi + 2];
    uint32_t start = 0, n = 0;
    if (lane < 27) {
      const float tx = qx * a.inv_c, ty = qy * a.inv_c, tz = qz * a.inv_c;
      const float gx = cell_gap(tx - floorf(tx), ox), gy = cell_gap(ty - floorf(ty), oy), gz = cell_gap(tz - floorf(tz), oz);
      // out of reach: a cell edge is 1.001 l, so l is sqrt(0.998003) edges; the coordinates in edges are within
      // 2^-24 relative of the exact ones, on both sides (NaN: kept, and no point passes the distance test)
      const float reach = 0.99801f + 1e-6f * fmaxf(fabsf(tx), fmaxf(fabsf(ty), fabsf(tz)));
      const unsigned long long k0 = cell_key(qx, qy, qz, a.inv_c);
      const unsigned long long m = (1ull << kCellBits) - 1;
      const long long cx = (long long)((k0 >> (2 * kCellBits)) & m) + ox;
      const long long cy = (long long)((k0 >> kCellBits) & m) + oy;
      const long long cz = (long long)(k0 & m) + oz;
      if (!(gx * gx + gy * gy + gz * gz > reach) && cx >= 0 && cy >= 0 && cz >= 0 && cx <= (long long)m &&
          cy <= (long long)m && cz <= (long long)m) {
        const unsigned long long k = ((unsigned long long)cx << (2 * kCellBits)) | ((unsigned long long)cy << kCellBits) |
                                     (unsigned long long)cz;
        uint32_t h = cell_hash(k, a.mask);
        for (uint32_t probe = 0;; ++probe, h = (h + 1u) & a.mask) {
          const uint4 c = __ldg(reinterpret_cast<const uint4*>(a.cells) + h);
          const unsigned long long hk = (unsigned long long)c.y << 32 | c.x;
          if (hk == k) {
            start = c.z;
            n = c.w + 1u;
            break;
          }
          if (hk == kEmpty || probe == a.mask) break;
        }
      }
    }
    uint32_t end = n;  // of this lane's run in the list
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const uint32_t v = __shfl_up_sync(0xffffffffu, end, o);
      if (lane >= o) end += v;
    }
    const uint32_t total = __shfl_sync(0xffffffffu, end, 31), pre = end - n;
    const uint32_t some = __ballot_sync(0xffffffffu, n != 0u);
    if (n) runof[__popc(some & (below >> 1))] = start - pre;
    __syncwarp();
    uint32_t met = 0u;         // classes of this lane's points
    const uint32_t* run = runof - 1;  // of the runs begun before the round, the last
    for (uint32_t b = 0; b < total; b += 32) {
      const uint32_t heads = __reduce_or_sync(0xffffffffu, n != 0u && pre - b < 32u ? 1u << (pre - b) : 0u);
      const uint32_t j = b + lane;
      if (j < total) {
        const float4 t = __ldg(a.runs + (uint32_t)(run[__popc(heads & below)] + j));
        const float ex = __fsub_rn(qx, t.x), ey = __fsub_rn(qy, t.y), ez = __fsub_rn(qz, t.z);
        const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(ex, ex), __fmul_rn(ey, ey)), __fmul_rn(ez, ez));
        bool in = d2 < g.l2_lo;
        if (!in && d2 < g.l2_hi) {  // the plain FP64 test, as the definition states it
          const double dx = (double)qx - (double)t.x, dy = (double)qy - (double)t.y, dz = (double)qz - (double)t.z;
          in = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz)) < g.l2_64;
        }
        const int label = label_of(t.w) & ((1 << kLabelBits) - 1);
        if (in && label < g.K1) {
          const float u = __saturatef(__fmaf_rn(-d2 * rsqrtf(fmaxf(d2, 1e-30f)), g.inv_l, 1.0f));
          const float w = u * u;
          sums[32 * label] = __fmaf_rn(w * w * u, kernel_q(w), sums[32 * label]);
          met |= 1u << label;
        }
      }
      run += __popc(heads);
    }
    met = __reduce_or_sync(0xffffffffu, met);
    float mine = 0.0f;  // the sum of class `lane`
    while (met) {       // warp-uniform
      const int k = __ffs((int)met) - 1;
      met &= met - 1u;
      float v = sums[32 * k];
      sums[32 * k] = 0.0f;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      if (lane == k) mine = g.sigma0_k[k] * v;
    }
    if (lane < g.K1) a.alpha[qi * g.K1 + lane] = __fadd_rn(a.alpha0, mine);
    __syncwarp();  // the run offsets are rewritten for the next query
  }
}

bool device_ptr(const void* p) {
  cudaPointerAttributes at;
  if (cudaPointerGetAttributes(&at, p) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  return at.type == cudaMemoryTypeDevice || at.type == cudaMemoryTypeManaged;
}

sbki_status fail(sbki_status s, const char* msg) {
  set_global_error(msg);
  return s;
}

}  // namespace
}  // namespace sbki

using namespace sbki;

extern "C" sbki_status sbki_query_points(const sbki_params* params, const float* xyzl, int64_t p, const float* pts,
                                         int64_t q, float* alpha_out) {
  if (!params || p < 0 || q < 0 || (p > 0 && !xyzl) || (q > 0 && (!pts || !alpha_out)))
    return fail(SBKI_ERR_INVALID_ARG, "query points: bad arguments");
  sbki_status st = validate_params(params);
  if (st != SBKI_OK) return st;
  if (params->sensor_model != 0) return fail(SBKI_ERR_INVALID_ARG, "query points: the counting model has no kernel");
  if (p > (int64_t)UINT32_MAX - 1) return fail(SBKI_ERR_INVALID_ARG, "query points: too many training points");
  if (q == 0) return SBKI_OK;
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
  if (cudaSetDevice(params->device) != cudaSuccess) return fail(SBKI_ERR_CUDA, "query points: cudaSetDevice failed");
  const Geom g = geometry_of(*params);
  cudaStream_t s = (cudaStream_t)params->cuda_stream;
  int sms = 1;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, params->device);
  const int64_t np = std::max<int64_t>(p, 1);
  uint64_t cap = 1024;  // slots: at most 3/4 in use
  while (3 * cap < 4 * (uint64_t)np && cap < (1ull << 32)) cap <<= 1;
  const uint32_t mask = (uint32_t)(cap - 1);
  // one device buffer for everything (this entry point allocates; it is a stateless query): a pair of
  // allocation and release per part took about 550 us a call, one pair takes 110
  const bool dev_train = p == 0 || device_ptr(xyzl), dev_pts = device_ptr(pts), dev_out = device_ptr(alpha_out);
  size_t bytes = 0;
  auto part = [&](size_t n) {
    const size_t at = bytes;
    bytes += (n + 255) & ~(size_t)255;
    return at;
  };
  const size_t at_dc = part(sizeof(DevCounters)), at_total = part(sizeof(uint32_t));
  const size_t at_cells = part(sizeof(Cell) * cap), at_keys = part(2 * sizeof(unsigned long long) * np);
  const size_t at_idx1 = part(sizeof(uint32_t) * np), at_idx2 = part(sizeof(uint32_t) * np);
  const size_t at_work = part(sizeof(uint32_t) * (size_t)radix_work_entries(np));
  const size_t at_train = dev_train ? 0 : part(sizeof(float4) * p), at_pts = dev_pts ? 0 : part(sizeof(float) * 3 * q),
               at_out = dev_out ? 0 : part(sizeof(float) * g.K1 * q);
  char* buf = nullptr;
  cudaError_t e = cudaSuccess;
  auto ok = [&](cudaError_t x) {
    if (e == cudaSuccess) e = x;
    return e == cudaSuccess;
  };
  ok(cudaMalloc(&buf, bytes));
  DevCounters* dc = reinterpret_cast<DevCounters*>(buf + at_dc);
  Cell* cells = reinterpret_cast<Cell*>(buf + at_cells);
  uint32_t* total = reinterpret_cast<uint32_t*>(buf + at_total);
  float4* runs = reinterpret_cast<float4*>(buf + at_keys);  // the sort's keys, no longer needed then
  const float4* train = reinterpret_cast<const float4*>(dev_train ? (const char*)xyzl : buf + at_train);
  const float* qp = dev_pts ? pts : reinterpret_cast<float*>(buf + at_pts);
  float* out = dev_out ? alpha_out : reinterpret_cast<float*>(buf + at_out);
  if (e == cudaSuccess && !dev_train) ok(cudaMemcpyAsync(buf + at_train, xyzl, sizeof(float4) * p, cudaMemcpyHostToDevice, s));
  if (e == cudaSuccess && !dev_pts) ok(cudaMemcpyAsync(buf + at_pts, pts, sizeof(float) * 3 * q, cudaMemcpyHostToDevice, s));
  if (e == cudaSuccess) ok(cudaMemsetAsync(buf, 0, at_cells, s));
  if (e == cudaSuccess) ok(cudaMemsetAsync(cells, 0xff, sizeof(Cell) * cap, s));
  // cells of edge just above l: every point within l of a query lies in the 27 cells around it
  const float inv_c = (float)(1.0 / (params->length_scale * 1.001));
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((np + kQThreads - 1) / kQThreads, (int64_t)sms * 8));
  if (e == cudaSuccess && p > 0) {
    const unsigned sgrid = (unsigned)std::min<uint64_t>(cap / kQThreads, (uint64_t)sms * 8);
    unsigned long long *k1 = reinterpret_cast<unsigned long long*>(buf + at_keys), *k2 = k1 + np;
    uint32_t *i1 = reinterpret_cast<uint32_t*>(buf + at_idx1), *i2 = reinterpret_cast<uint32_t*>(buf + at_idx2);
    int bits = 1;
    while (bits < 32 && ((uint64_t)p - 1) >> bits) ++bits;
    cell_count_kernel<<<grid, kQThreads, 0, s>>>(train, p, inv_c, cells, mask, i2, dc);
    cell_starts_kernel<<<sgrid, kQThreads, 0, s>>>(cells, mask, total);
    run_keys_kernel<<<grid, kQThreads, 0, s>>>(cells, i2, p, k1, i1);
    ok(cudaGetLastError());
    if (e == cudaSuccess)  // the runs' total is the number of points
      ok(radix_sort_pairs(k1, i1, k2, i2, total, np, bits, reinterpret_cast<uint32_t*>(buf + at_work), sms, dc, s));
    if (e == cudaSuccess) run_fill_kernel<<<grid, kQThreads, 0, s>>>(train, p, i1, runs, dc);
    ok(cudaGetLastError());
  }
  if (e == cudaSuccess) {
    QueryArgs a;
    a.g = g;
    a.inv_c = inv_c;
    a.runs = runs;
    a.cells = cells;
    a.mask = mask;
    a.pts = qp;
    a.q = q;
    a.alpha = out;
    a.alpha0 = (float)params->alpha0;
    a.dc = dc;
    const unsigned qgrid = (unsigned)std::max<int64_t>(1, std::min<int64_t>((q + kQWarps - 1) / kQWarps, (int64_t)sms * 6));
    // six CTAs per SM, whose columns take up to 203 KB of the shared memory
    ok(cudaFuncSetAttribute(query_points_kernel, cudaFuncAttributePreferredSharedMemoryCarveout, cudaSharedmemCarveoutMaxShared));
    query_points_kernel<<<qgrid, kQThreads, sizeof(float) * 32 * (g.K1 + 1) * kQWarps, s>>>(a);
    ok(cudaGetLastError());
  }
  if (e == cudaSuccess && !dev_out)
    ok(cudaMemcpyAsync(alpha_out, out, sizeof(float) * g.K1 * q, cudaMemcpyDeviceToHost, s));
  int32_t derr = 0;
  if (e == cudaSuccess) ok(cudaMemcpyAsync(&derr, &dc->err, sizeof(derr), cudaMemcpyDeviceToHost, s));
  if (e == cudaSuccess) ok(cudaStreamSynchronize(s));
  if (buf) cudaFree(buf);
  if (prev >= 0) cudaSetDevice(prev);
  if (e != cudaSuccess) {
    char msg[256];
    snprintf(msg, sizeof(msg), "query points: %s", cudaGetErrorString(e));
    return fail(SBKI_ERR_CUDA, msg);
  }
  if (derr != 0) return fail((sbki_status)derr, "query points: device error");
  return SBKI_OK;
}
