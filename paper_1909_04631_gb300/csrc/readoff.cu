// Read-off of the Dirichlet posterior at query points: Eq. (variance) for the
// mean E[theta^k] = alpha^k / sum alpha and V[theta^k] = E (1 - E) / (sum alpha + 1),
// the occupancy probability of Sec. V-C (sum of the occupied-class
// probabilities), the argmax label (ties to the lowest class) and the
// free / unknown / occupied state with the thresholds of Sec. V-A.  A voxel
// with no kernel mass (never reached, or outside every allocated block) reads
// as the prior alpha_0 and is unknown.
//
// The outputs of 32 consecutive query points are contiguous, so a warp takes
// 32 points: first a lane per point (hash lookup, the class column into shared
// memory, the sums), then a lane per output element, which makes every store
// of the [q, K+1] arrays a full line.  The quotients are formed in pairs of
// FP32 values (hi + lo, about 2^-46 relative), whose rounding to FP32 is that
// of the FP64 quotient in all but a 2^-20 share of the cases; FP64 itself runs
// at 1/64 of the FP32 rate on this chip and bound the kernel before, a lane's
// stores one sector each: 1.23M points x 20 classes, every output, took
// 1563 us a call and take 146 us (344 B a point: 62 us at the copy rate).  What
// bounds it now is instruction issue (88 % of the slots, 113 warp instructions a
// point); DRAM runs at 34 %.
// Points whose values leave the pairs' safe range (and states within 1e-9 of a
// threshold) take the FP64 form.
#include <algorithm>

#include "sbki_internal.cuh"

namespace sbki {
namespace {

struct QueryArgs {
  Geom g;
  float alpha0;
  double free_thresh, occ_thresh;
  const unsigned long long* hkeys;
  const int32_t* hvals;
  int64_t hash_cap;
  const float* alpha;
  const float* xyz;
  int64_t q;
  float* probs;
  float* var;
  float* mode;
  int32_t* label;
  float* p_occ;
  int32_t* state;
  int map;
};

__device__ int32_t lookup_block(const QueryArgs& a, unsigned long long key) {
  uint32_t slot = hash_slot(key, a.hash_cap);
  for (int probe = 0; probe < kMaxProbes; ++probe) {
    const unsigned long long k = a.hkeys[slot];
    if (k == key) return a.hvals[slot];
    if (k == kEmpty) return -1;
    slot = (uint32_t)((slot + 1) & (uint32_t)(a.hash_cap - 1));
  }
  return -1;
}

// An unevaluated sum hi + lo of two FP32 values, |lo| at most half an ulp of hi
// (Dekker's and Knuth's error-free sums and products).
struct Two {
  float hi, lo;
};
__device__ __forceinline__ Two two_sum(float a, float b) {  // a + b exactly
  const float s = __fadd_rn(a, b), bb = __fsub_rn(s, a);
  return {s, __fadd_rn(__fsub_rn(a, __fsub_rn(s, bb)), __fsub_rn(b, bb))};
}
__device__ __forceinline__ Two renorm(float hi, float lo) {
  const float s = __fadd_rn(hi, lo);
  return {s, __fsub_rn(lo, __fsub_rn(s, hi))};
}
__device__ __forceinline__ Two add(Two a, float b) {
  const Two s = two_sum(a.hi, b);
  return renorm(s.hi, __fadd_rn(s.lo, a.lo));
}
__device__ __forceinline__ Two mul(Two a, Two b) {
  const float p = __fmul_rn(a.hi, b.hi);
  const float e = __fmaf_rn(a.hi, b.hi, -p);
  return renorm(p, __fadd_rn(e, __fmaf_rn(a.hi, b.lo, __fmul_rn(a.lo, b.hi))));
}
__device__ __forceinline__ Two recip(Two a) {  // one correction of the rounded reciprocal
  const float r = __frcp_rn(a.hi);
  const float e = __fmaf_rn(-r, a.lo, __fmaf_rn(-r, a.hi, 1.0f));
  return renorm(r, __fmul_rn(r, e));
}

constexpr int kQWarps = 8;
// Range in which the pairs keep their accuracy: every alpha zero or at least
// kMinAlpha, and their sum at most kMaxSum (no factor or residual leaves FP32's
// normal range; far outside what scans or the default prior produce).
constexpr float kMinAlpha = 0x1p-30f, kMaxSum = 0x1p40f;
constexpr int kRowWide = 1 << 8, kRowMode = 1 << 9;  // row flags above the argmax class

// per warp: 32 rows of alpha (odd stride: no bank conflict by lane), then the rows' scalars
__host__ __device__ constexpr int row_stride(int K1) { return K1 | 1; }
__host__ __device__ constexpr size_t warp_smem(int K1) { return 32 * (sizeof(float) * (size_t)(row_stride(K1) + 3) + 2 * sizeof(float4)); }

__global__ void __launch_bounds__(32 * kQWarps) query_kernel(QueryArgs a, uint32_t recip_k1) {
  extern __shared__ __align__(16) unsigned char q_smem[];
  const Geom& g = a.g;
  const int K1 = g.K1, stride = row_stride(K1);
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  unsigned char* base = q_smem + warp * warp_smem(K1);
  float4* s_sum = reinterpret_cast<float4*>(base);  // (1/S, S), or S in FP64 in the first two words of a wide row
  float4* s_rest = s_sum + 32;                      // (S without the largest class, 1/(S + 1))
  float2* s_mode = reinterpret_cast<float2*>(s_rest + 32);  // 1 / sum (alpha - 1)
  int* s_flag = reinterpret_cast<int*>(s_mode + 32);
  float* s_al = reinterpret_cast<float*>(s_flag + 32);
  const int64_t i0 = ((int64_t)blockIdx.x * kQWarps + warp) * 32, i = i0 + lane;
  if (i0 >= a.q) return;  // warp-uniform
  const int rows = (int)min((int64_t)32, a.q - i0);
  if (i < a.q) {
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
      pool = lookup_block(a, pack_block(v[0] >> g.B_shift, v[1] >> g.B_shift, v[2] >> g.B_shift, a.map));
      const int m = g.B - 1;
      local = (((v[2] & m) << g.B_shift) + (v[1] & m)) * g.B + (v[0] & m);
    }
    const float* inc = pool >= 0 ? a.alpha + (size_t)pool * K1 * g.B3 + local : nullptr;
    float* row = s_al + lane * stride;
    float amax = -1.f, amin = 3.0e38f;
    bool any = false, safe = true;  // any: a class with kernel mass
    int best = 0;
    constexpr int kAhead = 8;  // class values in flight per lane
    for (int k0 = 0; k0 < K1; k0 += kAhead) {
      float d[kAhead];
#pragma unroll
      for (int j = 0; j < kAhead; ++j) d[j] = (inc && k0 + j < K1) ? __ldg(inc + (size_t)(k0 + j) * g.B3) : 0.f;
#pragma unroll
      for (int j = 0; j < kAhead; ++j)
        if (k0 + j < K1) {
          const float al = a.alpha0 + d[j];
          row[k0 + j] = al;
          any = any || d[j] > 0.f;
          safe = safe && d[j] >= 0.f && (al >= kMinAlpha || al == 0.f);
          amin = fminf(amin, al);
          if (al > amax) {
            amax = al;
            best = k0 + j;
          }
        }
    }
    // T: every class but the largest, so that S - alpha of the largest class does not cancel
    Two T = {0.f, 0.f}, M = {0.f, 0.f};
    for (int k = 0; k < K1; ++k)
      if (k != best) T = add(T, row[k]);
    const Two S = add(T, amax);
    const bool mode_ok = amin > 1.0f;
    safe = safe && S.hi >= kMinAlpha && S.hi <= kMaxSum;  // false for NaN
    double wide_s = 0.0, wide_po = 0.0, mass = 0.0;  // the FP64 form
    auto wide = [&]() {
      for (int k = 0; k < K1; ++k) {
        wide_s += row[k];
        mass += inc ? inc[(size_t)k * g.B3] : 0.f;
      }
      for (int k = 1; k < K1; ++k) wide_po += (double)row[k] / wide_s;
    };
    float po;
    int st = 1;
    if (safe) {
      const Two iS = recip(S);
      Two occ = T;  // classes 1..K
      if (best != 0) {
        occ = add(T, -row[0]);
        occ = add(occ, amax);
      }
      const Two p = mul(occ, iS);
      po = p.hi + p.lo;
      if (a.state && any) {
        double pd = (double)p.hi + (double)p.lo;
        if (fabs(pd - a.free_thresh) < 1e-9 || fabs(pd - a.occ_thresh) < 1e-9) {
          wide();
          pd = wide_po;
        }
        st = pd < a.free_thresh ? 0 : (pd > a.occ_thresh ? 2 : 1);
      }
      if (a.mode && mode_ok) {
        for (int k = 0; k < K1; ++k) {
          const Two t = two_sum(row[k], -1.0f);
          const Two m = add(M, t.hi);
          M = renorm(m.hi, m.lo + t.lo);
        }
        const Two iM = recip(M);
        s_mode[lane] = make_float2(iM.hi, iM.lo);
      }
      const Two iS1 = recip(add(S, 1.0f));
      s_sum[lane] = make_float4(iS.hi, iS.lo, S.hi, S.lo);
      s_rest[lane] = make_float4(T.hi, T.lo, iS1.hi, iS1.lo);
    } else {
      wide();
      po = (float)wide_po;
      if (mass > 0.0) st = wide_po < a.free_thresh ? 0 : (wide_po > a.occ_thresh ? 2 : 1);
      *reinterpret_cast<double*>(s_sum + lane) = wide_s;
    }
    s_flag[lane] = best | (safe ? 0 : kRowWide) | (mode_ok ? kRowMode : 0);
    if (a.label) a.label[i] = best;
    if (a.p_occ) a.p_occ[i] = po;
    if (a.state) a.state[i] = st;
  }
  __syncwarp();
  // a lane per output element of the warp's contiguous rows
  const int64_t o0 = i0 * K1;
  const int total = rows * K1;
  for (int e = lane; e < total; e += 32) {
    const int r = (int)small_div((uint32_t)e, recip_k1), k = e - r * K1;
    const int flag = s_flag[r];
    const float al = s_al[r * stride + k];
    float mean, var = 0.f, mode = __int_as_float(0x7fc00000);
    if (flag & kRowWide) {
      const double S = *reinterpret_cast<const double*>(s_sum + r), al64 = al;
      mean = (float)(al64 / S);
      if (a.var) var = (float)(al64 * (S - al64) / (S * S * (S + 1.0)));
      if (flag & kRowMode) mode = (float)((al64 - 1.0) / (S - (double)K1));
    } else {
      const float4 sm = s_sum[r];
      const Two iS = {sm.x, sm.y}, p = mul({al, 0.f}, iS);
      mean = p.hi;
      if (a.var) {
        const float4 rs = s_rest[r];
        Two rest = {rs.x, rs.y};  // S - alpha
        if (k != (flag & 0xff)) {
          rest = two_sum(sm.z, -al);
          rest = renorm(rest.hi, rest.lo + sm.w);
        }
        var = mul(mul(p, mul(rest, iS)), {rs.z, rs.w}).hi;
      }
      if (a.mode && (flag & kRowMode)) {
        const float2 iM = s_mode[r];
        mode = mul(two_sum(al, -1.0f), {iM.x, iM.y}).hi;
      }
    }
    a.probs[o0 + e] = mean;
    if (a.var) a.var[o0 + e] = var;
    if (a.mode) a.mode[o0 + e] = mode;
  }
}

}  // namespace

cudaError_t launch_query(const MapState& m, const float* xyz, int64_t q, float* probs, float* var, float* mode,
                         int32_t* label, float* p_occ, int32_t* state) {
  if (q <= 0) return cudaSuccess;
  QueryArgs a;
  a.g = m.g;
  a.alpha0 = (float)m.prm.alpha0;
  a.free_thresh = m.prm.free_thresh;
  a.occ_thresh = m.prm.occ_thresh;
  a.hkeys = m.hkeys;
  a.hvals = m.hvals;
  a.hash_cap = m.hash_cap;
  a.alpha = m.alpha;
  a.xyz = xyz;
  a.q = q;
  a.probs = probs;
  a.var = var;
  a.mode = mode;
  a.label = label;
  a.p_occ = p_occ;
  a.state = state;
  a.map = m.active_map;
  // 14 to 35 KB a CTA for 2 to 32 classes: under the 48 KB that need no opt-in
  static_assert(kQWarps * warp_smem(kMaxClasses) <= 48 * 1024, "read-off shared memory");
  const int K1 = m.g.K1;
  const uint32_t recip_k1 = ((1u << 20) + (uint32_t)K1 - 1u) / (uint32_t)K1;
  const int64_t per = 32 * kQWarps;
  query_kernel<<<(unsigned)((q + per - 1) / per), 32 * kQWarps, kQWarps * warp_smem(K1), m.stream>>>(a, recip_k1);
  return cudaGetLastError();
}

cudaError_t launch_gather_alpha(const MapState& m, float* out, int64_t nblocks) {
  return cudaMemcpyAsync(out, m.alpha, sizeof(float) * (size_t)nblocks * m.g.K1 * m.g.B3, cudaMemcpyDeviceToDevice,
                         m.stream);
}

}  // namespace sbki

namespace sbki {
namespace {

// 1 for every pool block of the selected map (scanned into output rows next)
__global__ void export_flags_kernel(const unsigned long long* __restrict__ pool_keys, uint32_t nb, int map,
                                    uint32_t* __restrict__ flags) {
  for (uint32_t b = blockIdx.x * blockDim.x + threadIdx.x; b < nb; b += gridDim.x * blockDim.x)
    flags[b] = map_of_block(pool_keys[b]) == map ? 1u : 0u;
}

// One row per voxel of every selected block: key (x, y, z) and alpha with prior.
__global__ void export_rows_kernel(const unsigned long long* __restrict__ pool_keys, const uint32_t* __restrict__ rowb,
                                   uint32_t nb, int map, Geom g, const float* __restrict__ alpha, float alpha0,
                                   int64_t* __restrict__ keys, float* __restrict__ out) {
  const int64_t total = (int64_t)nb * g.B3;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
    const uint32_t b = (uint32_t)(e / g.B3);
    const int li = (int)(e - (int64_t)b * g.B3);
    const unsigned long long k = pool_keys[b];
    if (map_of_block(k) != map) continue;
    const int64_t row = (int64_t)rowb[b] * g.B3 + li;
    int32_t bx, by, bz;
    unpack_block(k, bx, by, bz);
    if (keys) {
      keys[3 * row] = (int64_t)bx * g.B + li % g.B;
      keys[3 * row + 1] = (int64_t)by * g.B + (li / g.B) % g.B;
      keys[3 * row + 2] = (int64_t)bz * g.B + li / (g.B * g.B);
    }
    if (out)
      for (int c = 0; c < g.K1; ++c)
        out[row * g.K1 + c] = __fadd_rn(alpha0, alpha[((size_t)b * g.K1 + c) * g.B3 + li]);
  }
}

}  // namespace

cudaError_t launch_export_rows(const MapState& m, uint32_t nb, uint32_t* rowb, void* scan_tmp, int64_t* keys,
                               float* out) {
  const unsigned grid = (unsigned)std::max<int64_t>(1, std::min<int64_t>(((int64_t)nb + 255) / 256, 4096));
  export_flags_kernel<<<grid, 256, 0, m.stream>>>(m.pool_keys, nb, m.active_map, rowb);
  cudaError_t e = exclusive_scan_u32(rowb, nb, scan_tmp, m.stream);
  if (e != cudaSuccess) return e;
  const int64_t total = (int64_t)nb * m.g.B3;
  const unsigned g2 = (unsigned)std::max<int64_t>(1, std::min<int64_t>((total + 255) / 256, (int64_t)m.sm_count * 16));
  export_rows_kernel<<<g2, 256, 0, m.stream>>>(m.pool_keys, rowb, nb, m.active_map, m.g, m.alpha,
                                               (float)m.prm.alpha0, keys, out);
  return cudaGetLastError();
}

}  // namespace sbki
