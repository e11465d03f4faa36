// Exact integer pieces of the downsampling, shared by its two forms (sorted
// items, ingest.cu; occupied tiles, tiles.cu): decomposition of FP32 values,
// 128-bit sums, the one rounding of a mean, the fixed-point unit of a tile, and
// the operations that decide a beam's samples.
#pragma once
#include "exact_round.cuh"
#include "sbki_internal.cuh"

namespace sbki {

__device__ __forceinline__ int floor_i(float v) { return (int)floorf(v); }

// scan of global point gi: the last s with off[s] <= gi (empty scans are skipped)
__device__ __forceinline__ int scan_of(const int64_t* off, int ns, int64_t gi) {
  int lo = 0, hi = ns - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (off[mid] <= gi) lo = mid;
    else hi = mid - 1;
  }
  return lo;
}

// number of j >= 1 with fp32(j) * s < r  (the set is a prefix since fp32(j)*s is monotone in j)
__device__ __forceinline__ uint32_t free_count(float r, float s) {
  if (!(r > 0.0f)) return 0;
  float q = __fdiv_rn(r, s);
  int j = q < 1.6e7f ? (int)q : 16000000;
  for (int it = 0; it < 4 && j > 0 && !(__fmul_rn((float)j, s) < r); ++it) --j;
  for (int it = 0; it < 4 && __fmul_rn((float)(j + 1), s) < r; ++it) ++j;
  return (uint32_t)(j < 0 ? 0 : j);
}

struct U128 {
  unsigned long long lo, hi;
};

// |v| = m 2^e (m < 2^24 integer); returns false for zero
__device__ __forceinline__ bool decompose(float v, unsigned& m, int& e) {
  const unsigned b = __float_as_uint(v) & 0x7fffffffu;
  if (b == 0u) return false;
  const unsigned E = b >> 23;
  m = (b & 0x7fffffu) | (E ? 0x800000u : 0u);
  e = E ? (int)E - 150 : -149;
  return true;
}

__device__ __forceinline__ void u128_add(U128& t, unsigned long long lo, unsigned long long hi) {
  t.lo += lo;
  t.hi += hi + (t.lo < lo ? 1ull : 0ull);
}

// t += m 2^sh, 0 <= sh <= 103
__device__ __forceinline__ void u128_add_shifted(U128& t, unsigned long long m, int sh) {
  if (sh == 0) u128_add(t, m, 0ull);
  else if (sh < 64) u128_add(t, m << sh, m >> (64 - sh));
  else u128_add(t, 0ull, m << (sh - 64));
}

__device__ __forceinline__ int bitlen64(unsigned long long v) { return v ? 64 - __clzll((long long)v) : 0; }

// round(T 2^s / n) to FP32; false when the result is below the normal range
__device__ inline bool round_mean(U128 T, unsigned long long n, int s, float& out) {
  const int bt = T.hi ? 64 + bitlen64(T.hi) : bitlen64(T.lo);
  const int bn = bitlen64(n);
  const int k = 26 + bn - bt;  // q = floor(T 2^k / n) in [2^24, 2^27)
  unsigned long long q;
  bool sticky;
  if (k >= 0) {
    const unsigned long long num = T.lo << k;  // bt + k = 26 + bn <= 58 bits
    q = num / n;
    sticky = num - q * n != 0ull;
  } else {
    const int m = -k;
    unsigned long long ts, lost;
    if (m < 64) {
      ts = (T.lo >> m) | (m ? (T.hi << (64 - m)) : 0ull);
      lost = T.lo & ((1ull << m) - 1ull);
    } else {
      ts = T.hi >> (m - 64);
      lost = T.lo | (T.hi & ((m - 64 == 0) ? 0ull : ((1ull << (m - 64)) - 1ull)));
    }
    q = ts / n;
    sticky = lost != 0ull || ts - q * n != 0ull;
  }
  const int qb = bitlen64(q);
  if (qb - 1 - k + s < -126) return false;
  const int sh = qb - 24;
  unsigned long long mant = q >> sh;
  const unsigned long long rb = q & ((1ull << sh) - 1ull), half = 1ull << (sh - 1);
  if (rb > half || (rb == half && (sticky || (mant & 1ull)))) mant += 1ull;
  int e = sh - k + s;
  if (mant == (1ull << 24)) {
    mant >>= 1;
    e += 1;
  }
  out = ldexpf((float)mant, e);
  return true;
}

// (neg ? -1 : 1) round(W 2^-149 / n) to FP32, nearest with ties to even, for
// the 512-bit integer W of 16 32-bit words (lowest first) and 0 < n < 2^32.
static __device__ __noinline__ float round_words(const uint32_t* w, bool neg, unsigned long long n) {
  // quotient of (sum 2^96) / n, limb by limb from the top, in 19 limbs
  uint32_t q[19];
  unsigned long long r = 0ull;
  for (int j = 18; j >= 0; --j) {
    const unsigned long long cur = (r << 32) | (j >= 3 ? w[j - 3] : 0u);
    q[j] = (uint32_t)(cur / n);
    r = cur - (unsigned long long)q[j] * n;
  }
  int qb = 0;
  for (int j = 18; j >= 0 && !qb; --j)
    if (q[j]) qb = 32 * j + 32 - __clz((int)q[j]);
  if (qb == 0) return 0.0f;
  // value = q 2^(-149 - 96); keep 24 bits, fewer for a subnormal result
  const int lead = qb - 1 - 245;
  int keep = lead < -126 ? 24 - (-126 - lead) : 24;
  if (keep < 0) keep = 0;
  const int drop = qb - keep;
  auto bit = [&](int i) -> unsigned { return i >= 0 ? (q[i >> 5] >> (i & 31)) & 1u : 0u; };
  unsigned long long mant = 0ull;
  for (int i = qb - 1; i >= drop; --i) mant = (mant << 1) | bit(i);
  bool sticky = r != 0ull;
  for (int i = 0; i < drop - 1 && !sticky; ++i) sticky = bit(i) != 0u;
  if (bit(drop - 1) && (sticky || (mant & 1ull))) mant += 1ull;
  const float f = ldexpf((float)mant, drop - 245);
  return neg ? -f : f;
}

__device__ __forceinline__ float axis_of(const float4& p, int ax) { return ax == 0 ? p.x : (ax == 1 ? p.y : p.z); }

struct AxisAcc {
  int emin, emax;  // range of the members' last-mantissa-bit exponents
  bool neg, pos;   // a member below / above zero
  __device__ void init() {
    emin = 1 << 20;
    emax = -(1 << 20);
    neg = pos = false;
  }
  __device__ void see(float v) {
    unsigned m;
    int e;
    if (decompose(v, m, e)) {
      emin = min(emin, e);
      emax = max(emax, e);
      neg |= v < 0.0f;
      pos |= v > 0.0f;
    }
  }
  __device__ bool empty() const { return emax < emin; }
  __device__ bool fits(uint32_t n) const {  // one sign, and T stays below 2^127
    int lg = 0;
    while (lg < 32 && (1ull << lg) < n) ++lg;
    return empty() || (!(neg && pos) && emax - emin + 24 + lg <= 126);
  }
  __device__ void add(U128& t, float v) const {
    unsigned m;
    int e;
    if (decompose(v, m, e)) u128_add_shifted(t, m, e - emin);
  }
};

// One thread: exact mean of axis ax of members [a, b) for any FP32 input.
// Positive and negative members are summed apart, in 16 32-bit limbs in units
// of 2^-149 each (512 bits), and the smaller sum is subtracted from the larger.
__device__ inline float wide_mean(const float4* __restrict__ items, uint32_t a,
                           uint32_t b, int ax) {
  uint32_t wp[16], wn[16];
  for (int i = 0; i < 16; ++i) wp[i] = wn[i] = 0u;
  for (uint32_t i = a; i < b; ++i) {
    const float v = axis_of(items[i], ax);
    unsigned m;
    int e;
    if (!decompose(v, m, e)) continue;
    uint32_t* w = v < 0.0f ? wn : wp;
    const int sh = e + 149, li = sh >> 5, bi = sh & 31;
    unsigned long long add = (unsigned long long)m << bi;  // < 2^55
    for (int j = li; j < 16 && add; ++j) {
      const unsigned long long t = (unsigned long long)w[j] + (add & 0xffffffffull);
      w[j] = (uint32_t)t;
      add = (add >> 32) + (t >> 32);
    }
  }
  bool neg = false;  // the negative members outweigh the positive ones
  for (int j = 15; j >= 0; --j)
    if (wn[j] != wp[j]) {
      neg = wn[j] > wp[j];
      break;
    }
  uint32_t w[16];
  {
    const uint32_t* hi = neg ? wn : wp;
    const uint32_t* lo = neg ? wp : wn;
    unsigned long long borrow = 0ull;
    for (int j = 0; j < 16; ++j) {
      const unsigned long long d = (unsigned long long)hi[j] - lo[j] - borrow;
      w[j] = (uint32_t)d;
      borrow = (d >> 63) & 1ull;
    }
  }
  return round_words(w, neg, b - a);
}

__device__ inline float finish_axis(const AxisAcc& s, bool fits, U128 T, uint32_t n, const float4* items, uint32_t a, uint32_t b, int ax) {
  if (s.empty()) return 0.0f;
  float f;
  if (fits && round_mean(T, n, s.emin, f)) return s.neg ? -f : f;
  return wide_mean(items, a, b, ax);
}

// Single-pass form for an axis whose first member x0 has |x0| >= 2.5 ds: every
// member of the cell lies within ds (plus rounding) of x0, so it has x0's sign
// and its last mantissa bit's exponent is within [e0 - 1, e0 + 1] (e0: x0's);
// in units of 2^E, E = e0 - 1, every |x| is an integer below 2^26 and a 64-bit
// sum is exact for fewer than 2^32 members.  Cells near a coordinate plane
// (|x0| < 2.5 ds) take the two-pass AxisAcc path.
struct FastAxis {
  bool on, neg;
  int E;
  unsigned long long T;
  __device__ void init(float x0, float lim) {
    unsigned m;
    int e;
    on = fabsf(x0) >= lim && decompose(x0, m, e);
    neg = x0 < 0.0f;
    E = on ? e - 1 : 0;
    T = 0ull;
  }
  __device__ void add(float v) {
    unsigned m;
    int e;
    decompose(v, m, e);  // v != 0: |v| > ds
    T += (unsigned long long)m << (e - E);
  }
  __device__ float finish(uint32_t n) const {
    U128 t;
    t.lo = T;
    t.hi = 0ull;
    float f = 0.0f;
    round_mean(t, n, E, f);
    return neg ? -f : f;
  }
};

__device__ __forceinline__ unsigned long long warp_sum_u64(unsigned long long v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

__device__ __forceinline__ U128 warp_sum_u128(U128 t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long lo = __shfl_xor_sync(0xffffffffu, t.lo, o);
    const unsigned long long hi = __shfl_xor_sync(0xffffffffu, t.hi, o);
    u128_add(t, lo, hi);
  }
  return t;
}

__device__ __forceinline__ void warp_range(AxisAcc& s) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    s.emin = min(s.emin, __shfl_xor_sync(0xffffffffu, s.emin, o));
    s.emax = max(s.emax, __shfl_xor_sync(0xffffffffu, s.emax, o));
  }
  s.neg = __any_sync(0xffffffffu, s.neg);
  s.pos = __any_sync(0xffffffffu, s.pos);
}

// Exact mean of members [a, b) of items, by a whole warp; the mean is valid in
// lane 0.  An axis whose first member has |x0| >= 2.5 ds is summed in one pass
// in 64 bits (FastAxis); any other axis takes its exponent range first, then
// the 128-bit sum, else wide_mean.  The members lie in one cell.
__device__ inline void cell_mean_warp(const float4* __restrict__ items, uint32_t a, uint32_t b, const Geom& g,
                                      float out[3]) {
  const int lane = threadIdx.x & 31;
  const uint32_t n = b - a;
  AxisAcc w[3];
  FastAxis fa[3];
  U128 t[3];
  const float4 p0 = items[a];
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    w[c].init();
    t[c].lo = t[c].hi = 0ull;
    fa[c].init(axis_of(p0, c), g.fast_lim);
  }
  const bool two_pass = !fa[0].on || !fa[1].on || !fa[2].on;  // warp-uniform
  for (uint32_t i = a + lane; i < b; i += 32) {
    const float4 p = items[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      if (fa[c].on) fa[c].add(axis_of(p, c));
      else w[c].see(axis_of(p, c));
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c)
    if (fa[c].on) fa[c].T = warp_sum_u64(fa[c].T);
  bool fit[3] = {false, false, false};
  if (two_pass) {
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      warp_range(w[c]);
      fit[c] = !fa[c].on && w[c].fits(n);
    }
    for (uint32_t i = a + lane; i < b; i += 32) {
      const float4 p = items[i];
#pragma unroll
      for (int c = 0; c < 3; ++c)
        if (fit[c]) w[c].add(t[c], axis_of(p, c));
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) t[c] = warp_sum_u128(t[c]);
  }
  if (lane == 0)
    for (int c = 0; c < 3; ++c)
      out[c] = fa[c].on ? fa[c].finish(n) : finish_axis(w[c], fit[c], t[c], n, items, a, b, c);
}

constexpr int kSegShift = 24;      // binades between a tile's |x| bound and its members' smallest last bit
constexpr uint32_t kSegBad = 2u;
// The unit 2^E of a tile of 8^3 cells per axis: E lies kSegShift + 23 below the
// exponent of U = (8 |t| + 10) ds, an upper bound of |x| in the tile (t: the tile
// index on that axis), so x 2^-E is below 2^48.  meta holds E + 256 of axis a in
// bits 2 + 9a; scale the factors 2^-E; bad is kSegBad when a scale is outside
// the FP32 normal range.
struct TileUnit {
  uint32_t meta, bad;
  float scale[3];
};
__device__ __forceinline__ TileUnit unit_of_tile(const int t[3], const Geom& g) {
  TileUnit u;
  u.meta = 0u;
  u.bad = 0u;
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    const int mag = t[a] < 0 ? -t[a] : t[a];
    const float U = __fmul_rn((float)(kTileEdge * mag + kTileEdge + 2), g.ds);
    const int E = (int)(__float_as_uint(U) >> 23) - 150 - kSegShift;  // |x| < U < 2^(E + 48)
    u.meta |= (uint32_t)(E + 256) << (2 + 9 * a);
    const bool ok = E >= -126 && E <= 126;
    u.scale[a] = ok ? __uint_as_float((uint32_t)(127 - E) << 23) : 0.f;
    if (!ok) u.bad = kSegBad;
  }
  return u;
}
__device__ __forceinline__ int meta_E(uint32_t flags, int a) { return (int)((flags >> (2 + 9 * a)) & 511u) - 256; }

}  // namespace sbki
