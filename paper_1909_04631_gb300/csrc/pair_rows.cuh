// Pieces of the pair form shared by the fast accumulation and its backward pass,
// so both enumerate exactly the same pairs: half a warp per training point, two
// voxels adjacent in x per lane, candidates from mirrored lists.  The layout is
// described at the accumulation (accumulate_points.cu), which builds the lists.
#pragma once
#include "point_common.cuh"

namespace sbki {

constexpr float kFar = 1.0e30f;    // e^2 of the padding row (its e: 1e15)
constexpr float kFarOffset = 1.0e15f;
constexpr int kFastParts = 8;      // sub-voxel parts per axis of the candidate lists
constexpr int kGroup = 8;          // points whose rows one warp forms at once (4 lanes each)
constexpr int kFastAxis = 7;       // offsets per axis
constexpr int kSlotBytes = 256;    // one point's rows and scalars
constexpr uint32_t kYRows = 64u, kZRows = 128u, kScalars = 192u;  // byte offsets in a slot (X rows at 0)
constexpr int kFastPad = 128;      // entries per list at most: 8 rounds of 16 lanes
constexpr int kFastLists = kFastParts * (kFastParts / 2) * (kFastParts / 2);
// entries of a handle's lists: its tables and a list of padding
__host__ __device__ constexpr int list_entries(int tables, int pad) { return (tables * kFastLists + 1) * pad; }
// entry: bits 3-5 8 jy, bits 6-7 jx, bits 8-15 the Z row's byte offset in the slot
constexpr uint32_t kPadEntry = (8u * kFastAxis) | (kZRows << 8);  // Y padding row

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float2 lds_f2(uint32_t a) {
  float2 v;
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ uint4 lds_u4(uint32_t a) {
  uint4 v;
  asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u16(uint32_t a) {
  uint16_t v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ uint32_t lds_u32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float r;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// One axis of a training point: its voxel, the compensated offset to that
// voxel's centre and its sub-voxel part.
struct AxisFrame {
  int v0, part;
  float hi, lo;
};
__device__ __forceinline__ AxisFrame axis_frame(float x, const Geom& g) {
  AxisFrame f;
  f.v0 = floor_small(__fmul_rn(x, g.inv_res));
  centre_offset0(f.v0, x, g, f.hi, f.lo);
  const float phi = 0.5f - __fmul_rn(__fadd_rn(f.hi, f.lo), g.inv_res);
  f.part = min(kFastParts - 1, max(0, floor_small(phi * (float)kFastParts)));
  return f;
}

// FP64 re-decision of voxel j (0 or 1) of the pair that entry e names (rare;
// the point is loaded again and its mirrored rows are undone).
static __device__ __noinline__ bool band_decide(uint32_t e, int j, const float4* train, uint32_t i, int R, const Geom& g,
                                         double l2_64) {
  const float4 p = train[i];
  const AxisFrame fx = axis_frame(p.x, g), fy = axis_frame(p.y, g), fz = axis_frame(p.z, g);
  int jx = (int)(e >> 6) & 3, jy = (int)(e >> 3) & 7, jz = (int)((e >> 8) - kZRows) >> 3;
  const int odd = (fx.v0 - R) & 1;
  if (odd) jx = R - jx;
  if (fy.part >= kFastParts / 2) jy = 2 * R - jy;
  if (fz.part >= kFastParts / 2) jz = 2 * R - jz;
  return in_support64_call(fx.v0 - R - odd + 2 * jx + j, fy.v0 + jy - R, fz.v0 + jz - R, p.x, p.y, p.z, g.res64,
                           l2_64);
}

// Forms one lane's share of a point's rows (role 0, 1: the halves of X, 2: Y,
// 3: Z; f the frame of that axis, gl the point's place in the group).  kSquare:
// the rows hold e^2, else e.  cls is added to the Z parts.  Returns the axis's
// part for the list (mirrored where the rows are).
template <bool kSquare>
__device__ __forceinline__ int form_rows(unsigned char* slot, int gl, int role, const AxisFrame& f, uint32_t cls, int R,
                                         const Geom& g) {
  const int v0 = f.v0, m = g.B - 1, na = 2 * R + 1;
  const int vrel = v0 - (((v0 >> g.B_shift) - 1) << g.B_shift);  // from the block before the point's
  auto value = [](float e) { return kSquare ? __fmul_rn(e, e) : e; };
  if (role < 2) {
    const int odd = (v0 - R) & 1;
    float4* r = reinterpret_cast<float4*>(slot);
#pragma unroll
    for (int t = 0; t < 2; ++t) {
      const int u = 2 * role + ((gl + t) & 1);  // alternating order: the stores spread over the banks
      const int d = -R - odd + 2 * u, at = odd ? R - u : u;
      const float ea = centre_offset_at(d, f.hi, f.lo, g), eb = centre_offset_at(d + 1, f.hi, f.lo, g);
      const int v = vrel + d;
      if (at >= 0)  // a pair past the window has no mirror image (and is in no list)
        r[at] = make_float4(value(ea), value(eb),
                            __uint_as_float((4u << 24) * (uint32_t)(v >> g.B_shift) + (uint32_t)(v & m)), 0.f);
    }
    return odd ? kFastParts - 1 - f.part : f.part;
  }
  const bool flip = f.part >= kFastParts / 2;
  const int axshift = role == 2 ? g.B_shift : 2 * g.B_shift;
  const uint32_t dmul = (role == 2 ? 12u : 36u) << 24, base = role == 3 ? cls : 0u;
  float2* r = reinterpret_cast<float2*>(slot + (role == 2 ? kYRows : kZRows)) + (flip ? 2 * R : 0);
  const int sgn = flip ? -1 : 1;
  int j = min(gl, na - 1);  // a lane-dependent order, so the lanes of one store spread over the banks
#pragma unroll
  for (int t = 0; t < kFastAxis; ++t) {
    if (t < na) {
      const float e = centre_offset_at(j - R, f.hi, f.lo, g);
      const int v = vrel + j - R;
      r[sgn * j] = make_float2(
          value(e), __uint_as_float(dmul * (uint32_t)(v >> g.B_shift) + (((uint32_t)(v & m) << axshift) + base)));
      j = j + 1 == na ? 0 : j + 1;
    }
  }
  return flip ? kFastParts - 1 - f.part : f.part;
}

}  // namespace sbki
