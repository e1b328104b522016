// nav_cull.cuh -- a plain binary32 look at a daughter before its certified evaluation.
//
// Most daughters of a volume lie off a track's ray and farther away than the nearest one.  Moving a
// track into a daughter's frame in double-float and evaluating its solid there takes about 350
// instructions; the bounding box in plain binary32 takes about 50 and tells, with margins far above
// its rounding, that the ray misses the daughter (its DistanceToIn is then +inf) and, for boxes and
// full tubes, what its safety is within the margin.
#pragma once
#include "gv_desc.h"
#include "solid_fp32.cuh"

namespace gv {

// kCullBox, kCullTube: the plain safety is the solid's own; kCullOther: the bounding box only;
// kCullNever: always evaluated (no binary32 form).
enum : int32_t { kCullBox = 0, kCullTube = 1, kCullOther = 2, kCullNever = 3 };

// Per node: the world frame's rotation and translation, half extents of the bounding box around the
// origin of the solid's frame.
struct alignas(16) Cull {
  float R[9], t[3];
  float e[3], rmin;  // rmin: inner radius of a full tube
  float margin;      // 1e-6 + 4e-6 (|t|_1 + |e|_1): the placement's share of the margin (mm)
  int32_t tag, solid, pad;
};

// A track in world coordinates, plain binary32.
struct PlainTrack {
  float x, y, z, u, v, w, margin;
};
__device__ __forceinline__ PlainTrack plain_track(const f32::TrackF& W) {
  return {W.xh, W.yh, W.zh, W.u, W.v, W.w, 4e-6f * (fabsf(W.xh) + fabsf(W.yh) + fabsf(W.zh))};
}

struct PlainLocal {
  float q[3], margin;
};
__device__ __forceinline__ PlainLocal plain_local(const Cull& C, const PlainTrack& p) {
  const float dx = p.x - C.t[0], dy = p.y - C.t[1], dz = p.z - C.t[2];
  PlainLocal L;
#pragma unroll
  for (int i = 0; i < 3; i++) L.q[i] = fmaf(C.R[6 + i], dz, fmaf(C.R[3 + i], dy, C.R[i] * dx));
  // Rounding of the local point is below 6 2^-24 (|p|_1 + |t|_1); a direction error of 4 2^-24 moves
  // the ray by 2.4e-7 of the distance to the box.  Both are far below this margin.
  L.margin = p.margin + C.margin;
  return L;
}

// Does the ray certainly miss the bounding box?  The slabs are widened by the margin, so that a
// ray that meets the box meets the widened one in binary32 too, and not later: `from` is a lower
// bound of its entry.  `near`: the ray is nearly parallel to a face or starts on the plane of one;
// the certified binary32 results leave some of those to binary64, and whether they do shall not
// depend on this look.
__device__ __forceinline__ bool plain_miss(const Cull& C, const PlainTrack& p, const PlainLocal& L, float& from,
                                           bool& near) {
  float lo = 0.f, hi = f32::BIG, e[3];
  near = false;
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const float d = e[i] = fmaf(C.R[6 + i], p.w, fmaf(C.R[3 + i], p.v, C.R[i] * p.u));
    near |= fabsf(d) <= 1e-6f || fabsf(fabsf(L.q[i]) - C.e[i]) <= L.margin;
    const float inv = __fdividef(1.f, d), E = C.e[i] + L.margin;
    const float a = (-E - L.q[i]) * inv, b = (E - L.q[i]) * inv;
    lo = fmaxf(lo, fminf(a, b));
    hi = fminf(hi, fmaxf(a, b));
  }
  if (C.tag == kCullTube) {
    // A ray that passes the axis beyond the outer radius.  Its distance from the axis is
    // |q x e| / |e_xy|: for |e_xy| above 0.1 the direction's error moves it by less than the margin.
    const float c = L.q[0] * e[1] - L.q[1] * e[0], E = C.e[0] + L.margin, xy = fmaf(e[0], e[0], e[1] * e[1]);
    if (xy > 0.01f && c * c > 1.0001f * E * E * xy) hi = -f32::BIG;
  }
  from = lo;
  return lo > hi;
}

// Is the point certainly outside the bounding box (its code is OUTSIDE)?
__device__ __forceinline__ bool plain_outside(const Cull& C, const PlainLocal& L) {
  return fabsf(L.q[0]) > C.e[0] + L.margin || fabsf(L.q[1]) > C.e[1] + L.margin || fabsf(L.q[2]) > C.e[2] + L.margin;
}

// The safety (largest constraint value) of a box or a full tube, within the margin.
__device__ __forceinline__ float plain_safety(const Cull& C, const PlainLocal& L) {
  if (C.tag == kCullBox)
    return fmaxf(fmaxf(fabsf(L.q[0]) - C.e[0], fabsf(L.q[1]) - C.e[1]), fabsf(L.q[2]) - C.e[2]);
  const float r = sqrtf(fmaf(L.q[0], L.q[0], L.q[1] * L.q[1]));
  const float wall = fmaxf(r - C.e[0], C.rmin > 0.f ? C.rmin - r : -f32::BIG);
  return fmaxf(wall, fabsf(L.q[2]) - C.e[2]);
}

}  // namespace gv
