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

// kCullBox, kCullTube: the plain safety is the solid's own, and the entry has an upper bound too;
// kCullOther: the bounding box tells misses, plain_other (nav.cu) the safety within a wider margin;
// kCullNever: the same, but what is left has no certified binary32 evaluation, only a binary64 one.
enum : int32_t { kCullBox = 0, kCullTube = 1, kCullOther = 2, kCullNever = 3 };

// Per node: the world frame's rotation and translation, half extents of the bounding box around the
// origin of the solid's frame.
struct alignas(16) Cull {
  float R[9], t[3];
  float e[3], rmin;  // rmin: inner radius of a full tube
  float margin;      // 1e-6 + 4e-6 (|t|_1 + |e|_1): the placement's share of the margin (mm)
  int32_t tag, solid;
  int32_t family;  // 0 box, 1 trd/trap, 2 tube, 3 cone and polycone
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

// The times at which the ray q + t e (r2 = |q_xy|^2, b = q_xy e_xy, a = |e_xy|^2) enters and leaves
// radius R in plain binary32; wide: not later and not earlier than in truth, else the other way round.
// The discriminant's rounding is below 10 2^-24 a (r2 + R^2); dt is what its bound can move a time by.
__device__ __forceinline__ bool plain_circle(float r2, float b, float a, float R, bool wide, float& t0, float& t1, float& dt) {
  const float err = 2e-6f * a * fmaf(R, R, r2);
  const float disc = fmaf(b, b, -a * fmaf(-R, R, r2)) + (wide ? err : -err);
  const float s = sqrtf(fmaxf(disc, 0.f)), inv = __fdividef(1.f, a);
  t0 = (-b - s) * inv;
  t1 = (-b + s) * inv;
  dt = err * __fdividef(1.f, s * a);
  return disc > 0.f;
}

// The same look with bounds on the entry: not before `from`, and, when it is finite, not after `by`
// (a ray from a point certainly outside that certainly goes in).  A box is entered where the ray enters
// the box widened and shrunk by the margin; a full tube through its outer or its inner wall likewise
// (steep rays and rays through the end planes get no upper bound).
__device__ __forceinline__ bool plain_entry(const Cull& C, const PlainTrack& p, const PlainLocal& L, float& from,
                                            float& by) {
  float lo = 0.f, hi = f32::BIG, e[3], inv[3];
#pragma unroll
  for (int i = 0; i < 3; i++) {
    const float d = e[i] = fmaf(C.R[6 + i], p.w, fmaf(C.R[3 + i], p.v, C.R[i] * p.u));
    inv[i] = __fdividef(1.f, d);
    const float E = C.e[i] + L.margin, a = (-E - L.q[i]) * inv[i], b = (E - L.q[i]) * inv[i];
    lo = fmaxf(lo, fminf(a, b));
    hi = fminf(hi, fmaxf(a, b));
  }
  from = lo;
  by = f32::BIG;
  if (lo > hi) return true;
  const float m = L.margin;
  if (C.tag == kCullBox) {
    float l = -f32::BIG, h = f32::BIG;
    bool out = false;
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const float E = C.e[i] - m, a = (-E - L.q[i]) * inv[i], b = (E - L.q[i]) * inv[i];
      l = fmaxf(l, fminf(a, b));
      h = fminf(h, fmaxf(a, b));
      out |= fabsf(L.q[i]) > C.e[i] + m;
    }
    if (out && l <= h && l > 0.f) by = l;
  } else if (C.tag == kCullTube) {
    const float r2 = fmaf(L.q[0], L.q[0], L.q[1] * L.q[1]), a = fmaf(e[0], e[0], e[1] * e[1]);
    const float b = fmaf(L.q[0], e[0], L.q[1] * e[1]);
    if (a > 0.01f) {
      const float Ro = C.e[0], Ri = C.rmin, tm = 2.f * m * rsqrtf(a);  // the rounding of a time
      float t0, t1, dt, in = f32::BIG, dz = 0.f;  // in: certainly between the walls by then
      if (r2 > (Ro + m) * (Ro + m)) {
        if (!plain_circle(r2, b, a, Ro + m, true, t0, t1, dt) || t1 + tm < 0.f) return true;
        from = fmaxf(from, t0 - tm);
        if (Ro > m && plain_circle(r2, b, a, Ro - m, false, t0, t1, dt) && t0 > tm) {
          in = t0 + tm;
          dz = dt;
        }
      } else if (Ri > m && r2 < (Ri - m) * (Ri - m)) {
        if (plain_circle(r2, b, a, Ri - m, false, t0, t1, dt)) from = fmaxf(from, t1 - tm);
        plain_circle(r2, b, a, Ri + m, true, t0, t1, dt);
        in = t1 + tm;
        dz = dt;
      }
      if (Ro - Ri > 4.f * m && fabsf(fmaf(in, e[2], L.q[2])) < C.e[2] - 24.f * m - 2.f * dz) by = in;
    }
  }
  return from > hi;
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
