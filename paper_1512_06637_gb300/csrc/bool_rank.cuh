// bool_rank.cuh -- the binary64 results of a boolean solid from a binary32 ranking (as rank_fp64.cuh
// for primitives), for components that are boxes, trds, traps or two-plane polycones.
//
// Along the ray each component is an interval less at most two others (its hole and the wedge a wide
// phi segment leaves out), whose ends are crossings of its surfaces.  Their order is certified in
// binary32: from the start on, the first end at which the combined set is entered (for an outside
// point) or left (for an inside one) is the distance, and that one crossing is evaluated in binary64.  The
// safety is the one component's that the set operation picks.  Surface starts, sliding rays and
// anything not certain are left to the whole evaluation (bool_query).
#pragma once
#include "rank_fp64.cuh"

namespace gv {
namespace f32 {

// An interval of t with the crossings (ver_dist) at its ends; kVerGoalOut marks an end at which the
// component is left.
struct IvId {
  Val lo, hi;
  uint32_t il, ih;
};
__device__ __forceinline__ IvId ivid_all() { return {{-BIG, 0.f}, {BIG, 0.f}, 0u, 0u}; }
__device__ __forceinline__ IvId ivid_none() { return {{BIG, 0.f}, {-BIG, 0.f}, 0u, 0u}; }
__device__ __forceinline__ bool empty(const IvId& x) { return !(x.lo.v < x.hi.v); }
__device__ __forceinline__ void clip_lo(IvId& x, Val t, uint32_t id, bool& unsure) {
  if (x.lo.v > -BIG && t.v > -BIG && !apart(x.lo, t)) unsure = true;
  if (t.v > x.lo.v) { x.lo = t; x.il = id; }
}
__device__ __forceinline__ void clip_hi(IvId& x, Val t, uint32_t id, bool& unsure) {
  if (x.hi.v < BIG && t.v < BIG && !apart(x.hi, t)) unsure = true;
  if (t.v < x.hi.v) { x.hi = t; x.ih = id; }
}
// The constraint g + t gd <= 0.
__device__ __forceinline__ void clip_half(IvId& x, float g, float E, float gd, float egd, uint32_t id, bool& unsure) {
  if (fabsf(g) <= HF + E && fabsf(gd) <= egd + TAUF) unsure = true;  // along the surface
  if (fabsf(gd) <= egd) {
    if (fabsf(g) <= E) unsure = true;
    if (g > 0) x = ivid_none();
    return;
  }
  const float inv = __frcp_rn(gd), t = -g * inv;
  const Val tv{t, fmaf(fmaf(fabsf(t), egd, E), fabsf(inv), 5.f * U * fabsf(t))};
  if (gd > 0) clip_hi(x, tv, id | kVerGoalOut, unsure);
  else clip_lo(x, tv, id, unsure);
}

// A component along the ray: body less hole less wedge.
struct Along {
  IvId body, hole, wedge;
};

// A crossing nearly as short as a gap or a chord that vanishes, or of no certain length.
__device__ __forceinline__ void check_len(const IvId& x, bool& unsure) {
  if (x.lo.v > -BIG && x.hi.v < BIG && !apart(x.lo, x.hi)) unsure = true;
}

__device__ inline void along_planar(const Desc& S, const TrackF& T, Along& L, bool& unsure) {
  L.body = ivid_all();
  L.hole = L.wedge = ivid_none();
  if (S.type == kBox) {
    const float ph[3] = {T.xh, T.yh, T.zh}, pl[3] = {T.xl, T.yl, T.zl}, d[3] = {T.u, T.v, T.w};
#pragma unroll
    for (int i = 0; i < 3; i++) {
      const Gv g = abs_minus(ph[i], pl[i], S.Dh[i], S.Dl[i], T.fl);
      if (fabsf(d[i]) <= TAUF && fabsf(g.g) <= HF + g.E) unsure = true;
      if (d[i] == 0) {
        if (fabsf(g.g) <= g.E) unsure = true;
        if (g.g > 0) L.body = ivid_none();
        continue;
      }
      const bool toward = (ph[i] < 0) == (d[i] < 0);
      const float inv = __frcp_rn(fabsf(d[i])), a = g.g * inv, b = (S.Dh[i] + fabsf(ph[i])) * inv;
      const Val A{a, fmaf(g.E, inv, 5.f * U * fabsf(a))}, B{b, 9.f * U * b};
      clip_lo(L.body, toward ? Val{-B.v, B.e} : A, ver_dist(i + 1, 0), unsure);
      clip_hi(L.body, toward ? Val{-A.v, A.e} : B, ver_dist(i + 1, 0) | kVerGoalOut, unsure);
    }
  } else {
    for (int i = 0; i < 4; i++) {
      const Gv g = plane_g(S.plh[i], S.pll[i], S.plh[i][3], S.pll[i][3], T);
      const float a = S.plh[i][0] * T.u, b = S.plh[i][1] * T.v, c = S.plh[i][2] * T.w;
      clip_half(L.body, g.g, g.E, (a + b) + c, 8.f * U * (fabsf(a) + fabsf(b) + fabsf(c)) + 1e-30f, ver_dist(i + 1, 0), unsure);
    }
    const Gv g = abs_minus(T.zh, T.zl, S.dzh, S.dzl, T.fl);
    if (fabsf(T.w) <= TAUF && fabsf(g.g) <= HF + g.E) unsure = true;
    if (T.w == 0) {
      if (fabsf(g.g) <= g.E) unsure = true;
      if (g.g > 0) L.body = ivid_none();
    } else {
      const bool toward = (T.zh < 0) == (T.w < 0);
      const float inv = __frcp_rn(fabsf(T.w)), a = g.g * inv, b = (S.dzh + fabsf(T.zh)) * inv;
      const Val A{a, fmaf(g.E, inv, 5.f * U * fabsf(a))}, B{b, 9.f * U * b};
      clip_lo(L.body, toward ? Val{-B.v, B.e} : A, ver_dist(5, 0), unsure);
      clip_hi(L.body, toward ? Val{-A.v, A.e} : B, ver_dist(5, 0) | kVerGoalOut, unsure);
    }
  }
  check_len(L.body, unsure);
}

template <bool TUBE>
__device__ inline void along_pcon(const Desc& S, const TrackF& T, Along& L, bool& unsure) {
  L.body = ivid_all();
  L.hole = L.wedge = ivid_none();
  const F2 x2 = tprod(T.xh, T.xh), y2 = tprod(T.yh, T.yh);
  const F2 ss = tsum(x2.h, y2.h);
  const float low = ((ss.l + x2.l) + y2.l) + 2.f * (T.xh * T.xl + T.yh * T.yl);
  const float r2h = ss.h + low, r2l = low - (r2h - ss.h), rh = sqrtf(r2h);
  float rl = 0.f;
  if (rh > 0.f) {
    const F2 rr = tprod(rh, rh);
    rl = (((r2h - rr.h) - rr.l) + r2l) * __fdividef(0.5f, rh);
  }
  const F2 rad = radial_df(T), A0 = a0_df(T);
  const float mag = fabsf(T.xh * T.u) + fabsf(T.yh * T.v), erad = G42 * mag + 1e-30f, eRadial = 4.f * U * mag + 1e-30f;
  for (int in = 0; in < 2; in++) {
    if (in && !(S.inner & 1u)) continue;
    const float ah = in ? S.iah[0] : S.oah[0], al = in ? S.ial[0] : S.oal[0], bh = in ? S.ibh[0] : S.obh[0],
                bl = in ? S.ibl[0] : S.obl[0], k = in ? S.ik_[0] : S.ok_[0], a = TUBE ? 0.f : ah;
    const Lat W = lateral<TUBE>(ah, al, bh, bl, k, rh, rl, T, true);
    // along or tangent to the wall near the point: binary64
    const float aw = a * T.w * rh;
    if (fabsf(W.g) <= HF + W.E && fabsf(rad.h - aw) <= eRadial + 4.f * U * fabsf(aw) + 2.f * TAUF * rh * (1.f + fabsf(a)))
      unsure = true;
    const Quad q = quad32<TUBE, false, true>(a, TUBE ? 0.f : al, W, T, rad, erad, A0, rh, rl);
    unsure |= q.unsure;
    const Iv v = iv_region(q, W.g, W.E, unsure);
    const uint32_t id = ver_dist(in ? kInner : kOuter, 0);
    IvId x = v.empty ? ivid_none() : IvId{v.lo, v.hi, in ? id | kVerGoalOut : id, in ? id : id | kVerGoalOut};
    check_len(x, unsure);
    if (in) L.hole = x;
    else L.body = x;
  }
  {
    const float g0 = (S.zh[0] - T.zh) + (S.zl[0] - T.zl), g1 = (T.zh - S.zh[1]) + (T.zl - S.zl[1]);
    const float E0 = 4.f * U * fabsf(g0) + G42 * (fabsf(T.zh) + fabsf(S.zh[0])) + T.fl;
    const float E1 = 4.f * U * fabsf(g1) + G42 * (fabsf(T.zh) + fabsf(S.zh[1])) + T.fl;
    clip_half(L.body, g0, E0, -T.w, 0.f, ver_dist(kZLow, 0), unsure);
    clip_half(L.body, g1, E1, T.w, 0.f, ver_dist(kZLow, 1), unsure);
  }
  if (S.flags & kHasPhi) {
    const bool wide = S.flags & kPhiWide;
    IvId x = ivid_all();
    for (int j = 0; j < 2; j++) {
      const float *nh = j ? S.neh : S.nsh, *nl = j ? S.nel : S.nsl;
      const Gv g = phi_plane(nh, nl, T);
      const float a = nh[0] * T.u, b = nh[1] * T.v, e = 6.f * U * (fabsf(a) + fabsf(b)) + 1e-30f;
      const uint32_t id = ver_dist(j ? kPhiE : kPhiS, 0);
      if (wide) clip_half(x, -g.g, g.E, -(a + b), e, id, unsure);  // the wedge n.p > 0 left out
      else clip_half(L.body, g.g, g.E, a + b, e, id, unsure);
    }
    if (wide) {
      check_len(x, unsure);
      L.wedge = x;
    }
  }
  check_len(L.body, unsure);
}

// Is the point just after t (an end of one of the intervals, or 0) within x?  Unsure when an end that
// is not t itself lies within reach of t.
__device__ __forceinline__ bool within(const IvId& x, Val t, bool& unsure) {
  if (empty(x)) return false;
  if (x.lo.v != t.v && !apart(x.lo, t)) unsure = true;
  if (x.hi.v != t.v && !apart(x.hi, t)) unsure = true;
  return x.lo.v <= t.v && t.v < x.hi.v;
}
__device__ __forceinline__ bool within(const Along& L, Val t, bool& unsure) {
  const bool b = within(L.body, t, unsure), h = within(L.hole, t, unsure), w = within(L.wedge, t, unsure);
  return b && !h && !w;
}
// The nearest end after t: its value and crossing (sign bit kFromC for component c).
constexpr uint32_t kFromC = 1u << 31;
// Two ends at one value: unsure (binary64 may tell them apart).
__device__ __forceinline__ void next_end(const IvId& x, Val t, uint32_t from, Val& n, uint32_t& id, bool& unsure) {
  if (empty(x)) return;
  unsure |= n.v < BIG && (x.lo.v == n.v || x.hi.v == n.v);
  if (x.lo.v > t.v && x.lo.v < n.v) { n = x.lo; id = x.il | from; }
  if (x.hi.v > t.v && x.hi.v < n.v) { n = x.hi; id = x.ih | from; }
}

// Code and safety of a component (RANK, no distances).
__device__ inline void rank_safety(const Desc& S, const TrackF& T, R32& R) {
  R.flag = T.bad;
  R.code = 1;
  R.din = R.dout = R.sin = R.sout = 0.f;
  R.rank = 0u;
  R.te = R.se = 0.f;
  if (R.flag) return;
  const unsigned want = kWantCode | kWantSin | kWantSout;
  if (S.type == kBox) box32<false, true>(S, T, want, R);
  else if (S.type == kTrd || S.type == kTrap) planar32<false, true>(S, T, want, R);
  else if (S.type == kTube) pcon32<true, false, true>(S, T, want, R);
  else pcon32<false, false, true>(S, T, want, R);
}
__device__ inline void along(const Desc& S, const TrackF& T, Along& L, bool& unsure) {
  if (S.type == kBox || S.type == kTrd || S.type == kTrap) along_planar(S, T, L, unsure);
  else if (S.type == kTube) along_pcon<true>(S, T, L, unsure);
  else along_pcon<false>(S, T, L, unsure);
}

}  // namespace f32

namespace f64 {

// Do the ranked results cover this boolean?  (Host and device.)
__host__ __device__ inline bool bool_ranks(const Desc& a, const Desc& c) {
  const bool pa = a.type == kBox || a.type == kTrd || a.type == kTrap || a.nz == 2;
  const bool pc = c.type == kBox || c.type == kTrd || c.type == kTrap || c.nz == 2;
  return pa && pc && !((a.flags | c.flags) & kFp64Only);
}

// A component's results by a verdict on its safety or one of its crossings.
__device__ __forceinline__ void prim_ranked(const Desc& S, const Track& T, uint32_t rank, Result& R) {
  const Verdict V{rank};
  if (S.type == kBox) box_ranked(S, T, V, R);
  else if (S.type == kTrd || S.type == kTrap) planar_ranked(S, T, V, R);
  else pcon_ranked(S, T, V, R);
}

// A track in the second component's frame; unrotated: the same values (products with 0 and 1 are
// exact for finite tracks), 30 FP64 operations less.
__device__ __forceinline__ void bool_frame_finite(const Desc& S, const Track& T, Track& Tc) {
  if (S.unrotated) Tc = Track{xsub(T.x, S.bt[0]), xsub(T.y, S.bt[1]), xsub(T.z, S.bt[2]), T.u, T.v, T.w};
  else bool_frame(S, T, Tc);
}

// The verdict of a boolean: bit 0 the point is inside, 1 the safety takes a's, 2 c's, 3 the larger of two,
// 4-6 and 7-9 the constraints of a's and c's safeties, 10 and 11 the point is inside a, c, 12-14 the
// crossing that gives the distance (0: none), 15-16 its z-plane, 17 the component is left there, 18 it is
// c's.
struct BoolVerdict {
  uint32_t w;
  __device__ __forceinline__ bool in() const { return w & 1u; }
  __device__ __forceinline__ bool bit(int b) const { return (w >> b) & 1u; }
  __device__ __forceinline__ uint32_t dkind() const { return (w >> 12) & 7u; }
  __device__ __forceinline__ bool needs_c() const { return bit(2) || (dkind() != 0u && bit(18)); }
};

// The verdict on a track; false when the ranking is not certain.  Called, not inlined: its registers would
// spill the evaluation's.
static __device__ __noinline__ bool bool_verdict(const Desc& S, const Desc& A, const Desc& C, const Track& T, unsigned want, uint32_t& out) {
  const bool dirs = want & (kWantDin | kWantDout);
  const f32::TrackF Fa = split_track(T, dirs);
  if (Fa.bad) return false;
  Track Tc;
  bool_frame_finite(S, T, Tc);
  const f32::TrackF Fc = split_track(Tc, dirs);
  f32::R32 ra, rc;
  f32::rank_safety(A, Fa, ra);
  f32::rank_safety(C, Fc, rc);
  if (ra.flag || rc.flag || ra.code == 1 || rc.code == 1) return false;
  const int op = S.bop;
  const bool ia = ra.code == 0, ic = rc.code == 0;
  const bool in = op == kUnion ? ia || ic : op == kIntersection ? ia && ic : ia && !ic;
  uint32_t V = (in ? 1u : 0u) | Verdict{ra.rank}.skind() << 4 | Verdict{rc.rank}.skind() << 7 | (ia ? 1u << 10 : 0u) |
               (ic ? 1u << 11 : 0u);
  if (dirs) {
    f32::Along La, Lc;
    bool unsure = false;
    f32::along(A, Fa, La, unsure);
    f32::along(C, Fc, Lc, unsure);
    f32::Val t{0.f, 0.f};
    bool answered = false;
    uint32_t end = 0u;
    // the start agrees with the codes
    if (f32::within(La, t, unsure) != ia || f32::within(Lc, t, unsure) != ic) unsure = true;
    for (int guard = 0; guard < 12 && !unsure; guard++) {
      f32::Val n{f32::BIG, 0.f};
      f32::next_end(La.body, t, 0u, n, end, unsure);
      f32::next_end(La.hole, t, 0u, n, end, unsure);
      f32::next_end(La.wedge, t, 0u, n, end, unsure);
      f32::next_end(Lc.body, t, f32::kFromC, n, end, unsure);
      f32::next_end(Lc.hole, t, f32::kFromC, n, end, unsure);
      f32::next_end(Lc.wedge, t, f32::kFromC, n, end, unsure);
      if (unsure || n.v >= f32::BIG) break;
      t = n;
      const bool a = f32::within(La, t, unsure), c = f32::within(Lc, t, unsure);
      if ((op == kUnion ? a || c : op == kIntersection ? a && c : a && !c) != in) {
        answered = true;
        break;
      }
    }
    if (unsure || (in && !answered)) return false;
    if (answered) {
      const Verdict E{end};
      V |= E.dkind() << 12 | (uint32_t)E.dpiece() << 15 | (E.out() ? 1u << 17 : 0u) | ((end & f32::kFromC) ? 1u << 18 : 0u);
    }
  }
  if (want & (kWantSin | kWantSout)) {
    // a union is left (entered) through the component whose own safety is larger (smaller), an
    // intersection the other way round, a subtraction as a and not-c
    const float va = ia ? ra.sout : ra.sin, vc = ic ? rc.sout : rc.sin;
    const float ea = fmaf(2.f * f32::U, fabsf(va), ra.se), ec = fmaf(2.f * f32::U, fabsf(vc), rc.se);
    const bool largest = op == kUnion ? in : !in;
    bool use_a, use_c;
    if (op == kUnion) {
      use_a = in ? ia : true;
      use_c = in ? ic : true;
    } else {
      use_a = in ? true : !ia;
      use_c = in ? true : op == kIntersection ? !ic : ic;
    }
    if (use_a && use_c) {  // one of them certainly, else both in binary64
      const float lo_a = va - ea, hi_a = va + ea, lo_c = vc - ec, hi_c = vc + ec;
      if (largest ? lo_a > hi_c : hi_a < lo_c) use_c = false;
      else if (largest ? lo_c > hi_a : hi_c < lo_a) use_a = false;
    }
    V |= (use_a ? 2u : 0u) | (use_c ? 4u : 0u) | (largest ? 8u : 0u);
  }
  out = V;
  return true;
}

// The results of bool_query, bit for bit, by a verdict.
__device__ inline void bool_evaluate(const Desc& S, const Desc& A, const Desc& C, const Track& T, BoolVerdict V, Result& R) {
  const bool in = V.in(), ia = V.bit(10), ic = V.bit(11);
  R.code = in ? 0 : 2;
  R.sin = R.sout = R.din = R.dout = -1.0;
  Track Tc;
  if (V.needs_c()) bool_frame_finite(S, T, Tc);
  Result P;
  if (V.bit(1) || V.bit(2)) {
    double v = 0;
    if (V.bit(1)) {
      prim_ranked(A, T, (ia ? 0u : 2u) | f32::ver_safety((V.w >> 4) & 7u, 0), P);
      v = ia ? P.sout : P.sin;
    }
    if (V.bit(2)) {
      prim_ranked(C, Tc, (ic ? 0u : 2u) | f32::ver_safety((V.w >> 7) & 7u, 0), P);
      const double x = ic ? P.sout : P.sin;
      v = V.bit(1) ? (V.bit(3) ? dmax(v, x) : dmin(v, x)) : x;
    }
    if (in) R.sout = v;
    else R.sin = v;
  }
  double t = in ? 0.0 : GV_INF;
  if (V.dkind() != 0u) {
    const uint32_t id = f32::ver_dist(V.dkind(), (int)((V.w >> 15) & 3u)) | (V.bit(17) ? f32::kVerGoalOut : 0u);
    if (V.bit(18)) prim_ranked(C, Tc, id, P);
    else prim_ranked(A, T, id, P);
    t = V.bit(17) ? P.dout : P.din;
  }
  if (in) R.dout = t;
  else R.din = t;
}

// Groups tracks whose binary64 work is alike: the distance (none, a plane's crossing, a wall's), whether
// the second component's frame is needed, whether a safety needs a square root.
constexpr uint32_t kBoolClasses = 12;
__device__ __forceinline__ uint32_t bool_class(const Desc& A, const Desc& C, BoolVerdict V) {
  auto wall = [](const Desc& P, uint32_t kind) {
    return P.nz == 2 && (kind == f32::kOuter || kind == f32::kInner || kind == f32::kWhole);
  };
  const uint32_t d = V.dkind() == 0u ? 0u : wall(V.bit(18) ? C : A, V.dkind()) ? 2u : 1u;
  const bool root = (V.bit(1) && wall(A, (V.w >> 4) & 7u)) || (V.bit(2) && wall(C, (V.w >> 7) & 7u));
  return 4u * d + (V.needs_c() ? 2u : 0u) + (root ? 1u : 0u);
}

}  // namespace f64
}  // namespace gv
