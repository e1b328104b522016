// rank_fp64.cuh -- binary64 results from a binary32 ranking.
//
// The whole binary64 evaluation of a track (solid_fp64.cuh) forms every constraint value and every
// crossing of every surface, then keeps one of them per result.  The certified binary32 passes,
// instanced with RANK (solid_fp32.cuh), decide which one that is; only that constraint value and
// that crossing are then evaluated in binary64, by the same expressions as the whole evaluation, so
// the results have the same bits.  On GB300 the FP64 pipe issues one warp instruction in 16 clocks
// per SM and is what bounds the whole evaluation (226 FP64 warp instructions per 32 tracks of a
// cone, 859 of an 8-plane polycone); one crossing and one constraint value need about 60.  A track
// whose ranking is not certain (R32::flag) is evaluated whole.
#pragma once
#include "solid_fp32.cuh"
#include "solid_fp64.cuh"

namespace gv {
namespace f64 {

struct Verdict {
  uint32_t w;
  __device__ __forceinline__ int code() const { return (int)(w & 3u); }
  __device__ __forceinline__ uint32_t skind() const { return (w >> 3) & 7u; }
  __device__ __forceinline__ int spiece() const { return (int)((w >> 6) & 31u); }
  __device__ __forceinline__ uint32_t dkind() const { return (w >> 11) & 7u; }
  __device__ __forceinline__ int dpiece() const { return (int)((w >> 14) & 31u); }
  __device__ __forceinline__ bool out() const { return (w & f32::kVerGoalOut) != 0u; }
};

// All results from the safety's constraint value s and the distance t: the other distance and
// the safety of the wrong side are constants of the code.
__device__ __forceinline__ void rank_results(Verdict V, double s, double t, Result& R) {
  R.code = V.code();
  finish_safety(R.code, s, -s, R);
  const double other = R.code == 1 ? 0.0 : -1.0;
  R.dout = V.out() ? t : other;
  R.din = V.out() ? other : t;
}

__device__ __forceinline__ double rank_none(Verdict V) { return V.out() ? 0.0 : GV_INF; }

__device__ inline void box_ranked(const Desc& S, const Track& T, Verdict V, Result& R) {
  double s = 0, t = rank_none(V);
  const uint32_t sk = V.skind(), dk = V.dkind();
  if (sk == f32::kWhole) {
    s = box_s(S, T.x, T.y, T.z);
  } else if (sk != f32::kNone) {
    s = xsub(fabs(sk == 1 ? T.x : sk == 2 ? T.y : T.z), S.D[sk - 1]);
  }
  if (dk != f32::kNone) {
    const double p = dk == 1 ? T.x : dk == 2 ? T.y : T.z, d = dk == 1 ? T.u : dk == 2 ? T.v : T.w;
    const double face = copysign(S.D[dk - 1], d);
    t = ((V.out() ? face : -face) - p) / d;
  }
  rank_results(V, s, t, R);
}

__device__ inline void planar_ranked(const Desc& S, const Track& T, Verdict V, Result& R) {
  double s = 0, t = rank_none(V);
  const uint32_t sk = V.skind(), dk = V.dkind();
  auto side = [&](uint32_t i) {
    const double* P = S.pl[i - 1];
    return xsub(xadd(xadd(xmul(P[0], T.x), xmul(P[1], T.y)), xmul(P[2], T.z)), P[3]);
  };
  if (sk == f32::kWhole) s = planar_s(S, T.x, T.y, T.z);
  else if (sk == 5) s = xsub(fabs(T.z), S.dz);
  else if (sk != f32::kNone) s = side(sk);
  if (dk != f32::kNone) {
    double num, den;
    if (dk == 5) {
      const double face = copysign(S.dz, T.w);
      num = (V.out() ? face : -face) - T.z;
      den = T.w;
    } else {
      const double* P = S.pl[dk - 1];
      num = -side(dk);
      den = xadd(xadd(xmul(P[0], T.u), xmul(P[1], T.v)), xmul(P[2], T.w));
    }
    t = num / den;
  }
  rank_results(V, s, t, R);
}

// The crossing of r = a z + b by which the track leaves (plus) or enters {r <= R}, as line_cross
// forms it; the ranking has established that it exists (not a touch, on the nappe a z + b >= 0).
// num / den: the caller divides.
__device__ __forceinline__ void line_root(const Line& L, const Track& T, double r2, bool plus, double& num,
                                          double& den) {
  const double radial = xadd(xmul(T.x, T.u), xmul(T.y, T.v));
  const double A0 = xadd(xmul(T.u, T.u), xmul(T.v, T.v));
  const double P = xadd(xmul(L.a, T.z), L.b), D = xmul(L.a, T.w);
  const double A = xsub(A0, xmul(D, D)), B = xsub(radial, xmul(P, D)), C = xsub(r2, xmul(P, P));
  if (A == 0) {
    num = -C;
    den = 2 * B;
    return;
  }
  const double sq = sqrt(xsub(xmul(B, B), xmul(A, C)));
  const bool pos = B >= 0;
  const double q = pos ? -(B + sq) : sq - B;
  const bool by_a = pos != plus;  // tm = q / A, tp = C / q for B >= 0, the other way round below
  num = by_a ? q : C;
  den = by_a ? A : q;
}

__device__ inline void pcon_ranked(const Desc& S, const Track& T, Verdict V, Result& R) {
  double s = 0, t = rank_none(V);
  const uint32_t sk = V.skind(), dk = V.dkind();
  const bool dwall = dk == f32::kOuter || dk == f32::kInner;
  const bool swall = sk == f32::kOuter || sk == f32::kInner || sk == f32::kWhole;
  double r2 = 0;
  if (dwall || swall) r2 = xadd(xmul(T.x, T.x), xmul(T.y, T.y));
  if (sk != f32::kNone) {
    const int k = V.spiece();
    if (swall) {
      const double r = __dsqrt_rn(r2);
      if (sk == f32::kOuter) s = g_out(S.out[k], r, T.z);
      else if (sk == f32::kInner) s = g_in(S.in[k], r, T.z);
      else {
        const double gphi = (S.flags & kHasPhi) ? phi_g(S, phi_eval(S, T.x, T.y)) : -GV_INF;
        if (k != f32::kAllPieces) {
          s = s_closed(S, k, r, T.z, gphi);
        } else {
          s = s_closed(S, 0, r, T.z, gphi);
          for (int j = 1; j + 1 < S.nz; j++) s = dmin(s, s_closed(S, j, r, T.z, gphi));
        }
      }
    } else if (sk == f32::kZLow) {
      s = xsub(S.z[k], T.z);
    } else if (sk == f32::kZHigh) {
      s = xsub(T.z, S.z[k + 1]);
    } else {
      const double* n = sk == f32::kPhiS ? S.ns : S.ne;
      s = xadd(xmul(n[0], T.x), xmul(n[1], T.y));
    }
  }
  if (dk != f32::kNone) {
    const int k = V.dpiece();
    double num, den;
    if (dwall) {
      line_root(dk == f32::kOuter ? S.out[k] : S.in[k], T, r2, V.out() == (dk == f32::kOuter), num, den);
    } else if (dk == f32::kZLow) {
      num = S.z[k] - T.z;
      den = T.w;
    } else {
      const double* n = dk == f32::kPhiS ? S.ns : S.ne;
      num = -xadd(xmul(n[0], T.x), xmul(n[1], T.y));
      den = xadd(xmul(n[0], T.u), xmul(n[1], T.v));
    }
    t = num / den;
  }
  rank_results(V, s, t, R);
}

// A binary64 track split for the binary32 passes.
__device__ __forceinline__ f32::TrackF split_track(const Track& T, bool dirs) {
  auto w = [](double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return make_uint2((unsigned)b, (unsigned)(b >> 32));
  };
  return f32::track_from_words<true>(w(T.x), w(T.y), w(T.z), w(T.u), w(T.v), w(T.w), dirs);
}

// Families: 0 box, 1 trd/trap, 2 tube, 3 polycone, 4 cone (two z-planes).
template <int FAMILY, bool GIVEN = false>
__device__ __forceinline__ void rank32(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  R.flag = T.bad;
  if (!GIVEN) R.code = 1;
  R.din = R.dout = R.sin = R.sout = 0.f;
  R.rank = 0u;
  R.te = R.se = 0.f;
  if (R.flag) return;
  if (FAMILY == 0) f32::box32<false, true, GIVEN>(S, T, want, R);
  else if (FAMILY == 1) f32::planar32<false, true, GIVEN>(S, T, want, R);
  else if (FAMILY == 2) f32::pcon32<true, false, true, GIVEN>(S, T, want, R);
  else f32::pcon32<false, false, true, GIVEN>(S, T, want, R);
}

template <int FAMILY>
__device__ __forceinline__ void query_ranked(const Desc& S, const Track& T, Verdict V, Result& R) {
  if (FAMILY == 0) box_ranked(S, T, V, R);
  else if (FAMILY == 1) planar_ranked(S, T, V, R);
  else pcon_ranked(S, T, V, R);
}

// The whole evaluation of a track, and one that ranks first: the code from its binary64 decision
// quantity, the rest ranked with that code given.  It leaves the whole evaluation only the tracks whose
// crossings binary32 cannot order (with the code in binary64 about one in 10^5), and takes a shorter
// chain of binary64 operations than the whole one (a polycone: about 100 against 1500).
template <int FAMILY>
__device__ __forceinline__ void query_whole(const Desc& S, const Track& T, unsigned want, Result& R) {
  if (FAMILY == 0) box_query(S, T, want, R);
  else if (FAMILY == 1) planar_query(S, T, want, R);
  else pcon_query(S, T, want, R);
}
template <int FAMILY>
__device__ __forceinline__ bool query_given(const Desc& S, const Track& T, const f32::TrackF& F, unsigned want, Result& R) {
  const double s = FAMILY == 0 ? box_s(S, T.x, T.y, T.z) : FAMILY == 1 ? planar_s(S, T.x, T.y, T.z) : pcon_s(S, T.x, T.y, T.z);
  f32::R32 r;
  r.code = code_of(s);
  rank32<FAMILY, true>(S, F, want, r);
  if (r.flag) return false;
  query_ranked<FAMILY>(S, T, Verdict{r.rank}, R);
  return true;
}

// All of a track's results in binary64: ranked for multi-section polycones, whose whole evaluation is
// a chain of some 1500 operations (batched refinement of 1176 tracks 51 -> 28 us), and for boxes
// (10.7 -> 7.4 us); the whole evaluation of the others is as short as their ranking.
template <int FAMILY>
__device__ __noinline__ void whole_call(const Desc& S, const Track& T, unsigned want, Result& R) {
  query_whole<FAMILY>(S, T, want, R);
}
template <int FAMILY>
__device__ __forceinline__ void query_refined(const Desc& S, const Track& T, const f32::TrackF& F, unsigned want, Result& R) {
  if ((FAMILY == 0 || FAMILY == 3) && (want & (kWantDin | kWantDout))) {
    if (!query_given<FAMILY>(S, T, F, want, R)) whole_call<FAMILY>(S, T, want, R);
  } else {
    query_whole<FAMILY>(S, T, want, R);
  }
}

// Groups tracks whose binary64 work is alike: bit 0 a square root for the safety, then no
// division, a division, or a square root and a division for the distance.
constexpr uint32_t kRankClasses = 6;
template <int FAMILY>
__device__ __forceinline__ uint32_t rank_class(Verdict V) {
  const uint32_t sk = V.skind(), dk = V.dkind();
  if (FAMILY < 2) return dk != f32::kNone ? 2u : 0u;
  const uint32_t c = (sk == f32::kOuter || sk == f32::kInner || sk == f32::kWhole) ? 1u : 0u;
  return c + (dk == f32::kNone ? 0u : (dk == f32::kOuter || dk == f32::kInner) ? 4u : 2u);
}

}  // namespace f64
}  // namespace gv
