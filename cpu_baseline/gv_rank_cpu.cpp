// gv_rank_cpu.cpp -- the library's ranked binary64 evaluation (rank_fp64.cuh) compiled for the
// host, for tests that compare it with the whole binary64 evaluation (gv_cpu.cpp) without a GPU, and
// the navigation step's plain look at a placed daughter (nav_cull.cuh) likewise.
#include <cuda_runtime.h>  // the host stand-ins (shim/)
#include "bool_rank.cuh"
#include "nav_cull.cuh"
#include "rank_fp64.cuh"

using namespace gv;

template <int FAMILY>
static bool one(const Desc& S, const uint2* const p[6], int64_t i, bool dirs, const f64::Track& T, unsigned want,
                bool given, f64::Result& R) {
  const f32::TrackF F = f32::load_track<(FAMILY >= 2)>(p[0], p[1], p[2], p[3], p[4], p[5], i, dirs);
  if (given) return f64::query_given<FAMILY>(S, T, F, want, R);
  f32::R32 r;
  f64::rank32<FAMILY>(S, F, want, r);
  if (r.flag) return false;
  f64::query_ranked<FAMILY>(S, T, f64::Verdict{r.rank}, R);
  return true;
}

// The requested results of n tracks against a descriptor of gvcpu_build; ranked[i] tells whether
// track i had a certain verdict (its results are left alone if not).  given: the code from binary64.
extern "C" void gvcpu_query_ranked(const void* desc, int64_t n, const double* const* t, unsigned want, int given, int8_t* ranked,
                                   int8_t* inside, double* din, double* dout, double* sin, double* sout) {
  Desc S;
  std::memcpy(&S, desc, sizeof(Desc));
  const uint2* p[6];
  for (int c = 0; c < 6; c++) p[c] = reinterpret_cast<const uint2*>(t[c]);
  const bool dirs = want & (f64::kWantDin | f64::kWantDout);
#pragma omp parallel for schedule(static, 4096)
  for (int64_t i = 0; i < n; i++) {
    f64::Track T{t[0][i], t[1][i], t[2][i], 0, 0, 0};
    if (dirs) { T.u = t[3][i]; T.v = t[4][i]; T.w = t[5][i]; }
    f64::Result R;
    bool ok = false;
    if (!(S.flags & kFp64Only)) switch (S.type) {
      case kBox: ok = one<0>(S, p, i, dirs, T, want, given, R); break;
      case kTrd:
      case kTrap: ok = one<1>(S, p, i, dirs, T, want, given, R); break;
      case kTube: ok = one<2>(S, p, i, dirs, T, want, given, R); break;
      default: ok = one<3>(S, p, i, dirs, T, want, given, R); break;
    }
    ranked[i] = ok;
    if (!ok) continue;
    inside[i] = (int8_t)R.code;
    din[i] = R.din;
    dout[i] = R.dout;
    sin[i] = R.sin;
    sout[i] = R.sout;
  }
}

// The plain look at a box (tag 0), a full tube (1) or another solid (2) with half extents e and inner
// radius rmin, placed by R (row-major) and t, for n world tracks: out[7 i ..] = miss, from, by, miss of the
// look without bounds, certainly outside, safety, margin.
extern "C" void gvcpu_plain_look(int tag, const double* e, double rmin, const double* R, const double* t, int64_t n,
                                 const double* const* c, float* out) {
  Cull C;
  std::memset(&C, 0, sizeof(C));
  double mag = 0;
  for (int i = 0; i < 9; i++) C.R[i] = (float)R[i];
  for (int i = 0; i < 3; i++) {
    C.t[i] = (float)t[i];
    C.e[i] = (float)e[i];
    mag += std::fabs(t[i]) + e[i];
  }
  C.rmin = (float)rmin;
  C.margin = (float)(1e-6 + 4e-6 * mag);
  C.tag = tag;
  for (int64_t i = 0; i < n; i++) {
    const PlainTrack P{(float)c[0][i], (float)c[1][i], (float)c[2][i], (float)c[3][i], (float)c[4][i], (float)c[5][i],
                       4e-6f * (float)(std::fabs(c[0][i]) + std::fabs(c[1][i]) + std::fabs(c[2][i]))};
    const PlainLocal L = plain_local(C, P);
    float* o = out + 7 * i;
    float from;
    bool near;
    o[0] = plain_entry(C, P, L, o[1], o[2]) ? 1.f : 0.f;
    o[3] = plain_miss(C, P, L, from, near) ? 1.f : 0.f;
    o[4] = plain_outside(C, L) ? 1.f : 0.f;
    o[5] = tag <= kCullTube ? plain_safety(C, L) : 0.f;
    o[6] = L.margin;
  }
}

// A boolean op(a, c) of two descriptors, c placed by R (row-major) and t: the whole evaluation
// (whole[]: inside, din, dout, sin, sout as doubles, 5 per track) and the ranked one (0 in ranked[i] when not
// certain, or when the components have no ranked form).
extern "C" void gvcpu_bool(int op, const void* a, const void* c, const double* R, const double* t, int64_t n,
                           const double* const* tr, unsigned want, double* whole, double* got, int8_t* ranked) {
  Desc parts[2], S;
  std::memcpy(&parts[0], a, sizeof(Desc));
  std::memcpy(&parts[1], c, sizeof(Desc));
  std::memset(&S, 0, sizeof(S));
  S.type = kBool;
  S.bop = op;
  S.unrotated = 1;
  for (int i = 0; i < 9; i++) {
    S.bR[i] = R[i];
    if (R[i] != (i % 4 == 0 ? 1.0 : 0.0)) S.unrotated = 0;
  }
  for (int i = 0; i < 3; i++) S.bt[i] = t[i];
  S.parts = parts;
  const bool dirs = want & (f64::kWantDin | f64::kWantDout), forms = f64::bool_ranks(parts[0], parts[1]);
#pragma omp parallel for schedule(static, 1024)
  for (int64_t i = 0; i < n; i++) {
    f64::Track T{tr[0][i], tr[1][i], tr[2][i], 0, 0, 0};
    if (dirs) { T.u = tr[3][i]; T.v = tr[4][i]; T.w = tr[5][i]; }
    f64::Result r{0, 0, 0, 0, 0}, q{0, 0, 0, 0, 0};
    f64::bool_query(S, T, want, r);
    uint32_t V;
    ranked[i] = forms && f64::bool_verdict(S, parts[0], parts[1], T, want, V);
    if (ranked[i]) f64::bool_evaluate(S, parts[0], parts[1], T, f64::BoolVerdict{V}, q);
    const double w[5] = {(double)r.code, r.din, r.dout, r.sin, r.sout}, o[5] = {(double)q.code, q.din, q.dout, q.sin, q.sout};
    for (int k = 0; k < 5; k++) { whole[5 * i + k] = w[k]; got[5 * i + k] = o[k]; }
  }
}
