// nav.cu -- the navigation step over a tree of placed volumes.
//
// The detector is an ordered hierarchy of placed solids (Detector geometry
// subsection); in a step the particle moves by the smaller of the physics length
// and the distance to the next boundary (Physics subsection).  The geometry half
// of the step, per track located in node v:
//   step   = min( DistanceToOut of v's solid, DistanceToIn of every daughter c of v
//                 in c's frame p_c = R_c^T (p - t_c), d_c = R_c^T d ),
//   safety = min( SafetyToOut of v, SafetyToIn of every daughter ),
//   next   = the daughter that gives the step, or -1 (the track leaves v);
// -1 values (a point on the wrong side) are left out; among equal distances the
// lowest daughter index wins and a daughter wins over the mother.
// Locate descends from the world into the first daughter (in index order) that
// does not classify the point as outside.
//
// Kernels: binary64, a block-wide pool of tracks in phases (k_nav_pool), the candidates ranked in
// certified binary32 and only the deciding one evaluated in binary64 (the same bits); binary32, one thread
// per track over scanned daughters (k_nav_scan32) or kLanes lanes per track along a grid or in short baskets
// (k_nav_fp32), whose tracks with an ambiguous minimum or an uncertain daughter are recomputed by the
// binary64 step (k_nav_pool, short baskets k_nav_exact) from
// a worklist.  World-to-node
// transforms are composed on the host (binary64, no fused multiply-add) and
// applied on the device with round-to-nearest operations in a fixed order, so the
// binary64 results and codes agree with any evaluation that uses the same order.
#include <algorithm>
#include <cstring>
#include <new>
#include <vector>
#include <array>
#include "gv_internal.h"
#include "nav_cull.cuh"
#include "rank_fp64.cuh"
#include "solid_fp32.cuh"
#include "solid_fp64.cuh"

namespace gv {

struct alignas(16) NodeD {
  double R[9];      // global rotation (row-major), p_world = R p_local + t
  double t[3];
  float Rh[9], Rl[9], th[3], tl[3];  // binary32 splits of R and t
  int32_t desc;     // index into the solid table
  int32_t parent;
  int32_t first;    // daughters: children[first .. first + count)
  int32_t count;
  int32_t grid;     // voxel grid over the daughters (-1: none)
  int32_t never;    // some daughter has no binary32 form
};

// A uniform grid over the daughters of a node, in the node's frame: cell (i, j, k) lists
// (in increasing node index) the daughters whose bounding box, padded, meets the cell.
struct GridD {
  double lo[3], cell[3], inv[3];  // origin, cell edges, their inverses
  int32_t n[3];                   // cells per axis
  int32_t start;                  // first cell's entry in the geometry's cell table
  int32_t safe;                   // first cell's safety list (-1: none)
  float flo[3], fcell[3], finv[3];
};

// An entry of a cell's safety list: a daughter and a lower bound of its SafetyToIn at the cell's
// centre.  A list holds the kSafeList daughters of least bound, in increasing order.
struct SafeEnt {
  float s;
  int32_t node;
};
constexpr int kSafeList = 64;
// Lists are built for grids of at most these many daughters and cells (one evaluation per pair when the
// geometry is created: 3 M for 1728 daughters).
constexpr int kSafeDaughters = 8192, kSafeCells = 32768;
// All lists of a geometry together: 135 MB.  Volumes beyond have none: their safeties scan the daughters.
constexpr int64_t kSafeTotal = 1 << 18;

// Device pointers of a geometry's grids (grids == nullptr: no grid is used).
struct Vox {
  const GridD* grids;
  const int32_t* cells;  // per cell: [begin, end) into list
  const int32_t* list;
  const SafeEnt* safe;   // kSafeList entries per cell (node -1: fewer daughters)
  const float* safe_cut;  // per cell: a lower bound for the daughters not listed
};

// Nodes with at least this many daughters get a grid.
constexpr int kVoxelMin = 16;
// The steps walk a node's grid, and its cells carry safety lists, only from this many daughters on: a
// binary64 DDA costs more than a plain look at a few dozen daughters (nested detector, 32 daughters
// per shell: transport 24.2 ms walking their grids, then 14.9 ms scanning them).
constexpr int kWalk32Min = 128;

constexpr float kInf32 = __builtin_huge_valf();
constexpr int kLanes = 8;  // lanes per track in the binary32 kernel

}  // namespace gv

struct gv_geom {
  int device;
  int nnodes, nsolids;
  gv::NodeD* d_nodes = nullptr;
  int32_t* d_children = nullptr;
  gv::Desc* d_solids = nullptr;
  gv::Cull* d_cull = nullptr;  // per node
  gv::GridD* d_grids = nullptr;
  int32_t* d_cells = nullptr;
  int32_t* d_list = nullptr;
  gv::SafeEnt* d_safe = nullptr;
  float* d_safe_cut = nullptr;
  bool use_vox = true;
  bool walk32 = false;  // some node with a grid has at least kWalk32Min daughters
  bool never = false;   // some node has a daughter without a binary32 form
  std::vector<gv::NodeD> nodes;
  std::vector<gv::Cull> cull;
  std::vector<int32_t> children;
  std::vector<gv::Desc> solids;
  std::vector<gv::GridD> grids;
  std::vector<int32_t> cells, list;
};

namespace gv {

using f64::xadd;
using f64::xmul;
using f64::xsub;

// binary64 world -> node frame
__device__ __forceinline__ void to_local64(const NodeD& N, double x, double y, double z, double& lx, double& ly,
                                           double& lz) {
  const double v0 = xsub(x, N.t[0]), v1 = xsub(y, N.t[1]), v2 = xsub(z, N.t[2]);
  lx = xadd(xadd(xmul(N.R[0], v0), xmul(N.R[3], v1)), xmul(N.R[6], v2));
  ly = xadd(xadd(xmul(N.R[1], v0), xmul(N.R[4], v1)), xmul(N.R[7], v2));
  lz = xadd(xadd(xmul(N.R[2], v0), xmul(N.R[5], v1)), xmul(N.R[8], v2));
}
__device__ __forceinline__ void rot_local64(const NodeD& N, double u, double v, double w, double& lu, double& lv,
                                            double& lw) {
  lu = xadd(xadd(xmul(N.R[0], u), xmul(N.R[3], v)), xmul(N.R[6], w));
  lv = xadd(xadd(xmul(N.R[1], u), xmul(N.R[4], v)), xmul(N.R[7], w));
  lw = xadd(xadd(xmul(N.R[2], u), xmul(N.R[5], v)), xmul(N.R[8], w));
}

__device__ __forceinline__ void query64(const Desc& S, const f64::Track& T, unsigned want, f64::Result& R) {
  if (S.type == kBox) f64::box_query(S, T, want, R);
  else if (S.type == kTrd || S.type == kTrap) f64::planar_query(S, T, want, R);
  else if (S.type == kBool) f64::bool_query(S, T, want, R);
  else f64::pcon_query(S, T, want, R);
}

// The cell of a point given in the grid's node frame; false outside the grid (where no
// daughter is).
__device__ __forceinline__ bool grid_cell(const GridD& G, const double q[3], int c[3]) {
  for (int a = 0; a < 3; a++) {
    const double f = (q[a] - G.lo[a]) * G.inv[a];
    if (!(f >= 0.0 && f <= (double)G.n[a])) return false;
    c[a] = min((int)f, G.n[a] - 1);
  }
  return true;
}

// The daughters of node N to look at for a point (x, y, z) in world coordinates: all of
// them, or those listed in the point's cell when N has a grid.
__device__ __forceinline__ void candidates64(const NodeD& N, const int32_t* __restrict__ children, const Vox& vox,
                                             double x, double y, double z, const int32_t*& ids, int& count) {
  ids = children + N.first;
  count = N.count;
  if (!vox.grids || N.grid < 0) return;
  const GridD& G = vox.grids[N.grid];
  double q[3];
  to_local64(N, x, y, z, q[0], q[1], q[2]);
  int c[3];
  if (!grid_cell(G, q, c)) { count = 0; return; }
  const int cell = G.start + (c[2] * G.n[1] + c[1]) * G.n[0] + c[0];
  ids = vox.list + vox.cells[2 * cell];
  count = vox.cells[2 * cell + 1] - vox.cells[2 * cell];
}

// The same for a point in plain binary32 in N's frame (Cull of N), when it is certain which cell the
// point is in (false: not certain).
__device__ __forceinline__ bool candidates32(const NodeD& N, const Cull& C, const int32_t* __restrict__ children,
                                             const Vox& vox, const PlainTrack& P, const int32_t*& ids, int& count) {
  ids = children + N.first;
  count = N.count;
  if (!vox.grids || N.grid < 0) return true;
  const GridD& G = vox.grids[N.grid];
  const PlainLocal L = plain_local(C, P);
  int c[3];
  bool sure = true, out = false;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const float f = (L.q[a] - G.flo[a]) * G.finv[a], tol = 2.f * L.margin * G.finv[a] + 1e-6f * fabsf(f);
    const float k = floorf(f);
    sure &= f - k > tol && k + 1.f - f > tol && isfinite(f);
    out |= f < -tol || f > (float)G.n[a] + tol;
    c[a] = min(max((int)k, 0), G.n[a] - 1);
  }
  if (out) { count = 0; return true; }
  const int cell = G.start + (c[2] * G.n[1] + c[1]) * G.n[0] + c[0];
  ids = vox.list + vox.cells[2 * cell];
  count = vox.cells[2 * cell + 1] - vox.cells[2 * cell];
  return sure;
}

struct NavArgs {
  const double *x, *y, *z, *u, *v, *w;
  const int32_t* node;
  double *step, *safety;
  int32_t* next;
  int64_t n;
};

// A 3-D DDA over the cells of a grid that a ray (node frame) crosses, in order of entry.
struct Dda {
  int c[3], step[3];
  double tnext[3], tdelta[3];
  double tenter, t1;  // entry of the current cell, exit from the grid
  int left;           // cells that may still be visited (a ray crosses at most n0 + n1 + n2 - 2)
  // false: the ray misses the grid
  __device__ __forceinline__ bool begin(const GridD& G, const double q[3], const double e[3]) {
    double t0 = 0.0;
    t1 = CUDART_INF;
    for (int k = 0; k < 3; k++) {
      const double lo = G.lo[k], hi = G.lo[k] + G.n[k] * G.cell[k];
      if (e[k] == 0.0) {
        if (q[k] < lo || q[k] > hi) return false;
        continue;
      }
      const double ta = (lo - q[k]) / e[k], tb = (hi - q[k]) / e[k];
      t0 = fmax(t0, fmin(ta, tb));
      t1 = fmin(t1, fmax(ta, tb));
    }
    if (!(t0 <= t1)) return false;
    for (int k = 0; k < 3; k++) {
      const double f = (q[k] + t0 * e[k] - G.lo[k]) * G.inv[k];
      c[k] = min(max((int)floor(f), 0), G.n[k] - 1);
      if (e[k] > 0) { step[k] = 1; tnext[k] = (G.lo[k] + (c[k] + 1) * G.cell[k] - q[k]) / e[k]; tdelta[k] = G.cell[k] / e[k]; }
      else if (e[k] < 0) { step[k] = -1; tnext[k] = (G.lo[k] + c[k] * G.cell[k] - q[k]) / e[k]; tdelta[k] = -G.cell[k] / e[k]; }
      else { step[k] = 0; tnext[k] = CUDART_INF; tdelta[k] = CUDART_INF; }
    }
    tenter = t0;
    left = G.n[0] + G.n[1] + G.n[2] + 3;
    return true;
  }
  __device__ __forceinline__ int cell(const GridD& G) const { return G.start + (c[2] * G.n[1] + c[1]) * G.n[0] + c[0]; }
  // to the next cell; false once the ray has left the grid
  __device__ __forceinline__ bool advance(const GridD& G) {
    int k = 0;
    if (tnext[1] < tnext[k]) k = 1;
    if (tnext[2] < tnext[k]) k = 2;
    tenter = tnext[k];
    if (!(tenter <= t1) || --left <= 0) return false;
    c[k] += step[k];
    if (c[k] < 0 || c[k] >= G.n[k]) return false;
    tnext[k] += tdelta[k];
    return true;
  }
};

// Stop rule of the walk: no daughter in a cell entered after t can give a distance within
// the tie margin of `best`.
__device__ __forceinline__ bool walk_done(double tenter, double best) { return tenter > best + 4e-9 * (1.0 + best); }

// The world track in plain binary32 (hi parts).
__device__ __forceinline__ PlainTrack plain_world(const double p[3], const double d[3]) {
  const float x = (float)p[0], y = (float)p[1], z = (float)p[2];
  return {x, y, z, (float)d[0], (float)d[1], (float)d[2], 4e-6f * (fabsf(x) + fabsf(y) + fabsf(z))};
}
// No daughter first met at `from` or later can give a distance within a tie margin of `best`.
__device__ __forceinline__ bool beyond(float from, double best) { return (double)from > best + 1e-6 * (1.0 + best); }

// What is the same for every track of a launch.
struct Geo {
  const NodeD* nodes;
  const int32_t* children;
  const Desc* solids;
  const Cull* cull;
  int nnodes;
  Vox vox;
};

// The daughters of a node that a ray may enter, one after the other: all of them in index order, or,
// in a node with a grid, those listed in the cells along the ray; certain misses and daughters
// first met beyond the best distance so far are passed over.
struct Finder {
  const Geo& g;
  const NodeD& N;
  PlainTrack P;
  const GridD* G;  // nullptr: scan
  Dda D;
  int at, end, cells;  // next daughter and last one of the scan or of the current cell; cells left behind
  bool over;
  __device__ __forceinline__ Finder(const Geo& geo, const NodeD& node, const PlainTrack& plain, const double p[3],
                                    const double d[3])
      : g(geo), N(node), P(plain), G(nullptr), at(0), end(node.count), cells(0), over(false) {
    if (g.vox.grids && N.grid >= 0 && N.count >= kWalk32Min) {
      G = g.vox.grids + N.grid;
      double q[3], e[3];
      to_local64(N, p[0], p[1], p[2], q[0], q[1], q[2]);
      rot_local64(N, d[0], d[1], d[2], e[0], e[1], e[2]);
      over = !D.begin(*G, q, e);
      if (!over) cell();
    }
  }
  __device__ __forceinline__ void cell() {
    const int c = D.cell(*G);
    at = g.vox.cells[2 * c];
    end = g.vox.cells[2 * c + 1];
  }
  // go on where an earlier Finder of the same track stopped
  __device__ __forceinline__ void resume(int at0, int cells0) {
    if (G && !over) {
      for (; cells < cells0; cells++) D.advance(*G);
      cell();
    }
    at = at0;
  }
  // to the next cell of a grid
  __device__ __forceinline__ void leave_cell() {
    cells++;
    over = !D.advance(*G);
    if (!over) cell();
  }
  // the next daughter (-1: no more) given the best distance so far (`have`) and its node
  __device__ __forceinline__ int32_t next(bool have, double best, int32_t who) {
    while (!over) {
      for (; at < end; at++) {
        const int32_t id = G ? g.vox.list[at] : g.children[N.first + at];
        if (id == who) continue;  // listed in several cells
        const Cull& C = g.cull[id];
        float from;
        bool near;
        if (plain_miss(C, P, plain_local(C, P), from, near)) continue;
        if (have && beyond(from, best)) continue;
        at++;
        return id;
      }
      if (G) leave_cell();
      else over = true;
      over = over || (G && have && walk_done(D.tenter, best));
    }
    return -1;
  }
};

// The plain safety of a primitive (signed) in its own frame, and of a boolean.
static __device__ __noinline__ float plain_prim(const Desc& S, float x, float y, float z) {
  if (S.type == kBox) return fmaxf(fmaxf(fabsf(x) - S.Dh[0], fabsf(y) - S.Dh[1]), fabsf(z) - S.Dh[2]);
  if (S.type == kTrd || S.type == kTrap) {
    float v = fabsf(z) - S.dzh;
    for (int i = 0; i < 4; i++) v = fmaxf(v, fmaf(S.plh[i][2], z, fmaf(S.plh[i][1], y, S.plh[i][0] * x)) - S.plh[i][3]);
    return v;
  }
  const float r = sqrtf(fmaf(x, x, y * y));
  float phi = -f32::BIG, best = f32::BIG;
  if (S.flags & kHasPhi) {
    const float a = fmaf(S.nsh[0], x, S.nsh[1] * y), b = fmaf(S.neh[0], x, S.neh[1] * y);
    phi = (S.flags & kPhiWide) ? fminf(a, b) : fmaxf(a, b);
  }
  for (int k = 0; k + 1 < S.nz; k++) {
    float v = fmaxf((r - fmaf(S.oah[k], z, S.obh[k])) * S.ok_[k], fmaxf(S.zh[k] - z, z - S.zh[k + 1]));
    if ((S.inner >> k) & 1u) v = fmaxf(v, (fmaf(S.iah[k], z, S.ibh[k]) - r) * S.ik_[k]);
    best = fminf(best, v);
  }
  return fmaxf(best, phi);
}
static __device__ __noinline__ float plain_other(const Desc& S, float x, float y, float z) {
  if (S.type != kBool) return plain_prim(S, x, y, z);
  const double *M = S.bR, *t = S.bt;
  const float vx = x - (float)t[0], vy = y - (float)t[1], vz = z - (float)t[2];
  float q[3];
  for (int i = 0; i < 3; i++) q[i] = fmaf((float)M[6 + i], vz, fmaf((float)M[3 + i], vy, (float)M[i] * vx));
  const float a = plain_prim(S.parts[0], x, y, z), c = plain_prim(S.parts[1], q[0], q[1], q[2]);
  return S.bop == kUnion ? fminf(a, c) : S.bop == kIntersection ? fmaxf(a, c) : fmaxf(a, -c);
}

// The code of a point in a node's solid where plain binary32 can tell it: 2 certainly OUTSIDE, 0
// certainly INSIDE, else 1.
__device__ __forceinline__ int plain_code(const Geo& g, int32_t id, const PlainTrack& P) {
  const Cull& C = g.cull[id];
  const PlainLocal L = plain_local(C, P);
  if (plain_outside(C, L)) return 2;
  if (C.tag == kCullNever) return 1;
  const float s = C.tag <= kCullTube ? plain_safety(C, L) : plain_other(g.solids[C.solid], L.q[0], L.q[1], L.q[2]);
  const float m = C.tag <= kCullTube ? L.margin : 3.f * L.margin;
  return s > m ? 2 : s < -m ? 0 : 1;
}

// The cell of a grid whose safety list serves a point: the nearest one; its distance from the
// cell's centre (with margin).
__device__ __forceinline__ int safe_cell(const GridD& G, const NodeD& N, const Cull& C, const PlainTrack& P, float& dist) {
  const PlainLocal L = plain_local(C, P);
  int c[3];
  float d2 = 0.f;
#pragma unroll
  for (int a = 0; a < 3; a++) {
    c[a] = min(max((int)((L.q[a] - G.flo[a]) * G.finv[a]), 0), G.n[a] - 1);
    const float m = L.q[a] - (G.flo[a] + ((float)c[a] + 0.5f) * G.fcell[a]);
    d2 = fmaf(m, m, d2);
  }
  dist = 1.00001f * sqrtf(d2) + 4.f * L.margin;
  return (c[2] * G.n[1] + c[1]) * G.n[0] + c[0];
}

// A lower bound of the safety of a daughter.  (Without it a whole evaluation took the SafetyToIn of every
// daughter that is no box or full tube in binary64: step with safety among 512 daughters, a third of the
// tracks on surfaces, 300 tracks 3150 -> 1224 us, 200003 tracks 17.2 -> 6.2 ms.)
__device__ __forceinline__ float safety_from(const Geo& g, const Cull& C, const PlainTrack& P) {
  const PlainLocal L = plain_local(C, P);
  if (C.tag <= kCullTube) return plain_safety(C, L) - L.margin;
  // the walls' and the second component's rounding
  return plain_other(g.solids[C.solid], L.q[0], L.q[1], L.q[2]) - 3.f * L.margin;
}

// The daughters of a node that may have the least SafetyToIn, one after the other; a daughter whose
// lower bound exceeds the least safety so far is passed over.  With a safety list the daughters come
// in the order of their safety at the cell's centre s_c, and s_c less the point's distance from the
// centre is a lower bound (a safety changes by at most the distance between two points).  `never`:
// only the daughters without a binary32 form (else only the others).
struct Nearest {
  const Geo& g;
  const NodeD& N;
  const PlainTrack& P;
  const SafeEnt* list;  // nullptr: scan
  float dist, cut;
  int at;
  bool never;
  __device__ __forceinline__ Nearest(const Geo& geo, const NodeD& node, const Cull& C, const PlainTrack& p, bool nv)
      : g(geo), N(node), P(p), list(nullptr), dist(0.f), cut(kInf32), at(0), never(nv) {
    if (g.vox.grids && N.grid >= 0 && g.vox.grids[N.grid].safe >= 0) {
      const GridD& G = g.vox.grids[N.grid];
      const int cell = G.safe + safe_cell(G, N, C, P, dist);
      list = g.vox.safe + (int64_t)cell * kSafeList;
      cut = g.vox.safe_cut[cell];
    }
  }
  __device__ __forceinline__ void restart(bool nv) { at = 0; never = nv; }
  // are the daughters that no list holds certainly farther than `least`?
  __device__ __forceinline__ bool complete(double least) const { return !list || (double)(cut - dist) > least; }
  __device__ __forceinline__ int32_t next(double least) {
    const int count = list ? kSafeList : N.count;
    while (at < count) {
      int32_t id;
      if (list) {
        const SafeEnt E = list[at];
        if (E.node < 0 || (double)(E.s - dist) > least) break;
        id = E.node;
      } else {
        id = g.children[N.first + at];
      }
      at++;
      const Cull& C = g.cull[id];
      if ((C.tag == kCullNever) != never) continue;
      if ((double)safety_from(g, C, P) > least) continue;
      return id;
    }
    at = count;
    return -1;
  }
};

struct Step {
  double step, safety, second;  // second: the next smaller candidate, or a lower bound above every tie margin
  int32_t next;
};

__device__ __forceinline__ void local64(const NodeD& C, const double p[3], const double d[3], f64::Track& T) {
  to_local64(C, p[0], p[1], p[2], T.x, T.y, T.z);
  rot_local64(C, d[0], d[1], d[2], T.u, T.v, T.w);
}

// The step of a track in node v in binary64 throughout.
static __device__ __noinline__ void nav_exact(const Geo& g, int32_t v, const double p[3], const double d[3], bool want_saf,
                                              Step& out) {
  const NodeD& N = g.nodes[v];
  f64::Track T;
  f64::Result R;
  local64(N, p, d, T);
  query64(g.solids[N.desc], T, f64::kWantDout | (want_saf ? f64::kWantSout : 0u), R);
  double best = R.dout, runner = CUDART_INF, saf = R.sout;
  bool have = best >= 0, have_s = want_saf && saf >= 0;
  int32_t who = -1;
  Finder F(g, N, plain_world(p, d), p, d);
  for (int32_t id; (id = F.next(have, best, who)) >= 0;) {
    local64(g.nodes[id], p, d, T);
    query64(g.solids[g.nodes[id].desc], T, f64::kWantDin, R);
    const double t = R.din;
    if (t >= 0 && (!have || t < best || (t == best && (who == -1 || id < who)))) {
      if (have && best < runner) runner = best;
      best = t; who = id; have = true;
    } else if (t >= 0 && t < runner) {
      runner = t;
    }
  }
  if (want_saf) {
    Nearest S(g, N, g.cull[v], F.P, false);
    for (int pass = 0; pass < 2; pass++) {
      if (pass) {  // a list that may leave out the nearest: every daughter
        if (S.complete(have_s ? saf : CUDART_INF)) break;
        S.list = nullptr;
      }
      for (int nv = 0; nv < 2; nv++) {
        S.restart(nv != 0);
        for (int32_t id; (id = S.next(have_s ? saf : CUDART_INF)) >= 0;) {
          local64(g.nodes[id], p, d, T);
          query64(g.solids[g.nodes[id].desc], T, f64::kWantSin, R);
          if (R.sin >= 0 && (!have_s || R.sin < saf)) { saf = R.sin; have_s = true; }
        }
      }
    }
  }
  out.step = have ? best : -1.0;
  out.next = have ? who : -1;
  out.safety = have_s ? saf : -1.0;
  out.second = runner;
}

// Volume kinds for gathering tracks that run the same code (the paper's baskets of
// particles in one kind of volume): solid type, whether the volume has daughters and a grid.
constexpr int kKinds = 32;  // volume kinds (the last one: an empty slot)

__device__ __forceinline__ int volume_kind(const NodeD* __restrict__ nodes, const Desc* __restrict__ solids, int32_t v,
                                           const Vox& vox) {
  const NodeD& N = nodes[v];
  const int type = solids[N.desc].type;  // 0..6
  return type * 4 + (N.count > 0 ? 2 : 0) + (vox.grids && N.grid >= 0 ? 1 : 0);
}

// Order the m entries of a block by kind (counting sort in shared memory): perm[r] is the
// entry of rank r.  Block-uniform: every thread of the block calls it.
__device__ __forceinline__ void order_by_kind(int kind, int m, int* scount, int* perm) {
  const int t = threadIdx.x;
  if (t < kKinds) scount[t] = 0;
  __syncthreads();
  if (t < m) atomicAdd(&scount[kind], 1);
  __syncthreads();
  if (t == 0) {
    int acc = 0;
    for (int k = 0; k < kKinds; k++) { const int c = scount[k]; scount[k] = acc; acc += c; }
  }
  __syncthreads();
  if (t < m) perm[atomicAdd(&scount[kind], 1)] = t;
  __syncthreads();
}

// The same for a tile of len tracks (more than one per thread): perm[r] is the offset of rank r.
__device__ __forceinline__ void order_tile(const NodeD* __restrict__ nodes, const Desc* __restrict__ solids, int nnodes,
                                           const int32_t* __restrict__ node, int len, const Vox& vox, int* scount,
                                           uint8_t* skind, uint16_t* perm) {
  const int t = threadIdx.x;
  if (t < kKinds) scount[t] = 0;
  __syncthreads();
  for (int j = t; j < len; j += blockDim.x) {
    const int32_t v = node[j];
    const int kind = (v >= 0 && v < nnodes) ? volume_kind(nodes, solids, v, vox) : kKinds - 2;
    skind[j] = (uint8_t)kind;
    atomicAdd(&scount[kind], 1);
  }
  __syncthreads();
  if (t == 0) {
    int acc = 0;
    for (int k = 0; k < kKinds; k++) { const int c = scount[k]; scount[k] = acc; acc += c; }
  }
  __syncthreads();
  for (int j = t; j < len; j += blockDim.x) perm[atomicAdd(&scount[skind[j]], 1)] = (uint16_t)j;
  __syncthreads();
}

// ------------------------------------------------------------ binary32

// World point (split) -> node frame in double-float; direction rotated in binary32.
__device__ __forceinline__ f32::TrackF to_local32(const NodeD& N, const f32::TrackF& W) {
  using f32::F2;
  using f32::tprod;
  using f32::tsum;
  float dh[3], dl[3];
  const float ph[3] = {W.xh, W.yh, W.zh}, pl[3] = {W.xl, W.yl, W.zl};
  for (int k = 0; k < 3; k++) {
    const F2 s = tsum(ph[k], -N.th[k]);
    const float lo = s.l + (pl[k] - N.tl[k]);
    dh[k] = s.h + lo;
    dl[k] = lo - (dh[k] - s.h);
  }
  f32::TrackF L;
  float* oh[3] = {&L.xh, &L.yh, &L.zh};
  float* ol[3] = {&L.xl, &L.yl, &L.zl};
  for (int i = 0; i < 3; i++) {
    const F2 p0 = tprod(N.Rh[i], dh[0]), p1 = tprod(N.Rh[3 + i], dh[1]), p2 = tprod(N.Rh[6 + i], dh[2]);
    const F2 s1 = tsum(p0.h, p1.h), s2 = tsum(s1.h, p2.h);
    float lo = (s1.l + s2.l) + ((p0.l + p1.l) + p2.l);
    lo += N.Rh[i] * dl[0] + N.Rl[i] * dh[0];
    lo += N.Rh[3 + i] * dl[1] + N.Rl[3 + i] * dh[1];
    lo += N.Rh[6 + i] * dl[2] + N.Rl[6 + i] * dh[2];
    const float h = s2.h + lo;
    *oh[i] = h;
    *ol[i] = lo - (h - s2.h);
  }
  // direction in double-float as well: the quadratic coefficients use its low part
  const float uh[3] = {W.u, W.v, W.w}, ul[3] = {W.ul, W.vl, W.wl};
  float* dh_[3] = {&L.u, &L.v, &L.w};
  float* dl_[3] = {&L.ul, &L.vl, &L.wl};
  for (int i = 0; i < 3; i++) {
    const F2 p0 = tprod(N.Rh[i], uh[0]), p1 = tprod(N.Rh[3 + i], uh[1]), p2 = tprod(N.Rh[6 + i], uh[2]);
    const F2 s1 = tsum(p0.h, p1.h), s2 = tsum(s1.h, p2.h);
    float lo = (s1.l + s2.l) + ((p0.l + p1.l) + p2.l);
    lo += N.Rh[i] * ul[0] + N.Rl[i] * uh[0];
    lo += N.Rh[3 + i] * ul[1] + N.Rl[3 + i] * uh[1];
    lo += N.Rh[6 + i] * ul[2] + N.Rl[6 + i] * uh[2];
    const float h = s2.h + lo;
    *dh_[i] = h;
    *dl_[i] = lo - (h - s2.h);
  }
  L.zkey = 0;
  L.keyed = false;
  // The local point differs from the binary64 R^T (p - t) by the splits of p and t and the
  // double-float rounding: 2^-42 of |p|_1 + |t|_1 bounds it per coordinate; the rotated
  // direction is good to 2^-42 per component.
  L.fl = fmaf(f32::G42, fabsf(W.xh) + fabsf(W.yh) + fabsf(W.zh) + fabsf(N.th[0]) + fabsf(N.th[1]) + fabsf(N.th[2]),
              f32::FLOOR);
  L.dfl = f32::G42;
  L.bad = W.bad;
  return L;
}

// The planar and polycone-family passes are called, not inlined: inlined into the
// navigation kernel, the union of every family's code needed 247 registers (one block per
// SM); called, the kernel fits two blocks per SM (boxes, the common daughters, stay inline).
__device__ __noinline__ void planar32_call(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  f32::planar32<true>(S, T, want, R);
}
__device__ __noinline__ void tube32_call(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  f32::pcon32<true, true>(S, T, want, R);
}
__device__ __noinline__ void pcon32_call(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  f32::pcon32<false, true>(S, T, want, R);
}

__device__ __forceinline__ void query32(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  R.flag = T.bad;
  R.code = 1;
  R.din = R.dout = R.sin = R.sout = 0.f;
  if (R.flag) return;
  if (S.flags & kFp64Only) {  // features finer than binary32 resolves: binary64 only
    R.flag = true;
    return;
  }
  // frame tracks: the bounds add the local coordinates' and direction's own errors
  if (S.type == kBox) f32::box32<true>(S, T, want, R);
  else if (S.type == kTrd || S.type == kTrap) planar32_call(S, T, want, R);
  else if (S.type == kTube) tube32_call(S, T, want, R);
  else if (S.type == kBool) R.flag = true;  // booleans: binary64 only
  else pcon32_call(S, T, want, R);
}

// The ranking instances of the passes in a placed volume's frame (rank_fp64.cuh).
__device__ __noinline__ void planar_rank_call(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  f32::planar32<true, true>(S, T, want, R);
}
__device__ __noinline__ void tube_rank_call(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  f32::pcon32<true, true, true>(S, T, want, R);
}
__device__ __noinline__ void pcon_rank_call(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  f32::pcon32<false, true, true>(S, T, want, R);
}
__device__ __forceinline__ void rank_local32(const Desc& S, const f32::TrackF& T, unsigned want, f32::R32& R) {
  R.flag = T.bad || S.type == kBool || (S.flags & kFp64Only);
  R.code = 1;
  R.din = R.dout = R.sin = R.sout = 0.f;
  R.rank = 0u;
  R.te = R.se = 0.f;
  if (R.flag) return;
  if (S.type == kBox) f32::box32<true, true>(S, T, want, R);
  else if (S.type == kTrd || S.type == kTrap) planar_rank_call(S, T, want, R);
  else if (S.type == kTube) tube_rank_call(S, T, want, R);
  else pcon_rank_call(S, T, want, R);
}
// The ranking with the code from binary64, for a track whose code binary32 cannot certify.
static __device__ __noinline__ void rank_given_call(const Desc& S, const f64::Track& T64, const f32::TrackF& T, unsigned want,
                                                    f32::R32& R) {
  R.flag = T.bad || S.type == kBool || (S.flags & kFp64Only);
  if (R.flag) return;
  R.code = f64::code_of(f64::prim_s(S, T64.x, T64.y, T64.z));
  R.din = R.dout = R.sin = R.sout = 0.f;
  R.rank = 0u;
  R.te = R.se = 0.f;
  if (S.type == kBox) f32::box32<true, true, true>(S, T, want, R);
  else if (S.type == kTrd || S.type == kTrap) f32::planar32<true, true, true>(S, T, want, R);
  else if (S.type == kTube) f32::pcon32<true, true, true, true>(S, T, want, R);
  else f32::pcon32<false, true, true, true>(S, T, want, R);
}
__device__ __noinline__ void planar_ranked_call(const Desc& S, const f64::Track& T, f64::Verdict V, f64::Result& R) {
  f64::planar_ranked(S, T, V, R);
}
__device__ __noinline__ void pcon_ranked_call(const Desc& S, const f64::Track& T, f64::Verdict V, f64::Result& R) {
  f64::pcon_ranked(S, T, V, R);
}
__device__ __forceinline__ void ranked_local64(const Desc& S, const f64::Track& T, uint32_t rank, f64::Result& R) {
  const f64::Verdict V{rank};
  if (S.type == kBox) f64::box_ranked(S, T, V, R);
  else if (S.type == kTrd || S.type == kTrap) planar_ranked_call(S, T, V, R);
  else pcon_ranked_call(S, T, V, R);
}

// half of the output tolerance: the certified binary32 results are within it
__device__ __forceinline__ float half_tol(float t) { return 0.5f * (t < 1e-4f ? 1e-9f : 1e-5f * t); }

// Two smallest candidates (value, error, key); key = daughter order (or node index on a
// grid walk), mother = kMother.  With DEDUP the two keys are distinct: a key already held
// is not added again (a daughter met in several cells gives the same value each time);
// without it (every daughter evaluated once) the second key is not tracked.
template <bool DEDUP>
struct Top2 {
  float b1, e1, b2, e2;
  int w1, w2;
  __device__ __forceinline__ void add(float t, float e, int w) {
    if (DEDUP && (w == w1 || w == w2)) return;
    if (t < b1 || (t == b1 && w < w1)) {
      if (DEDUP) w2 = w1;
      b2 = b1; e2 = e1; b1 = t; e1 = e; w1 = w;
    } else if (t < b2) {
      b2 = t; e2 = e;
      if (DEDUP) w2 = w;
    }
  }
};

// Merge the Top2 of the lanes selected by `mask` (a group of kLanes lanes, xor offsets).
template <bool DEDUP>
__device__ __forceinline__ void group_merge(unsigned mask, Top2<DEDUP>& top) {
  constexpr int kNone = 0x7fffffff;
  for (int off = kLanes / 2; off > 0; off >>= 1) {
    const float ob1 = __shfl_xor_sync(mask, top.b1, off), oe1 = __shfl_xor_sync(mask, top.e1, off);
    const float ob2 = __shfl_xor_sync(mask, top.b2, off), oe2 = __shfl_xor_sync(mask, top.e2, off);
    const int ow1 = __shfl_xor_sync(mask, top.w1, off);
    const int ow2 = DEDUP ? __shfl_xor_sync(mask, top.w2, off) : kNone;
    top.add(ob1, oe1, ow1);
    top.add(ob2, oe2, ow2);
  }
}

// One thread per track, for geometries whose nodes are scanned (no grid walk): the block takes its
// tracks in order of volume kind in tiles of 1024; every daughter gets the plain look of
// nav_cull.cuh, and only those it leaves (a ray that may meet the daughter, a safety that may be
// the least) are evaluated with certified bounds.  A lane leaves from none to a dozen daughters, so
// the warp gathers its 32 tracks' (track, daughter) pairs in shared memory and evaluates them 32 at
// a time, one per lane; each lane then reads its own pairs' results.
// Measured (GB300, nested detector, 2^22 tracks with safety): 12.0 -> 2.80 ms (before: 8 lanes per
// track, every daughter evaluated: 1214 warp instructions per track at 18 of 32 lanes; now 263 at 26).
// Without the pairs, each lane evaluating its own daughters: 5.8 ms (12 lanes).  Three blocks per SM
// (80 registers) 2.73, tiles of 2048 2.72 ms.
constexpr int kScanTile = 1024;
constexpr int kScanPairs = 256;  // pairs a warp evaluates per round
struct ScanWarp {
  float w[12][32];           // the warp's tracks, split (world frame)
  int32_t node[32];
  uint32_t pair[kScanPairs]; // track's lane << 27 | daughter order
  float din[kScanPairs], sin[kScanPairs];  // results (din NaN: flagged)
};
__global__ void __launch_bounds__(256, 2) k_nav_scan32(const NodeD* __restrict__ nodes, const int32_t* __restrict__ children,
                                                       const Desc* __restrict__ solids, const Cull* __restrict__ cull,
                                                       int nnodes, NavArgs a, uint32_t* __restrict__ wl,
                                                       unsigned long long* __restrict__ cnt, Vox vox) {
  constexpr int kMother = 0x7ffffffe, kNone = 0x7fffffff;
  const unsigned lane = threadIdx.x & 31u;
  const bool want_saf = a.safety != nullptr;
  const unsigned want = f32::kWantDin | (want_saf ? f32::kWantSin : 0u);
  const uint2 *X = reinterpret_cast<const uint2*>(a.x), *Y = reinterpret_cast<const uint2*>(a.y),
              *Z = reinterpret_cast<const uint2*>(a.z), *Ux = reinterpret_cast<const uint2*>(a.u),
              *Uy = reinterpret_cast<const uint2*>(a.v), *Uz = reinterpret_cast<const uint2*>(a.w);
  __shared__ int scount[kKinds];
  __shared__ uint16_t sperm[kScanTile];
  __shared__ uint8_t skind[kScanTile];
  __shared__ ScanWarp swarp[8];
  ScanWarp& Q = swarp[threadIdx.x >> 5];
  const int tile = a.n >= (int64_t)gridDim.x * kScanTile ? kScanTile : 256;  // short baskets: more blocks
  for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < a.n; t0 += (int64_t)gridDim.x * tile) {  // block-uniform
    const int len = a.n - t0 < tile ? (int)(a.n - t0) : tile;
    order_tile(nodes, solids, nnodes, a.node + t0, len, vox, scount, skind, sperm);
    for (int r0 = 0; r0 < len; r0 += 256) {
      const int r = r0 + (int)threadIdx.x;
      const bool valid = r < len;
      const int64_t i = t0 + (valid ? sperm[r] : 0);
      bool flag = false;
      Top2<false> top{F_INF, 0.f, F_INF, 0.f, kNone, kNone};
      float saf = F_INF, mdout = 0.f, mssf = 0.f;
      int32_t v = -1;
      PlainTrack P;
      int count = 0;
      const int32_t* ids = nullptr;
      if (valid) {
        v = a.node[i];
        flag = v < 0 || v >= nnodes || nodes[v].never;  // a daughter without binary32 form: binary64
      }
      if (valid && !flag) {
        const f32::TrackF W = f32::load_track(X, Y, Z, Ux, Uy, Uz, i, true);
        const float c[12] = {W.xh, W.yh, W.zh, W.xl, W.yl, W.zl, W.u, W.v, W.w, W.ul, W.vl, W.wl};
#pragma unroll
        for (int k = 0; k < 12; k++) Q.w[k][lane] = c[k];
        const NodeD& N = nodes[v];
        f32::R32 R;
        query32(solids[N.desc], to_local32(N, W), f32::kWantDout | (want_saf ? f32::kWantSout : 0u), R);
        flag = W.bad || R.flag || R.dout < 0;  // a point outside its own volume: binary64 decides
        top.add(R.dout, half_tol(R.dout), kMother);
        if (want_saf) saf = R.sout;
        mdout = R.dout;
        mssf = saf;
        P = plain_track(W);
        ids = children + N.first;
        count = flag ? 0 : N.count;
      }
      // The plain look.  s1, s2: the two daughters of least plain safety among those not evaluated
      // anyway; s3 the third's; ub the upper bound of the least safety.
      float s1 = F_INF, s2 = F_INF, s3 = F_INF, ub = saf;
      int j1 = -1, j2 = -1, j0 = 0;
      bool all = false;  // evaluate every daughter (several of nearly the same safety)
      while (__any_sync(0xffffffffu, j0 < count)) {
        unsigned mask = 0u;
        const int m = min(32, count - j0);
        for (int b = 0; b < m; b++) {
          const Cull& C = cull[ids[j0 + b]];
          const int tag = C.tag;
          bool take = all;
          if (!take) {
            const PlainLocal L = plain_local(C, P);
            float from;
            bool near;
            take = !plain_miss(C, P, L, from, near) || near;
            if (want_saf) {
              const bool own = tag <= kCullTube;
              const float s = own ? plain_safety(C, L) : plain_other(solids[C.solid], L.q[0], L.q[1], L.q[2]);
              const float m = own ? L.margin : 3.f * L.margin, lb = s - m;
              ub = fminf(ub, s < m ? F_INF : s + m);  // a point not outside gives none
              if (take) {  // evaluated anyway
              } else if (lb < s1) {
                s3 = s2; s2 = s1; j2 = j1; s1 = lb; j1 = j0 + b;
              } else if (lb < s2) {
                s3 = s2; s2 = lb; j2 = j0 + b;
              } else {
                s3 = fminf(s3, lb);
              }
            }
          }
          if (take) mask |= 1u << b;
        }
        const int first = j0;
        j0 += 32;
        if (want_saf && !all && m > 0 && j0 >= count) {  // the last daughters: those of least safety too
          if (s3 <= ub) {  // start over, without the look
            all = true;
            j0 = 0;
            mask = 0u;
            top = Top2<false>{mdout, half_tol(mdout), F_INF, 0.f, kMother, kNone};
            saf = mssf;
          } else {
            if (!(s1 <= ub)) j1 = -1;
            if (!(s2 <= ub)) j2 = -1;
          }
        }
        const bool ends = want_saf && !all && m > 0 && j0 >= count;
        // evaluate the pairs in rounds
        unsigned extra = ends ? (j1 >= 0 ? 1u : 0u) | (j2 >= 0 ? 2u : 0u) : 0u;
        while (__any_sync(0xffffffffu, mask | extra)) {
          const int mine = __popc(mask) + __popc(extra);
          int at = mine;
          for (int o = 1; o < 32; o <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, at, o);
            if ((int)lane >= o) at += up;
          }
          const int total = min(__shfl_sync(0xffffffffu, at, 31), kScanPairs);
          at -= mine;
          int end = at;
          while ((mask | extra) && end < kScanPairs) {
            int j;
            if (mask) {
              j = first + __ffs(mask) - 1;
              mask &= mask - 1u;
            } else {
              j = (extra & 1u) ? j1 : j2;
              extra &= extra - 1u;
            }
            Q.pair[end++] = lane << 27 | (uint32_t)j;
          }
          Q.node[lane] = v;
          __syncwarp();
          for (int q = (int)lane; q < total; q += 32) {
            const uint32_t e = Q.pair[q];
            const unsigned l = e >> 27;
            f32::TrackF W;
            W.xh = Q.w[0][l]; W.yh = Q.w[1][l]; W.zh = Q.w[2][l];
            W.xl = Q.w[3][l]; W.yl = Q.w[4][l]; W.zl = Q.w[5][l];
            W.u = Q.w[6][l]; W.v = Q.w[7][l]; W.w = Q.w[8][l];
            W.ul = Q.w[9][l]; W.vl = Q.w[10][l]; W.wl = Q.w[11][l];
            W.bad = false;
            const NodeD& C = nodes[children[nodes[Q.node[l]].first + (int)(e & 0x7ffffffu)]];
            f32::R32 R;
            query32(solids[C.desc], to_local32(C, W), want, R);
            Q.din[q] = R.flag ? CUDART_NAN_F : R.din;
            Q.sin[q] = R.sin;
          }
          __syncwarp();
          for (int q = at; q < end; q++) {
            const float t = Q.din[q];
            flag |= isnan(t);
            if (t >= 0) top.add(t, half_tol(t), (int)(Q.pair[q] & 0x7ffffffu));
            if (want_saf && Q.sin[q] >= 0) saf = fminf(saf, Q.sin[q]);
          }
          __syncwarp();
        }
      }
      if (valid && !flag) {
        // the winner must be certain: the runner-up's interval may not meet it; no finite step:
        // binary64 decides
        flag = !isfinite(top.b1) || top.b2 - top.e2 <= top.b1 + top.e1;
        if (!flag) {
          a.step[i] = (double)top.b1;
          if (want_saf) a.safety[i] = isfinite(saf) ? (double)saf : -1.0;
          a.next[i] = top.w1 == kMother ? -1 : ids[top.w1];
        }
      }
      const bool push = valid && flag;
      const unsigned m = __ballot_sync(0xffffffffu, push);
      if (m) {
        unsigned long long at = 0;
        const int leader = __ffs(m) - 1;
        if ((int)lane == leader) at = atomicAdd(cnt, (unsigned long long)__popc(m));
        at = __shfl_sync(0xffffffffu, at, leader);
        if (push) wl[at + __popc(m & ((1u << lane) - 1u))] = (uint32_t)i;
      }
    }
    __syncthreads();  // the tile's shared arrays are reused by the next tile
  }
}

// Geometries with nodes whose daughters the pass finds by walking their grid: kLanes lanes per track.
// A listed daughter that the ray certainly misses (nav_cull.cuh) gets no certified evaluation: that is
// most of them, and the frame change and pass of the rest bound the walk.  Measured (GB300, 1728
// daughters, 2^18 tracks without safety, the same bits): 10.8 -> 4.2 ms; 1000 daughters, 10^5 tracks:
// 4.8 -> 2.0 ms.  Leaving the walk at the first flag gained nothing.
// WALK false: every node is scanned (short baskets; one instance for both cost 300 tracks 2 of 29 us).
template <bool WALK>
__global__ void __launch_bounds__(256, 2) k_nav_fp32(const NodeD* __restrict__ nodes, const int32_t* __restrict__ children,
                                                  const Desc* __restrict__ solids, const Cull* __restrict__ cull,
                                                  int nnodes, NavArgs a,
                                                  uint32_t* __restrict__ wl, unsigned long long* __restrict__ cnt,
                                                  Vox vox) {
  constexpr int kMother = 0x7ffffffe, kNone = 0x7fffffff;
  const unsigned lane = threadIdx.x & 31u, sub = lane & (kLanes - 1);
  const unsigned gmask = ((1u << kLanes) - 1u) << (lane & ~(unsigned)(kLanes - 1));
  const bool want_saf = a.safety != nullptr;
  const int64_t tracks_per_block = blockDim.x / kLanes;
  const int64_t stride = (int64_t)gridDim.x * tracks_per_block;
  const uint2 *X = reinterpret_cast<const uint2*>(a.x), *Y = reinterpret_cast<const uint2*>(a.y),
              *Z = reinterpret_cast<const uint2*>(a.z), *Ux = reinterpret_cast<const uint2*>(a.u),
              *Uy = reinterpret_cast<const uint2*>(a.v), *Uz = reinterpret_cast<const uint2*>(a.w);
  __shared__ int scount[kKinds];
  __shared__ int sperm[256];
  for (int64_t base = (int64_t)blockIdx.x * tracks_per_block; base < a.n; base += stride) {  // block-uniform
    // the block's tracks in order of the kind of volume they are in (a warp's four tracks
    // then mostly run the same path)
    int kind = kKinds - 1;
    if (threadIdx.x < tracks_per_block && base + threadIdx.x < a.n) {
      const int32_t v0 = a.node[base + threadIdx.x];
      kind = (v0 >= 0 && v0 < nnodes) ? volume_kind(nodes, solids, v0, vox) : kKinds - 2;
    }
    order_by_kind(kind, (int)tracks_per_block, scount, sperm);
    const int64_t i = base + sperm[threadIdx.x / kLanes];
    const bool valid = i < a.n;
    bool flag = false;
    Top2<WALK> top{F_INF, 0.f, F_INF, 0.f, kNone, kNone};
    float saf = F_INF;
    int32_t v = -1;
    bool walked = false;  // keys are node indices (grid walk) rather than daughter order
    if (valid) {
      v = a.node[i];
      if (v < 0 || v >= nnodes) {
        flag = true;
      } else {
        const NodeD& N = nodes[v];
        walked = WALK && vox.grids && N.grid >= 0 && N.count >= kWalk32Min;
        flag = N.never && (want_saf || !walked);  // a daughter without binary32 form would be met: binary64
      }
    }
    if (valid && !flag) {
      const f32::TrackF W = f32::load_track(X, Y, Z, Ux, Uy, Uz, i, true);
      const NodeD& N = nodes[v];
      if (sub == 0) {  // the mother on the group's first lane
        const f32::TrackF L = to_local32(N, W);
        f32::R32 R;
        query32(solids[N.desc], L, f32::kWantDout | (want_saf ? f32::kWantSout : 0u), R);
        flag |= R.flag || R.dout < 0;  // a point outside its own volume: binary64 decides
        top.add(R.dout, half_tol(R.dout), kMother);
        if (want_saf) saf = R.sout;
      }
      const unsigned want = (walked ? 0u : f32::kWantDin) | (want_saf ? f32::kWantSin : 0u);
      for (int j = sub; want != 0u && j < N.count; j += kLanes) {
        const NodeD& C = nodes[children[N.first + j]];
        const f32::TrackF L = to_local32(C, W);
        f32::R32 R;
        query32(solids[C.desc], L, want, R);
        flag |= R.flag;
        if (!walked && R.din >= 0) top.add(R.din, half_tol(R.din), j);
        if (want_saf && R.sin >= 0) saf = fminf(saf, R.sin);
      }
      if (walked) {  // DistanceToIn of the daughters listed along the ray, cell by cell
        const GridD& G = vox.grids[N.grid];
        double q[3], e[3];
        to_local64(N, a.x[i], a.y[i], a.z[i], q[0], q[1], q[2]);
        rot_local64(N, a.u[i], a.v[i], a.w[i], e[0], e[1], e[2]);
        const PlainTrack P = plain_track(W);
        Dda D;
        if (D.begin(G, q, e)) {
          do {
            // every lane of the group holds the group's two best after the merge
            group_merge(gmask, top);
            const double bound = (double)top.b1 + (double)top.e1;
            if (isfinite(top.b1) && walk_done(D.tenter, bound)) break;
            const int cell = D.cell(G);
            for (int j = vox.cells[2 * cell] + (int)sub; j < vox.cells[2 * cell + 1]; j += kLanes) {
              const int32_t id = vox.list[j];
              const Cull& B = cull[id];
              float from;
              bool near;
              if (B.tag != kCullNever && plain_miss(B, P, plain_local(B, P), from, near) && !near) continue;
              const NodeD& C = nodes[id];
              const f32::TrackF L = to_local32(C, W);
              f32::R32 R;
              query32(solids[C.desc], L, f32::kWantDin, R);
              flag |= R.flag;
              if (R.din >= 0) top.add(R.din, half_tol(R.din), id);
            }
          } while (D.advance(G));
        }
      }
    }
    // combine the group's lanes with shuffles (xor within the group of kLanes)
    group_merge(0xffffffffu, top);
    for (int off = kLanes / 2; off > 0; off >>= 1) {
      const float os = __shfl_xor_sync(0xffffffffu, saf, off);
      const int of = __shfl_xor_sync(0xffffffffu, (int)flag, off);
      saf = fminf(saf, os);
      flag |= of != 0;
    }
    // the winner must be certain: the runner-up's interval may not meet it
    if (valid && !flag && isfinite(top.b1) && top.b2 - top.e2 <= top.b1 + top.e1) flag = true;
    if (valid && !flag && !isfinite(top.b1)) flag = true;  // no finite step: binary64 decides
    if (valid && sub == 0 && !flag) {
      const NodeD& N = nodes[v];
      a.step[i] = (double)top.b1;
      if (want_saf) a.safety[i] = isfinite(saf) ? (double)saf : -1.0;
      a.next[i] = top.w1 == kMother ? -1 : walked ? top.w1 : children[N.first + top.w1];
    }
    const bool push = valid && sub == 0 && flag;
    const unsigned m = __ballot_sync(0xffffffffu, push);
    if (m) {
      unsigned long long at = 0;
      const int leader = __ffs(m) - 1;
      if ((int)lane == leader) at = atomicAdd(cnt, (unsigned long long)__popc(m));
      at = __shfl_sync(0xffffffffu, at, leader);
      if (push) wl[at + __popc(m & ((1u << lane) - 1u))] = (uint32_t)i;
    }
  }
}

// ------------------------------------------------- binary64 steps, ranked in binary32

// The binary32 track of a binary64 point and direction, split as the bulk pass splits its
// inputs (world frame: no frame error yet).
__device__ __forceinline__ f32::TrackF track_from(const double p[3], const double d[3]) {
  auto bits = [](double v) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    return make_uint2((unsigned)b, (unsigned)(b >> 32));
  };
  f32::TrackF T;
  T.bad = false;
  T.fl = f32::FLOOR;
  T.dfl = 0.f;
  T.keyed = false;
  T.zkey = 0;
  f32::split(bits(p[0]), T.xh, T.xl, T.bad);
  f32::split(bits(p[1]), T.yh, T.yl, T.bad);
  f32::split(bits(p[2]), T.zh, T.zl, T.bad);
  T.u = f32::trunc_hi(bits(d[0]), T.bad);
  T.v = f32::trunc_hi(bits(d[1]), T.bad);
  T.w = f32::trunc_hi(bits(d[2]), T.bad);
  bool unused = false;
  float h;
  f32::split(bits(d[0]), h, T.ul, unused);
  f32::split(bits(d[1]), h, T.vl, unused);
  f32::split(bits(d[2]), h, T.wl, unused);
  return T;
}

// The step of nav_exact, bit for bit, for the tracks of a block's pool, with the candidates ranked by
// certified binary32 intervals.  The block works in phases, every one over all of its tracks, so that
// its warps run the same code at the same time (the passes of all families together exceed the
// instruction cache) and the lanes of a warp mostly one family:
//   gather    each track's candidates: the mother's exit and the daughters a plain look leaves
//             (Finder), up to kPoolPairs (track, volume) pairs
//   evaluate  the pairs in order of solid family, one per lane: certified distance and verdict
//   merge     the nearest interval and the lower bound of the others; tracks with more daughters that
//             may be nearer gather again
//   finish    in order of the nearest volume's family: its crossing in binary64 (rank_fp64.cuh)
// The least safety comes from plain binary32 values with margins; the one or two daughters (and the
// mother) within reach of the least are evaluated in binary64.  A track whose nearest interval is not
// apart from the others by more than the tie margins goes to nav_exact.
// Measured (GB300, same bits as evaluating every candidate in binary64): step with safety among 1728
// daughters, 2^18 tracks, 112 -> 2.5 ms (every daughter's safety in binary64 kept the FP64 pipe 81% busy;
// ranking per thread, without phases: 9.9 ms, instruction fetch); transport in the nested detector, 2^20
// tracks, 32 steps, 56.7 -> 11.5 ms (per thread 21.3 ms; 14.9 before the
// relocation in step and the gathered physics).  Bound by latency: one block per SM, 14-20% of the
// issue slots, 6-18 of 32 lanes.  1024 threads (64 registers) against 512: step 2.5 against 2.8 ms, transport
// then 15.0 against 14.9 ms.
constexpr int kPoolPairs = 4;
enum : uint8_t { kSlotIdle = 0, kSlotMore = 1, kSlotRanked = 2, kSlotExact = 3 };
enum : int { kKeyBox = 0, kKeyPlanar = 1, kKeyTube = 2, kKeyPcon = 3, kKeyNever = 4, kKeyExact = 5, kKeys = 6 };

template <int SLOTS>
struct StepPool {
  double p[3][SLOTS], d[3][SLOTS];
  int32_t v[SLOTS], who[SLOTS];
  float lo[SLOTS], hi[SLOTS], second[SLOTS];  // nearest candidate's interval, lower bound of the others
  uint32_t rank[SLOTS], mrank[SLOTS];         // verdicts of the nearest and of the mother
  float slo[SLOTS], shi[SLOTS];               // the mother's safety
  float from[SLOTS];                          // no daughter left is entered before
  int32_t at[SLOTS], cells[SLOTS];            // where its Finder stopped
  int32_t pid[kPoolPairs * SLOTS];            // pairs: the volume; results: t (NaN: not certain), error, verdict
  float t[kPoolPairs * SLOTS], e[kPoolPairs * SLOTS];
  uint32_t prank[kPoolPairs * SLOTS];
  uint16_t order[kPoolPairs * SLOTS], perm[SLOTS];
  uint8_t state[SLOTS], np[SLOTS];
  int cnt[2][8];  // by key, of the two sorts in turn
  __device__ __forceinline__ void get(int s, double P[3], double D[3]) const {
    for (int c = 0; c < 3; c++) { P[c] = p[c][s]; D[c] = d[c][s]; }
  }
};

__device__ __forceinline__ int pool_key(const Cull& C) {
  if (C.tag == kCullNever) return kKeyNever;
  return C.family;
}

// Exclusive sums of cnt[0..kKeys) (every thread calls it); returns the total.
__device__ __forceinline__ int key_sums(int* cnt) {
  __syncthreads();
  int total = 0;
  for (int k = 0; k < kKeys; k++) total += cnt[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    int run = 0;
    for (int k = 0; k < kKeys; k++) { const int c = cnt[k]; cnt[k] = run; run += c; }
  }
  __syncthreads();
  return total;
}

// Rank the pool's tracks (state kSlotMore, v valid; the slots perm[0..n)): afterwards every one is
// kSlotRanked or kSlotExact.  Every thread of the block calls it.
template <int NT, int SLOTS>
__device__ __forceinline__ void pool_rank(const Geo& g, StepPool<SLOTS>& Q, int n, bool want_saf) {
  const int tid = threadIdx.x;
  bool first = true;
  while (true) {
    if (tid < kKeys) Q.cnt[0][tid] = 0;
    __syncthreads();
    for (int r = tid; r < n; r += NT) {
      const int s = Q.perm[r];
      int k = 0;
      if (Q.state[s] == kSlotMore) {
        const int32_t v = Q.v[s];
        const NodeD& N = g.nodes[v];
        if (first && g.cull[v].tag == kCullNever) {
          Q.state[s] = kSlotExact;
        } else {
          double p[3], d[3];
          Q.get(s, p, d);
          const PlainTrack P = plain_world(p, d);
          int32_t* pid = Q.pid + kPoolPairs * s;
          if (first) pid[k++] = v;
          if (g.vox.grids && N.grid >= 0 && N.count >= kWalk32Min) {
            Finder F(g, N, P, p, d);
            if (!first) F.resume(Q.at[s], Q.cells[s]);
            const double best = first ? 0.0 : (double)Q.hi[s];
            const int32_t who = first ? -1 : Q.who[s];
            float from = 0.f;
            // up to kPoolPairs pairs, and no farther than the cell that brings two daughters
            while (k < kPoolPairs) {
              const int32_t id = F.next(!first, best, who);
              if (id < 0) break;
              pid[k++] = id;
              if (F.at >= F.end && k >= 2) {
                F.leave_cell();
                if (!F.over) from = (float)F.D.tenter * (1.f - 1e-6f);
                if (k >= 3) break;
              }
            }
            Q.at[s] = F.at;
            Q.cells[s] = F.cells;
            Q.from[s] = F.over ? kInf32 : from;
          } else {
            // the three daughters that may be entered first (later rounds: the next three); `by`: one
            // of those seen is certainly entered by then
            float f1 = kInf32, f2 = kInf32, f3 = kInf32, f4 = kInf32, by = first ? kInf32 : Q.hi[s];
            int32_t c1 = -1, c2 = -1, c3 = -1;
            const float past = first ? -1.f : Q.from[s];
            const int32_t past_id = first ? -1 : Q.at[s];
            for (int j = 0; j < N.count; j++) {
              const int32_t id = g.children[N.first + j];
              const Cull& C = g.cull[id];
              float f, u;
              if (plain_entry(C, P, plain_local(C, P), f, u)) continue;
              by = fminf(by, u);
              if (f > by || f < past || (f == past && id <= past_id)) continue;
              if (f < f1) { f4 = f3; f3 = f2; c3 = c2; f2 = f1; c2 = c1; f1 = f; c1 = id; }
              else if (f < f2) { f4 = f3; f3 = f2; c3 = c2; f2 = f; c2 = id; }
              else if (f < f3) { f4 = f3; f3 = f; c3 = id; }
              else f4 = fminf(f4, f);
            }
            float from = kInf32;
            int32_t last = -1;
            const float fs[3] = {f1, f2, f3};
            const int32_t cs[3] = {c1, c2, c3};
#pragma unroll
            for (int c = 0; c < 3; c++)
              if (cs[c] >= 0 && !beyond(fs[c], (double)by)) {
                pid[k++] = cs[c];
                from = fs[c];
                last = cs[c];
              }
            const bool rest = c3 >= 0 && last == c3 && !beyond(f4, (double)by) && f4 < kInf32;
            Q.at[s] = last;
            Q.from[s] = rest ? from : kInf32;
          }
          for (int c = 0; c < k; c++) atomicAdd(&Q.cnt[0][pool_key(g.cull[Q.pid[kPoolPairs * s + c]])], 1);
        }
      }
      Q.np[s] = (uint8_t)k;
    }
    const int total = key_sums(Q.cnt[0]);
    for (int r = tid; r < n; r += NT) {
      const int s = Q.perm[r];
      for (int c = 0; c < Q.np[s]; c++) {
        const int i = kPoolPairs * s + c;
        Q.order[atomicAdd(&Q.cnt[0][pool_key(g.cull[Q.pid[i]])], 1)] = (uint16_t)i;
      }
    }
    __syncthreads();
    for (int q = tid; q < total; q += NT) {
      const int i = Q.order[q], s = i / kPoolPairs;
      const bool mother = first && i % kPoolPairs == 0;
      const int32_t id = Q.pid[i];
      const NodeD& C = g.nodes[id];
      const Desc& S = g.solids[C.desc];
      double p[3], d[3];
      Q.get(s, p, d);
      if (g.cull[id].tag == kCullNever) {  // no binary32 form: the binary64 value itself
        f64::Track T;
        f64::Result R;
        local64(C, p, d, T);
        query64(S, T, f64::kWantDin, R);
        const float t = (float)R.din;
        Q.t[i] = t;
        Q.e[i] = t < f32::BIG ? 2.f * f32::U * fabsf(t) : 0.f;  // the cast's rounding: near ties go to nav_exact
        Q.prank[i] = ~0u;
      } else {
        f32::R32 R;
        const unsigned want = !mother ? f32::kWantDin : want_saf ? f32::kWantDout | f32::kWantSout : f32::kWantDout;
        const f32::TrackF L = to_local32(C, track_from(p, d));
        rank_local32(S, L, want, R);
        if (R.flag) {
          f64::Track T;
          local64(C, p, d, T);
          rank_given_call(S, T, L, want, R);
        }
        const float t = mother ? R.dout : R.din;
        Q.t[i] = R.flag || (mother && t < 0.f) ? CUDART_NAN_F : t;
        Q.e[i] = fmaf(2.f * f32::U, fabsf(t), R.te);
        Q.prank[i] = R.rank;
        if (mother) {
          const float es = fmaf(2.f * f32::U, fabsf(R.sout), R.se);
          Q.slo[s] = R.sout - es;
          Q.shi[s] = R.sout + es;
        }
      }
    }
    __syncthreads();
    bool more = false;
    for (int r = tid; r < n; r += NT) {
      const int s = Q.perm[r], k = Q.np[s];
      if (Q.state[s] != kSlotMore) continue;
      float lo, hi, second;
      int32_t who;
      uint32_t rank;
      int c = 0;
      if (first) {
        const int i = kPoolPairs * s;
        lo = Q.t[i] - Q.e[i]; hi = Q.t[i] + Q.e[i]; second = kInf32;
        who = -1;
        rank = Q.mrank[s] = Q.prank[i];
        c = 1;
      } else {
        lo = Q.lo[s]; hi = Q.hi[s]; second = Q.second[s]; who = Q.who[s]; rank = Q.rank[s];
      }
      bool ok = !isnan(hi);
      for (; c < k; c++) {
        const int i = kPoolPairs * s + c;
        const float t = Q.t[i], l = t - Q.e[i], h = t + Q.e[i];
        ok &= !isnan(t);
        if (!(t >= 0.f)) continue;
        if (h < hi) {
          second = fminf(second, lo);
          lo = l; hi = h; who = Q.pid[i]; rank = Q.prank[i];
        } else if (Q.pid[i] != who) {
          second = fminf(second, l);
        }
      }
      Q.lo[s] = lo; Q.hi[s] = hi; Q.second[s] = second; Q.who[s] = who; Q.rank[s] = rank;
      if (!ok) Q.state[s] = kSlotExact;
      else if (beyond(Q.from[s], (double)hi) || Q.from[s] == kInf32)
        Q.state[s] = second - hi > 4e-9f * (1.f + hi) && hi < f32::BIG ? kSlotRanked : kSlotExact;
      else more = true;
    }
    first = false;
    if (!__syncthreads_or(more)) break;
  }
}

// The candidates for a ranked track's least safety: the mother (bit 0 of the result) and up to two
// daughters j1, j2 (-1: none); false in `ok` when a third one is within reach.
template <int SLOTS>
__device__ __forceinline__ bool pool_safety(const Geo& g, const StepPool<SLOTS>& Q, int s, int32_t& j1, int32_t& j2, bool& ok) {
  const int32_t v = Q.v[s];
  const NodeD& N = g.nodes[v];
  double p[3], d[3];
  Q.get(s, p, d);
  const PlainTrack P = plain_world(p, d);
  float ub = Q.shi[s], s1 = kInf32, s2 = kInf32, s3 = kInf32;  // least upper bound; the least lower bounds
  j1 = j2 = -1;
  const SafeEnt* list = nullptr;
  float dist = 0.f, cut = kInf32;
  int count = N.count;
  if (g.vox.grids && N.grid >= 0 && g.vox.grids[N.grid].safe >= 0) {
    const GridD& G = g.vox.grids[N.grid];
    const int cell = G.safe + safe_cell(G, N, g.cull[v], P, dist);
    list = g.vox.safe + (int64_t)cell * kSafeList;
    cut = g.vox.safe_cut[cell];
    count = kSafeList;
  }
  for (int at = 0; at < count; at++) {
    int32_t id;
    if (list) {
      const SafeEnt E = list[at];
      if (E.node < 0 || E.s - dist > ub) break;
      id = E.node;
    } else {
      id = g.children[N.first + at];
    }
    const Cull& C = g.cull[id];
    const PlainLocal L = plain_local(C, P);
    float sf, m = L.margin;
    if (C.tag <= kCullTube) {
      sf = plain_safety(C, L);
    } else {
      sf = plain_other(g.solids[C.solid], L.q[0], L.q[1], L.q[2]);
      m *= 3.f;  // the walls' and the second component's rounding
    }
    if (!(sf < m)) ub = fminf(ub, sf + m);  // a point not certainly outside gives no upper bound
    const float lb = sf - m;
    if (lb < s1) {
      s3 = s2; s2 = s1; j2 = j1; s1 = lb; j1 = id;
    } else if (lb < s2) {
      s3 = s2; s2 = lb; j2 = id;
    } else {
      s3 = fminf(s3, lb);
    }
  }
  ok = s3 > ub && (!list || cut - dist > ub);
  if (!(s1 <= ub)) j1 = -1;
  if (!(s2 <= ub)) j2 = -1;
  return Q.slo[s] <= ub;
}

// The binary64 step of slot s after pool_rank (and, with want_saf, its safety candidates).
template <int SLOTS>
__device__ __forceinline__ void pool_finish(const Geo& g, const StepPool<SLOTS>& Q, int s, bool want_saf, Step& out) {
  const int32_t v = Q.v[s];
  double p[3], d[3];
  Q.get(s, p, d);
  if (Q.state[s] == kSlotExact) {
    nav_exact(g, v, p, d, want_saf, out);
    return;
  }
  const int32_t who = Q.who[s];
  const uint32_t rank = Q.rank[s];
  f64::Track T;
  f64::Result R;
  const NodeD& M = g.nodes[who < 0 ? v : who];
  local64(M, p, d, T);
  if (rank == ~0u) query64(g.solids[M.desc], T, f64::kWantDin, R);
  else ranked_local64(g.solids[M.desc], T, rank, R);
  out.step = who < 0 ? R.dout : R.din;
  out.next = who;
  out.second = (double)Q.second[s];
  if (want_saf) {
    const int32_t j[3] = {Q.np[s] ? v : -1, Q.pid[kPoolPairs * s], Q.pid[kPoolPairs * s + 1]};
    double saf = CUDART_INF;
    for (int c = 0; c < 3; c++) {
      if (j[c] < 0) continue;
      const NodeD& C = g.nodes[j[c]];
      local64(C, p, d, T);
      double val;
      if (c == 0) {
        ranked_local64(g.solids[C.desc], T, Q.mrank[s] & ~(7u << 11), R);  // the safety only
        val = R.sout;
      } else {
        query64(g.solids[C.desc], T, f64::kWantSin, R);
        val = R.sin;
      }
      if (val >= 0 && val < saf) saf = val;
    }
    out.safety = saf < CUDART_INF ? saf : -1.0;
  }
}

// Order the pool's n tracks (perm) by the family of the volume that finishes them, into order[].
template <int NT, int SLOTS>
__device__ __forceinline__ void pool_order(const Geo& g, StepPool<SLOTS>& Q, int n) {
  const int tid = threadIdx.x;
  auto key = [&](int s) {
    if (Q.state[s] != kSlotRanked) return (int)kKeyExact;
    return pool_key(g.cull[Q.who[s] < 0 ? Q.v[s] : Q.who[s]]);
  };
  if (tid < kKeys) Q.cnt[1][tid] = 0;
  __syncthreads();
  for (int r = tid; r < n; r += NT) atomicAdd(&Q.cnt[1][key(Q.perm[r])], 1);
  key_sums(Q.cnt[1]);
  for (int r = tid; r < n; r += NT) {
    const int s = Q.perm[r];
    Q.order[atomicAdd(&Q.cnt[1][key(s)], 1)] = (uint16_t)s;
  }
  __syncthreads();
}

// Order the pool's live slots (live(s)) by volume kind into perm[0..n); returns n.
template <int NT, int SLOTS, class Live>
__device__ __forceinline__ int pool_kinds(const Geo& g, StepPool<SLOTS>& Q, int* scount, Live live) {
  const int tid = threadIdx.x;
  if (tid < kKinds) scount[tid] = 0;
  __syncthreads();
  for (int s = tid; s < SLOTS; s += NT)
    if (live(s)) atomicAdd(&scount[volume_kind(g.nodes, g.solids, Q.v[s], g.vox)], 1);
  __syncthreads();
  int n = 0;
  for (int k = 0; k < kKinds; k++) n += scount[k];
  __syncthreads();
  if (tid == 0) {
    int run = 0;
    for (int k = 0; k < kKinds; k++) { const int c = scount[k]; scount[k] = run; run += c; }
  }
  __syncthreads();
  for (int s = tid; s < SLOTS; s += NT)
    if (live(s)) Q.perm[atomicAdd(&scount[volume_kind(g.nodes, g.solids, Q.v[s], g.vox)], 1)] = (uint16_t)s;
  __syncthreads();
  return n;
}

// The binary64 step of the tracks 0..n-1, or (wl) of the n listed ones, in tiles of at most SLOTS
// tracks per block, short ones spread over every block.
constexpr int kNavSlots = 1024, kNavThreads = 1024;
// Binary32 baskets of at most this many tracks do not fill the GPU one thread per track: 8 lanes take a
// track (k_nav_fp32; not where volumes have 128 daughters and more to scan, or daughters without a binary32
// form, which go to binary64 at once), and what is left goes to k_nav_exact.  Measured (GB300, with safety, against k_nav_scan32 and
// k_nav_pool): nested detector, 300 tracks 46 -> 30 us, 8000 tracks 54 -> 35 us (16000: 54.1 against 53.1 us);
// 512 daughters of all kinds, 300 tracks 1530 -> 697 us, 8000 tracks 1895 -> 928 us.
constexpr int64_t kShortBasket = 8192;
__global__ void __launch_bounds__(kNavThreads, 1) k_nav_pool(Geo g, NavArgs a, const uint32_t* __restrict__ wl,
                                                              const unsigned long long* __restrict__ cnt) {
  extern __shared__ __align__(16) unsigned char pool_bytes[];
  StepPool<kNavSlots>& Q = *reinterpret_cast<StepPool<kNavSlots>*>(pool_bytes);
  __shared__ int scount[kKinds];
  const int tid = threadIdx.x;
  const bool want_saf = a.safety != nullptr;
  const int64_t total = cnt ? (int64_t)*cnt : a.n;
  const int64_t share = (total + gridDim.x - 1) / gridDim.x;
  const int tile = share >= kNavSlots ? kNavSlots : max((int)share, 8);
  for (int64_t t0 = (int64_t)blockIdx.x * tile; t0 < total; t0 += (int64_t)gridDim.x * tile) {
    const int len = total - t0 < tile ? (int)(total - t0) : tile;
    for (int s = tid; s < kNavSlots; s += kNavThreads) {
      Q.state[s] = kSlotIdle;
      if (s >= len) continue;
      const int64_t i = wl ? (int64_t)wl[t0 + s] : t0 + s;
      const int32_t v = a.node[i];
      if (v < 0 || v >= g.nnodes) {
        a.step[i] = -1.0; a.next[i] = -1;
        if (want_saf) a.safety[i] = -1.0;
        continue;
      }
      Q.v[s] = v;
      Q.p[0][s] = a.x[i]; Q.p[1][s] = a.y[i]; Q.p[2][s] = a.z[i];
      Q.d[0][s] = a.u[i]; Q.d[1][s] = a.v[i]; Q.d[2][s] = a.w[i];
      Q.state[s] = kSlotMore;
    }
    __syncthreads();
    const int n = pool_kinds<kNavThreads>(g, Q, scount, [&](int s) { return Q.state[s] == kSlotMore; });
    pool_rank<kNavThreads>(g, Q, n, want_saf);
    if (want_saf) {
      for (int r = tid; r < n; r += kNavThreads) {
        const int s = Q.perm[r];
        if (Q.state[s] != kSlotRanked) continue;
        int32_t j1, j2;
        bool ok;
        Q.np[s] = pool_safety(g, Q, s, j1, j2, ok) ? 1 : 0;
        Q.pid[kPoolPairs * s] = j1;
        Q.pid[kPoolPairs * s + 1] = j2;
        if (!ok) Q.state[s] = kSlotExact;
      }
      __syncthreads();
    }
    pool_order<kNavThreads>(g, Q, n);
    for (int r = tid; r < n; r += kNavThreads) {
      const int s = Q.order[r];
      const int64_t i = wl ? (int64_t)wl[t0 + s] : t0 + s;
      Step o;
      pool_finish(g, Q, s, want_saf, o);
      a.step[i] = o.step;
      if (want_saf) a.safety[i] = o.safety;
      a.next[i] = o.next;
    }
    __syncthreads();  // the pool is reused by the next tile
  }
}

// The listed tracks evaluated whole, one per thread, consecutive ones in consecutive blocks of one
// warp: the refinement of baskets up to kShortBasket, whose few tracks the pool's phases would only delay.
// Bound by the latency of one track's chain (blocks of 64 threads, one per SM: 958 against 731 us for 3000
// tracks among 512 daughters).
__global__ void __launch_bounds__(32) k_nav_exact(Geo g, NavArgs a, const uint32_t* __restrict__ wl,
                                                  const unsigned long long* __restrict__ cnt) {
  const int64_t m = (int64_t)*cnt, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t j = (int64_t)threadIdx.x * gridDim.x + blockIdx.x; j < m; j += stride) {
    const int64_t i = wl[j];
    const int32_t v = a.node[i];
    Step o{-1.0, -1.0, 0.0, -1};
    if (v >= 0 && v < g.nnodes) {
      const double p[3] = {a.x[i], a.y[i], a.z[i]}, d[3] = {a.u[i], a.v[i], a.w[i]};
      nav_exact(g, v, p, d, a.safety != nullptr, o);
    }
    a.step[i] = o.step;
    if (a.safety) a.safety[i] = o.safety;
    a.next[i] = o.next;
  }
}

// ------------------------------------------------------------ transport loop

// Locate one point in binary64 (gv_nav_locate's definition: from the world down, enter
// the first daughter, in index order or in the point's grid cell, that does not classify
// the point OUTSIDE; -1 outside the world) and report whether any classification on the
// way was SURFACE (the point lies on a boundary within the tolerance).
static __device__ __noinline__ int32_t locate64_surf(const Geo& g, double x, double y, double z, bool& surf) {
  const NodeD* nodes = g.nodes;
  const Desc* solids = g.solids;
  const double p[3] = {x, y, z}, d0[3] = {0.0, 0.0, 0.0};
  const PlainTrack P = plain_world(p, d0);
  f64::Track T{0, 0, 0, 0, 0, 0};
  f64::Result R;
  to_local64(nodes[0], x, y, z, T.x, T.y, T.z);
  query64(solids[nodes[0].desc], T, f64::kWantCode, R);
  surf |= R.code == 1;
  if (R.code == 2) return -1;
  int32_t v = 0;
  for (int depth = 0; depth < 64; depth++) {
    const NodeD& N = nodes[v];
    int32_t into = -1;
    const int32_t* ids;
    int count;
    candidates64(N, g.children, g.vox, x, y, z, ids, count);  // a daughter whose band holds the point is listed
    for (int j = 0; j < count; j++) {
      const int32_t c = ids[j];
      if (plain_code(g, c, P) == 2) continue;
      to_local64(nodes[c], x, y, z, T.x, T.y, T.z);
      query64(solids[nodes[c].desc], T, f64::kWantCode, R);
      surf |= R.code == 1;
      if (R.code != 2) { into = c; break; }
    }
    if (into < 0) break;
    v = into;
  }
  return v;
}

// Locate as locate64_surf, with the codes taken in binary32 when every one on the way is
// certified (a certified code is the binary64 one); otherwise locate64_surf decides.
// Lanes go down the tree with plain codes until they need a certified one, and take that together.
__device__ __forceinline__ int32_t locate_rank32(const Geo& g, double x, double y, double z, bool& surf) {
  const double p[3] = {x, y, z}, d0[3] = {0.0, 0.0, 0.0};
  const f32::TrackF W = track_from(p, d0);
  const PlainTrack P = plain_track(W);
  bool ok = !W.bad, done = W.bad, sf = false;
  int32_t v = -1;                // the node reached
  const int32_t* ids = nullptr;  // the daughters to look at (first the world), the next one
  int at = 0, count = 1, depth = 0;
  const unsigned lanes = __activemask();
  while (__any_sync(lanes, !done)) {
    int32_t need = -1, into = -1;
    while (!done && at < count) {
      const int32_t c = ids ? ids[at] : 0;
      const int look = plain_code(g, c, P);
      if (look == 2) { at++; continue; }
      if (look == 0) into = c;
      else need = c;
      break;
    }
    __syncwarp(lanes);
    if (need >= 0) {
      f32::R32 R;
      query32(g.solids[g.nodes[need].desc], to_local32(g.nodes[need], W), f32::kWantCode, R);
      if (R.flag) {
        ok = false;
        done = true;
      } else {
        sf |= R.code == 1;
        if (R.code != 2) into = need;
        else at++;
      }
    } else if (into < 0) {
      done = true;  // in none of the daughters
    }
    __syncwarp(lanes);
    if (into >= 0) {
      v = into;
      at = 0;
      done = ++depth > 64;
      if (!candidates32(g.nodes[v], g.cull[v], g.children, g.vox, P, ids, count))
        candidates64(g.nodes[v], g.children, g.vox, x, y, z, ids, count);
    }
  }
  if (ok) {
    surf |= sf;
    return v;
  }
  return locate64_surf(g, x, y, z, surf);
}

// gv_nav_locate: one thread per track, the codes in binary32 where they are certain.
__global__ void __launch_bounds__(256, 2) k_locate32(Geo g, const double* __restrict__ x, const double* __restrict__ y,
                                                  const double* __restrict__ z, int32_t* __restrict__ out, int64_t n) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride) {
    bool surf = false;
    out[i] = locate_rank32(g, x[i], y[i], z[i], surf);
  }
}

struct TransportArgs {
  const double *x, *y, *z, *u, *v, *w;  // start points and directions
  const int32_t* node0;                 // start volumes
  const int32_t* material;              // material of every node
  const double* sigma_n;                // n sigma of (scatter, absorb) per material, 1/mm
  const double* xi;                     // random numbers, [n][kmax][4], in (0, 1]
  int32_t kmax, nmat, nnodes;
  int8_t* reason;
  int32_t* steps;
  double *xo, *yo, *zo, *path;
  int32_t* last;
  int8_t* tie;
  int64_t n;
};

constexpr double kPush = 1e-6;  // probe distance past a boundary for the relocation (mm)

// The state of one track in the loop.
struct Flight {
  double p[3], d[3], len;
  int32_t v, k, why;
  bool near, live;
  bool reloc;  // at a boundary, to be located again (the second half of a step)
};

__device__ __forceinline__ void flight_begin(const TransportArgs& a, int64_t i, Flight& F) {
  F.p[0] = a.x[i]; F.p[1] = a.y[i]; F.p[2] = a.z[i];
  F.d[0] = a.u[i]; F.d[1] = a.v[i]; F.d[2] = a.w[i];
  F.v = a.node0[i];
  F.k = 0;
  F.why = GV_TRUNCATED;
  F.near = false;
  F.reloc = false;
  F.len = 0.0;
  F.live = F.v >= 0 && F.v < a.nnodes && a.kmax > 0;
  if (F.v < 0) F.why = GV_ESCAPED;
  else if (F.v >= a.nnodes) F.why = GV_LOST;
}

// Bounds in binary32 of the sampled step -log(xi) / sigma (sigma <= 0: none, +inf).
__device__ __forceinline__ float free_path_from(double xi, double sigma) {
  const float s = (float)sigma;
  if (!(sigma > 0)) return F_INF;
  // the argument's rounding moves the logarithm by at most 1.2e-7; the rest is relative
  const float v = -logf((float)xi), lo = __fdividef(v - fmaf(4e-6f, fabsf(v), 4e-7f), s);
  return v < 80.f && s > 1e-30f ? lo : 0.f;  // beyond binary32: binary64 decides
}

// One step of the loop of the Physics subsection (see gv.h), after its geometry (o), in two parts.
// First: lost tracks, and those whose physics steps both exceed the boundary distance by more than the
// tie margin, certainly in binary32: these go to the boundary.  True: the physics step decides.
__device__ __forceinline__ bool flight_geometry(const TransportArgs& a, int64_t i, const Step& o, Flight& F) {
  const double* r = a.xi + ((size_t)i * (size_t)a.kmax + (size_t)F.k) * 4;
  const double dgeo = o.step;
  const int32_t m = a.material[F.v];
  if (dgeo < 0 || m < 0 || m >= a.nmat) { F.why = GV_LOST; F.live = false; return false; }
  if (fabs(o.second - dgeo) <= 1e-9 * (1.0 + dgeo)) F.near = true;
  const float reach = (float)dgeo * 1.00001f + 1e-6f;
  if (!(free_path_from(r[0], a.sigma_n[2 * m]) > reach && free_path_from(r[1], a.sigma_n[2 * m + 1]) > reach)) return true;
  F.k++;
  for (int j = 0; j < 3; j++) F.p[j] = xadd(F.p[j], xmul(dgeo, F.d[j]));
  F.len = xadd(F.len, dgeo);
  F.reloc = true;  // the probe point past the boundary is located by flight_locate
  return false;
}

// Second: the physics step in binary64 against the boundary distance and, when the process acts first,
// the process.
__device__ __forceinline__ void flight_physics(const TransportArgs& a, int64_t i, double dgeo, Flight& F) {
  const double* r = a.xi + ((size_t)i * (size_t)a.kmax + (size_t)F.k) * 4;
  const int32_t m = a.material[F.v];
  const double sig0 = a.sigma_n[2 * m], sig1 = a.sigma_n[2 * m + 1];
  const double s0 = sig0 > 0 ? -log(r[0]) / sig0 : CUDART_INF;
  const double s1 = sig1 > 0 ? -log(r[1]) / sig1 : CUDART_INF;
  const int proc = s1 < s0 ? 1 : 0;
  const double sp = proc ? s1 : s0;
  if (fabs(sp - dgeo) <= 1e-9 * (1.0 + dgeo)) F.near = true;
  F.k++;
  if (sp < dgeo) {  // the process acts before the boundary
    for (int j = 0; j < 3; j++) F.p[j] = xadd(F.p[j], xmul(sp, F.d[j]));
    F.len = xadd(F.len, sp);
    if (proc == 1) { F.why = GV_ABSORBED; F.live = false; return; }
    const double ca = xsub(xmul(2.0, r[2]), 1.0), b = xmul(6.283185307179586, r[3]);
    const double sa = sqrt(fmax(0.0, xsub(1.0, xmul(ca, ca))));
    double sb, cb;
    sincos(b, &sb, &cb);
    F.d[0] = xmul(sa, cb); F.d[1] = xmul(sa, sb); F.d[2] = ca;
  } else {  // to the boundary
    for (int j = 0; j < 3; j++) F.p[j] = xadd(F.p[j], xmul(dgeo, F.d[j]));
    F.len = xadd(F.len, dgeo);
    F.reloc = true;
    return;
  }
  if (F.k >= a.kmax) F.live = false;  // truncated
}

// The second half of a step that ended at a boundary: locate the probe point past it.
__device__ inline void flight_locate(const Geo& g, const TransportArgs& a, Flight& F) {
  bool surf = false;
  F.reloc = false;
  const double q0 = xadd(F.p[0], xmul(kPush, F.d[0])), q1 = xadd(F.p[1], xmul(kPush, F.d[1])),
               q2 = xadd(F.p[2], xmul(kPush, F.d[2]));
  F.v = locate_rank32(g, q0, q1, q2, surf);
  F.near |= surf;
  if (F.v < 0) { F.why = GV_ESCAPED; F.live = false; return; }
  if (F.k >= a.kmax) F.live = false;  // truncated
}

__device__ __forceinline__ void flight_end(const TransportArgs& a, int64_t i, const Flight& F) {
  a.reason[i] = (int8_t)F.why;
  a.steps[i] = F.k;
  a.xo[i] = F.p[0]; a.yo[i] = F.p[1]; a.zo[i] = F.p[2];
  a.path[i] = F.len;
  a.last[i] = F.why == GV_ESCAPED ? -1 : F.v;
  a.tie[i] = F.near ? 1 : 0;
}

// The transport loop in baskets (the paper's scheduler gathers particles that sit in the same kind
// of volume, so that they run the same code): a block keeps a pool of tracks in shared memory and
// loops: dead slots take the next tracks of the block's range; pool_rank ranks every live track's step
// and pool_finish evaluates it in binary64; then the process or the boundary takes the track on, and
// those at a boundary, gathered into the first warps, are located again.  Tracks take from one to kmax
// steps; the pool keeps the block busy until its range is used up.
constexpr int kFlightSlots = 1024, kFlightThreads = 512;
struct FlightPool {
  StepPool<kFlightSlots> q;
  double len[kFlightSlots];
  int64_t idx[kFlightSlots];
  int32_t k[kFlightSlots];
  uint8_t why[kFlightSlots], near[kFlightSlots], live[kFlightSlots], reloc[kFlightSlots];
  unsigned long long next;
  int scount[kKinds], nreloc, nphys;
  double dgeo[kFlightSlots];
};

__device__ __forceinline__ void flight_load(const FlightPool& P, int s, Flight& F) {
  P.q.get(s, F.p, F.d);
  F.len = P.len[s]; F.v = P.q.v[s]; F.k = P.k[s]; F.why = P.why[s]; F.near = P.near[s]; F.live = true; F.reloc = false;
}
__device__ __forceinline__ void flight_store(FlightPool& P, int s, const Flight& F) {
  for (int c = 0; c < 3; c++) { P.q.p[c][s] = F.p[c]; P.q.d[c][s] = F.d[c]; }
  P.len[s] = F.len; P.q.v[s] = F.v; P.k[s] = F.k; P.why[s] = (uint8_t)F.why; P.near[s] = F.near;
}

__global__ void __launch_bounds__(kFlightThreads, 1) k_transport(Geo g, TransportArgs a) {
  extern __shared__ __align__(16) unsigned char pool_bytes[];
  FlightPool& P = *reinterpret_cast<FlightPool*>(pool_bytes);
  const int t = threadIdx.x;
  const int64_t chunk = (a.n + gridDim.x - 1) / gridDim.x;
  const int64_t begin = (int64_t)blockIdx.x * chunk;
  const int64_t end = begin + chunk < a.n ? begin + chunk : a.n;
  if (t == 0) P.next = (unsigned long long)(begin < end ? begin : end);
  for (int s = t; s < kFlightSlots; s += kFlightThreads) P.live[s] = 0;
  __syncthreads();
  while (true) {
    // dead slots take the next tracks of the range
    bool any = false;
    for (int s = t; s < kFlightSlots; s += kFlightThreads) {
      if (!P.live[s]) {
        const unsigned long long j = atomicAdd(&P.next, 1ull);
        if ((int64_t)j < end) {
          Flight F;
          flight_begin(a, (int64_t)j, F);
          any = true;
          if (F.live) {
            P.idx[s] = (int64_t)j;
            flight_store(P, s, F);
            P.live[s] = 1;
          } else {
            flight_end(a, (int64_t)j, F);
          }
        }
      }
      P.q.state[s] = P.live[s] ? kSlotMore : kSlotIdle;
      any |= P.live[s] != 0;
    }
    if (!__syncthreads_or(any)) break;
    const int n = pool_kinds<kFlightThreads>(g, P.q, P.scount, [&](int s) { return P.live[s] != 0; });
    pool_rank<kFlightThreads>(g, P.q, n, false);
    pool_order<kFlightThreads>(g, P.q, n);
    if (t == 0) P.nreloc = P.nphys = 0;
    __syncthreads();
    // what the step came to: the track goes on (to be located when at a boundary) or ends
    auto settle = [&](int s, const Flight& F) {
      if (F.live) {
        flight_store(P, s, F);
        if (F.reloc) P.q.perm[atomicAdd(&P.nreloc, 1)] = (uint16_t)s;
      } else {
        flight_end(a, P.idx[s], F);
        P.live[s] = 0;
      }
    };
    for (int r = t; r < n; r += kFlightThreads) {
      const int s = P.q.order[r];
      Step o;
      pool_finish(g, P.q, s, false, o);
      Flight F;
      flight_load(P, s, F);
      if (flight_geometry(a, P.idx[s], o, F)) {  // gathered, so that the logarithms run on full warps
        P.near[s] = F.near;
        P.dgeo[s] = o.step;
        P.q.pid[atomicAdd(&P.nphys, 1)] = s;
      } else {
        settle(s, F);
      }
    }
    __syncthreads();
    for (int r = t; r < P.nphys; r += kFlightThreads) {
      const int s = P.q.pid[r];
      Flight F;
      flight_load(P, s, F);
      flight_physics(a, P.idx[s], P.dgeo[s], F);
      settle(s, F);
    }
    __syncthreads();
    // the tracks at a boundary
    const int nreloc = P.nreloc;
    for (int r = t; r < nreloc; r += kFlightThreads) {
      const int s = P.q.perm[r];
      Flight F;
      flight_load(P, s, F);
      flight_locate(g, a, F);
      if (F.live) {
        P.q.v[s] = F.v; P.near[s] = F.near;
      } else {
        flight_end(a, P.idx[s], F);
        P.live[s] = 0;
      }
    }
    __syncthreads();
  }
}

// The safety lists of one grid (one block per cell): lower bounds of the daughters' SafetyToIn at the
// cell's centre by the plain look, then kSafeList times the least of them.  A thread keeps the least of
// its own daughters and looks for the next one only when that is taken.  Measured (GB300, gv_geom_create
// of 4096 and 8000 daughters): 24.7 -> 6.4 and 77.3 -> 12.8 ms, of which 1.4 and 4.0 are these lists (before: every
// SafetyToIn in binary64, and every value read again for every entry of a list).
__global__ void __launch_bounds__(256) k_safe_lists(Geo g, int node, SafeEnt* __restrict__ list, float* __restrict__ cut) {
  extern __shared__ float val[];
  __shared__ unsigned long long best[2][8];
  const NodeD& N = g.nodes[node];
  const GridD& G = g.vox.grids[N.grid];
  const int cell = blockIdx.x, i = cell % G.n[0], j = cell / G.n[0] % G.n[1], k = cell / G.n[0] / G.n[1];
  const double q[3] = {G.lo[0] + (i + 0.5) * G.cell[0], G.lo[1] + (j + 0.5) * G.cell[1], G.lo[2] + (k + 0.5) * G.cell[2]};
  double p[3], d[3] = {0.0, 0.0, 0.0};
  for (int r = 0; r < 3; r++) p[r] = N.R[3 * r] * q[0] + N.R[3 * r + 1] * q[1] + N.R[3 * r + 2] * q[2] + N.t[r];
  const PlainTrack P = plain_world(p, d);
  auto key = [&](int c) { return (unsigned long long)__float_as_uint(val[c]) << 32 | (unsigned)c; };
  // values are not negative: their bit patterns order them
  unsigned long long own = ~0ull;
  for (int c = threadIdx.x; c < N.count; c += blockDim.x) {
    const Cull& C = g.cull[g.children[N.first + c]];
    const PlainLocal L = plain_local(C, P);
    const bool exact = C.tag <= kCullTube;
    const float s = exact ? plain_safety(C, L) : plain_other(g.solids[C.solid], L.q[0], L.q[1], L.q[2]);
    val[c] = fmaxf(s - (exact ? 1.f : 3.f) * L.margin, 0.f);
    own = min(own, key(c));
  }
  const int64_t at = (int64_t)(G.safe + cell) * kSafeList;
  for (int e = 0; e <= kSafeList; e++) {
    unsigned long long m = own;
    for (int o = 16; o > 0; o >>= 1) m = min(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0) best[e & 1][threadIdx.x >> 5] = m;
    __syncthreads();
    for (int w = 0; w < 8; w++) m = min(m, best[e & 1][w]);
    const bool none = (unsigned)(m >> 32) >= 0x7f800000u;  // all taken
    const int c = (int)(m & 0xffffffffu);
    if (threadIdx.x == 0) {
      const float s = none ? F_INF : __uint_as_float((unsigned)(m >> 32));
      if (e < kSafeList) list[at + e] = none ? SafeEnt{F_INF, -1} : SafeEnt{s, g.children[N.first + c]};
      else cut[G.safe + cell] = s;
    }
    if (!none && c % (int)blockDim.x == (int)threadIdx.x) {
      val[c] = F_INF;
      own = ~0ull;
      for (int b = threadIdx.x; b < N.count; b += blockDim.x) own = min(own, key(b));
    }
  }
}

}  // namespace gv

using namespace gv;

static void split_f(double v, float& h, float& l) {
  h = (float)v;
  l = (float)(v - (double)h);
}

namespace gv {

// Half-extents of an origin-centred box holding the solid in its own frame, recorded by
// the solid's constructor.
static void solid_half(const Desc& h, double e[3]) {
  for (int i = 0; i < 3; i++) e[i] = h.ext[i];
}

// Grids for the nodes with at least kVoxelMin daughters: the box around the daughters'
// (padded) bounding boxes in the node's frame, cut into about one cell per daughter.
static void build_grids(gv_geom* g) {
  for (int v = 0; v < g->nnodes; v++) {
    NodeD& N = g->nodes[v];
    N.grid = -1;
    if (N.count < kVoxelMin) continue;
    std::vector<std::array<double, 6>> box(N.count);  // lo, hi per daughter in v's frame
    double glo[3] = {1e300, 1e300, 1e300}, ghi[3] = {-1e300, -1e300, -1e300};
    for (int j = 0; j < N.count; j++) {
      const NodeD& C = g->nodes[g->children[N.first + j]];
      // p_v = Rv^T (Rc p_c + tc - tv): M = Rv^T Rc, b = Rv^T (tc - tv)
      double M[9], b[3], e[3];
      for (int r = 0; r < 3; r++) {
        for (int c = 0; c < 3; c++)
          M[3 * r + c] = N.R[0 * 3 + r] * C.R[0 * 3 + c] + N.R[1 * 3 + r] * C.R[1 * 3 + c] + N.R[2 * 3 + r] * C.R[2 * 3 + c];
        b[r] = N.R[0 * 3 + r] * (C.t[0] - N.t[0]) + N.R[1 * 3 + r] * (C.t[1] - N.t[1]) + N.R[2 * 3 + r] * (C.t[2] - N.t[2]);
      }
      solid_half(g->solids[C.desc], e);
      for (int r = 0; r < 3; r++) {
        const double h = std::fabs(M[3 * r]) * e[0] + std::fabs(M[3 * r + 1]) * e[1] + std::fabs(M[3 * r + 2]) * e[2];
        const double pad = 1e-6 * (1.0 + std::fabs(b[r]) + h);  // far above the rounding of any frame change
        box[j][r] = b[r] - h - pad;
        box[j][3 + r] = b[r] + h + pad;
        glo[r] = std::fmin(glo[r], box[j][r]);
        ghi[r] = std::fmax(ghi[r], box[j][3 + r]);
      }
    }
    GridD G;
    const double vol = std::fmax((ghi[0] - glo[0]) * (ghi[1] - glo[1]) * (ghi[2] - glo[2]), 1e-300);
    const double edge = std::cbrt(vol / N.count);
    for (int r = 0; r < 3; r++) {
      G.n[r] = (int)std::min(64.0, std::max(1.0, std::ceil((ghi[r] - glo[r]) / edge)));
      G.lo[r] = glo[r];
      G.cell[r] = (ghi[r] - glo[r]) / G.n[r];
      G.inv[r] = 1.0 / G.cell[r];
      G.flo[r] = (float)G.lo[r];
      G.fcell[r] = (float)G.cell[r];
      G.finv[r] = (float)G.inv[r];
    }
    G.safe = -1;
    G.start = (int)(g->cells.size() / 2);
    const int ncell = G.n[0] * G.n[1] * G.n[2];
    std::vector<std::vector<int32_t>> lists(ncell);
    for (int j = 0; j < N.count; j++) {  // daughters in increasing node index
      int c0[3], c1[3];
      for (int r = 0; r < 3; r++) {
        c0[r] = std::max(0, std::min(G.n[r] - 1, (int)std::floor((box[j][r] - G.lo[r]) * G.inv[r])));
        c1[r] = std::max(0, std::min(G.n[r] - 1, (int)std::floor((box[j][3 + r] - G.lo[r]) * G.inv[r])));
      }
      for (int k = c0[2]; k <= c1[2]; k++)
        for (int jj = c0[1]; jj <= c1[1]; jj++)
          for (int i = c0[0]; i <= c1[0]; i++) lists[(k * G.n[1] + jj) * G.n[0] + i].push_back(g->children[N.first + j]);
    }
    for (int q = 0; q < ncell; q++) {
      g->cells.push_back((int32_t)g->list.size());
      g->list.insert(g->list.end(), lists[q].begin(), lists[q].end());
      g->cells.push_back((int32_t)g->list.size());
    }
    N.grid = (int)g->grids.size();
    g->grids.push_back(G);
    if (N.count >= kWalk32Min) g->walk32 = true;
  }
}

// The plain records of nav_cull.cuh.
static void build_cull(gv_geom* g) {
  g->cull.resize(g->nnodes);
  for (int v = 0; v < g->nnodes; v++) {
    const NodeD& N = g->nodes[v];
    const Desc& h = g->solids[N.desc];
    Cull& C = g->cull[v];
    std::memset(&C, 0, sizeof(C));
    for (int i = 0; i < 9; i++) C.R[i] = (float)N.R[i];
    double mag = 0;
    for (int i = 0; i < 3; i++) {
      C.t[i] = (float)N.t[i];
      C.e[i] = (float)h.ext[i];
      mag += std::fabs(N.t[i]) + h.ext[i];
    }
    C.margin = (float)(1e-6 + 4e-6 * mag);
    C.solid = N.desc;
    C.family = h.type == kBox ? 0 : h.type == kTrd || h.type == kTrap ? 1 : h.type == kTube ? 2 : 3;
    if (h.type == kBool || (h.flags & kFp64Only)) C.tag = kCullNever;
    else if (h.type == kBox) C.tag = kCullBox;
    else if (h.type == kTube && !(h.flags & kHasPhi)) C.tag = kCullTube;
    else C.tag = kCullOther;
    if (C.tag == kCullNever && N.parent >= 0) {
      g->nodes[N.parent].never = 1;
      g->never = true;
    }
    if (C.tag == kCullTube && (h.inner & 1u)) C.rmin = (float)h.in[0].b;  // a = 0: the radius
  }
}

// Device memory for the safety lists of `cells` cells.  The lists only spare a safety the scan of all
// daughters, so a geometry that finds no memory for them (false) does without; e: any other error.
static bool alloc_safe(gv_geom* g, int64_t cells, cudaError_t& e) {
  e = cudaMalloc(&g->d_safe, sizeof(SafeEnt) * kSafeList * (size_t)cells);
  if (e == cudaSuccess) e = cudaMalloc(&g->d_safe_cut, sizeof(float) * (size_t)cells);
  if (e != cudaErrorMemoryAllocation) return e == cudaSuccess;
  cudaGetLastError();  // leave no error behind for the launch checks
  e = cudaSuccess;
  if (g->d_safe) cudaFree(g->d_safe);
  g->d_safe = nullptr;
  g->d_safe_cut = nullptr;
  for (GridD& G : g->grids) G.safe = -1;
  return false;
}

}  // namespace gv

static gv::Vox vox_of(const gv_geom* g) {
  if (!g->use_vox || !g->d_grids) return gv::Vox{nullptr, nullptr, nullptr, nullptr, nullptr};
  return gv::Vox{g->d_grids, g->d_cells, g->d_list, g->d_safe, g->d_safe_cut};
}

static gv::Geo geo_of(const gv_geom* g) {
  return gv::Geo{g->d_nodes, g->d_children, g->d_solids, g->d_cull, g->nnodes, vox_of(g)};
}

extern "C" {

gv_status gv_geom_create(int32_t nnodes, const gv_solid* const* node_solid, const int32_t* parent, const double* R,
                         const double* t, gv_geom** out) {
  if (!out) return set_error(GV_ERR_INVALID_ARG, "geom: out handle pointer is NULL");
  if (nnodes <= 0 || !node_solid || !parent || !R || !t) return set_error(GV_ERR_INVALID_ARG, "geom: empty or NULL table");
  if (parent[0] != -1) return set_error(GV_ERR_INVALID_ARG, "geom: node 0 must be the world (parent -1)");
  for (int i = 1; i < nnodes; i++)
    if (parent[i] < 0 || parent[i] >= i) return set_error(GV_ERR_INVALID_ARG, "geom: parents must precede children");
  for (int i = 0; i < nnodes; i++)
    if (!node_solid[i]) return set_error(GV_ERR_INVALID_ARG, "geom: NULL solid");
  for (int i = 0; i < 12 * nnodes; i++)
    if (!std::isfinite(i < 9 * nnodes ? R[i] : t[i - 9 * nnodes])) return set_error(GV_ERR_INVALID_ARG, "geom: non-finite placement");
  gv_geom* g = new (std::nothrow) gv_geom;
  if (!g) return set_error(GV_ERR_OUT_OF_MEMORY, "host allocation failed");
  g->nnodes = nnodes;
  g->nodes.resize(nnodes);
  std::vector<const gv_solid*> uniq;
  for (int v = 0; v < nnodes; v++) {
    NodeD& N = g->nodes[v];
    std::memset(&N, 0, sizeof(N));
    const double* L = R + 9 * v;
    const double* tl = t + 3 * v;
    if (parent[v] < 0) {
      for (int k = 0; k < 9; k++) N.R[k] = L[k];
      for (int k = 0; k < 3; k++) N.t[k] = tl[k];
    } else {  // compose with the parent's global placement (binary64, no fused multiply-add)
      const NodeD& P = g->nodes[parent[v]];
      for (int i = 0; i < 3; i++) {
        for (int j = 0; j < 3; j++)
          N.R[3 * i + j] = (P.R[3 * i + 0] * L[0 * 3 + j] + P.R[3 * i + 1] * L[1 * 3 + j]) + P.R[3 * i + 2] * L[2 * 3 + j];
        N.t[i] = ((P.R[3 * i + 0] * tl[0] + P.R[3 * i + 1] * tl[1]) + P.R[3 * i + 2] * tl[2]) + P.t[i];
      }
    }
    for (int k = 0; k < 9; k++) split_f(N.R[k], N.Rh[k], N.Rl[k]);
    for (int k = 0; k < 3; k++) split_f(N.t[k], N.th[k], N.tl[k]);
    N.parent = parent[v];
    int idx = -1;
    for (size_t k = 0; k < uniq.size(); k++)
      if (uniq[k] == node_solid[v]) { idx = (int)k; break; }
    if (idx < 0) { idx = (int)uniq.size(); uniq.push_back(node_solid[v]); }
    N.desc = idx;
  }
  // daughters in increasing node index
  std::vector<int> cnt(nnodes, 0);
  for (int v = 1; v < nnodes; v++) cnt[parent[v]]++;
  int acc = 0;
  for (int v = 0; v < nnodes; v++) { g->nodes[v].first = acc; g->nodes[v].count = cnt[v]; acc += cnt[v]; }
  g->children.assign(std::max(acc, 1), 0);
  std::vector<int> fill(nnodes, 0);
  for (int v = 1; v < nnodes; v++) {
    const int p = parent[v];
    g->children[g->nodes[p].first + fill[p]++] = v;
  }
  g->nsolids = (int)uniq.size();
  const int nrec = table_size(uniq.data(), g->nsolids);  // booleans carry their components along
  for (const gv_solid* u : uniq) g->solids.push_back(u->h);  // host copies for the grid builder
  build_grids(g);
  build_cull(g);
  int64_t safe_cells = 0;  // cells with a safety list
  for (int v = 0; v < nnodes; v++) {
    if (g->nodes[v].grid < 0) continue;
    GridD& G = g->grids[g->nodes[v].grid];
    const int64_t cells = (int64_t)G.n[0] * G.n[1] * G.n[2];
    if (g->nodes[v].count < kWalk32Min || g->nodes[v].count > kSafeDaughters || cells > kSafeCells || safe_cells + cells > kSafeTotal) continue;
    G.safe = (int32_t)safe_cells;
    safe_cells += cells;
  }
  cudaError_t e = cudaGetDevice(&g->device);
  if (e == cudaSuccess) e = cudaMalloc(&g->d_nodes, sizeof(NodeD) * nnodes);
  if (e == cudaSuccess) e = cudaMalloc(&g->d_children, sizeof(int32_t) * g->children.size());
  if (e == cudaSuccess) e = cudaMalloc(&g->d_cull, sizeof(Cull) * nnodes);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_cull, g->cull.data(), sizeof(Cull) * nnodes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&g->d_solids, sizeof(Desc) * nrec);
  if (e == cudaSuccess) g->solids = table_records(uniq.data(), g->nsolids, g->d_solids);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_nodes, g->nodes.data(), sizeof(NodeD) * nnodes, cudaMemcpyHostToDevice);
  if (e == cudaSuccess)
    e = cudaMemcpy(g->d_children, g->children.data(), sizeof(int32_t) * g->children.size(), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(g->d_solids, g->solids.data(), sizeof(Desc) * nrec, cudaMemcpyHostToDevice);
  if (e == cudaSuccess && !g->grids.empty()) {
    e = cudaMalloc(&g->d_grids, sizeof(GridD) * g->grids.size());
    if (e == cudaSuccess) e = cudaMalloc(&g->d_cells, sizeof(int32_t) * g->cells.size());
    if (e == cudaSuccess) e = cudaMalloc(&g->d_list, sizeof(int32_t) * std::max<size_t>(g->list.size(), 1));
    if (e == cudaSuccess && safe_cells > 0 && !alloc_safe(g, safe_cells, e)) safe_cells = 0;
    if (e == cudaSuccess) e = cudaMemcpy(g->d_grids, g->grids.data(), sizeof(GridD) * g->grids.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess) e = cudaMemcpy(g->d_cells, g->cells.data(), sizeof(int32_t) * g->cells.size(), cudaMemcpyHostToDevice);
    if (e == cudaSuccess && !g->list.empty())
      e = cudaMemcpy(g->d_list, g->list.data(), sizeof(int32_t) * g->list.size(), cudaMemcpyHostToDevice);
  }
  if (e == cudaSuccess && safe_cells > 0) {
    for (int v = 0; e == cudaSuccess && v < nnodes; v++) {
      if (g->nodes[v].grid < 0 || g->grids[g->nodes[v].grid].safe < 0) continue;
      const GridD& G = g->grids[g->nodes[v].grid];
      k_safe_lists<<<G.n[0] * G.n[1] * G.n[2], 256, sizeof(float) * g->nodes[v].count>>>(geo_of(g), v, g->d_safe, g->d_safe_cut);
      e = cudaGetLastError();
    }
    if (e == cudaSuccess) e = cudaStreamSynchronize(nullptr);
  }
  if (e != cudaSuccess) {
    gv_geom_destroy(g);
    return e == cudaErrorMemoryAllocation ? set_error(GV_ERR_OUT_OF_MEMORY, "geom: cudaMalloc failed") : cuda_error(e, "geom upload");
  }
  *out = g;
  return GV_OK;
}

void gv_geom_destroy(gv_geom* g) {
  if (!g) return;
  if (g->d_nodes) cudaFree(g->d_nodes);
  if (g->d_children) cudaFree(g->d_children);
  if (g->d_solids) cudaFree(g->d_solids);
  if (g->d_cull) cudaFree(g->d_cull);
  if (g->d_grids) cudaFree(g->d_grids);
  if (g->d_cells) cudaFree(g->d_cells);
  if (g->d_list) cudaFree(g->d_list);
  if (g->d_safe) cudaFree(g->d_safe);
  if (g->d_safe_cut) cudaFree(g->d_safe_cut);
  delete g;
}

gv_status gv_geom_set_voxels(gv_geom* g, int32_t enable) {
  if (!g) return set_error(GV_ERR_INVALID_ARG, "geom: NULL geometry");
  g->use_vox = enable != 0;
  return GV_OK;
}

int32_t gv_geom_voxel_count(const gv_geom* g) { return g ? (int32_t)g->grids.size() : 0; }

int32_t gv_geom_node_count(const gv_geom* g) { return g ? g->nnodes : 0; }

static cudaError_t launch_nav_pool(const gv_geom* g, const gv::NavArgs& a, int64_t blocks, const uint32_t* wl,
                                   const unsigned long long* cnt, cudaStream_t st) {
  const int bytes = (int)sizeof(gv::StepPool<gv::kNavSlots>);
  const cudaError_t e = cudaFuncSetAttribute(gv::k_nav_pool, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (e != cudaSuccess) return e;
  gv::k_nav_pool<<<(unsigned)blocks, gv::kNavThreads, bytes, st>>>(geo_of(g), a, wl, cnt);
  return cudaGetLastError();
}

gv_status gv_nav_locate(const gv_geom* g, const gv_tracks* t, int32_t* node, void* stream) {
  const gv::Range range("gv_nav_locate");
  if (!g || !t) return set_error(GV_ERR_INVALID_ARG, "locate: NULL geometry or tracks");
  if (t->n < 0) return set_error(GV_ERR_INVALID_ARG, "locate: negative track count");
  if (t->n == 0) return GV_OK;
  if (!t->x || !t->y || !t->z || !node) return set_error(GV_ERR_INVALID_ARG, "locate: NULL array");
  int64_t blocks = std::min<int64_t>((t->n + 255) / 256, (int64_t)sm_count() * 8);
  k_locate32<<<(unsigned)blocks, 256, 0, (cudaStream_t)stream>>>(geo_of(g), t->x, t->y, t->z, node, t->n);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GV_OK : cuda_error(e, "locate launch");
}

gv_status gv_nav_step(const gv_geom* g, const gv_tracks* t, const int32_t* node, gv_precision prec, double* step,
                      double* safety, int32_t* next, gv_workspace* ws, void* stream) {
  const gv::Range range("gv_nav_step");
  if (!g || !t) return set_error(GV_ERR_INVALID_ARG, "nav: NULL geometry or tracks");
  if (prec != GV_FP64 && prec != GV_FP32_REFINE) return set_error(GV_ERR_INVALID_ARG, "unknown precision");
  if (t->n < 0) return set_error(GV_ERR_INVALID_ARG, "nav: negative track count");
  if (t->n == 0) return GV_OK;
  if (!t->x || !t->y || !t->z || !t->dx || !t->dy || !t->dz || !node || !step || !next)
    return set_error(GV_ERR_INVALID_ARG, "nav: NULL array");
  const void* ptrs[8] = {t->x, t->y, t->z, t->dx, t->dy, t->dz, step, safety};  // safety may be NULL
  for (int i = 0; i < 8; i++)
    if ((uintptr_t)ptrs[i] & 7u) return set_error(GV_ERR_INVALID_ARG, "nav: arrays must be 8-byte aligned");
  NavArgs a{t->x, t->y, t->z, t->dx, t->dy, t->dz, node, step, safety, next, t->n};
  cudaStream_t st = (cudaStream_t)stream;
  const int sms = sm_count();
  if (prec == GV_FP64) {
    const cudaError_t e = launch_nav_pool(g, a, std::min<int64_t>((t->n + 7) / 8, sms), nullptr, nullptr, st);
    if (e != cudaSuccess) return cuda_error(e, "nav launch");
  } else {
    if (!ws) return set_error(GV_ERR_INVALID_ARG, "nav: GV_FP32_REFINE needs a workspace");
    if (ws->cap < t->n) return set_error(GV_ERR_OUT_OF_MEMORY, "nav: workspace smaller than the basket");
    ws->fused_blocks = 0;  // this pass counts its refinements in the counter
    cudaError_t e = cudaMemsetAsync(ws->counter, 0, sizeof(unsigned long long), st);
    if (e != cudaSuccess) return cuda_error(e, "nav: counter reset");
    const Vox vox = vox_of(g);
    const bool brief = t->n <= kShortBasket;
    const bool walk = vox.grids && g->walk32;
    if (walk || (brief && !g->never && !g->walk32)) {
      const int64_t per_block = 256 / kLanes;
      const int64_t blocks = std::min<int64_t>((t->n + per_block - 1) / per_block, (int64_t)sms * 8);
      (walk ? k_nav_fp32<true> : k_nav_fp32<false>)<<<(unsigned)blocks, 256, 0, st>>>(
          g->d_nodes, g->d_children, g->d_solids, g->d_cull, g->nnodes, a, ws->idx, ws->counter, vox);
    } else {
      const int64_t blocks = std::min<int64_t>((t->n + 255) / 256, (int64_t)sms * 2);
      k_nav_scan32<<<(unsigned)blocks, 256, 0, st>>>(g->d_nodes, g->d_children, g->d_solids, g->d_cull, g->nnodes, a,
                                                     ws->idx, ws->counter, vox);
    }
    if (brief) k_nav_exact<<<(unsigned)std::min<int64_t>(t->n, (int64_t)sms * 4), 32, 0, st>>>(geo_of(g), a, ws->idx, ws->counter);
    else e = launch_nav_pool(g, a, sms, ws->idx, ws->counter, st);
    if (e != cudaSuccess) return cuda_error(e, "nav launch");
  }
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GV_OK : cuda_error(e, "nav launch");
}

gv_status gv_transport(const gv_geom* g, const gv_tracks* t, const int32_t* node0, const int32_t* node_material,
                       const double* sigma_n, int32_t nmat, const double* xi, int32_t kmax, gv_precision prec,
                       const gv_transport_out* out, void* stream) {
  const gv::Range range("gv_transport");
  if (!g || !t || !out) return set_error(GV_ERR_INVALID_ARG, "transport: NULL geometry, tracks or outputs");
  if (t->n < 0) return set_error(GV_ERR_INVALID_ARG, "transport: negative track count");
  if (kmax < 1 || nmat < 1) return set_error(GV_ERR_INVALID_ARG, "transport: kmax and nmat must be >= 1");
  if (prec != GV_FP64 && prec != GV_FP32_REFINE) return set_error(GV_ERR_INVALID_ARG, "unknown precision");
  if (t->n == 0) return GV_OK;
  if (!t->x || !t->y || !t->z || !t->dx || !t->dy || !t->dz || !node0 || !node_material || !sigma_n || !xi ||
      !out->reason || !out->steps || !out->x || !out->y || !out->z || !out->path || !out->last || !out->tie)
    return set_error(GV_ERR_INVALID_ARG, "transport: NULL array");
  const void* ptrs[11] = {t->x, t->y, t->z, t->dx, t->dy, t->dz, sigma_n, xi, out->x, out->y, out->path};
  for (int i = 0; i < 11; i++)
    if ((uintptr_t)ptrs[i] & 7u) return set_error(GV_ERR_INVALID_ARG, "transport: arrays must be 8-byte aligned");
  if ((uintptr_t)out->z & 7u) return set_error(GV_ERR_INVALID_ARG, "transport: arrays must be 8-byte aligned");
  TransportArgs a{t->x, t->y, t->z, t->dx, t->dy, t->dz, node0, node_material, sigma_n, xi, kmax, nmat, g->nnodes,
                  out->reason, out->steps, out->x, out->y, out->z, out->path, out->last, out->tie, t->n};
  // One block per SM: each owns a contiguous range of tracks and keeps its pool full from it, so it
  // drains (slots empty while its last tracks finish) once per range.
  const int sms = sm_count();
  const int64_t blocks = std::min<int64_t>((t->n + 31) / 32, sms);
  const int bytes = (int)sizeof(FlightPool);
  const cudaError_t ea = cudaFuncSetAttribute(k_transport, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
  if (ea != cudaSuccess) return cuda_error(ea, "transport launch");
  k_transport<<<(unsigned)blocks, kFlightThreads, bytes, (cudaStream_t)stream>>>(geo_of(g), a);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? GV_OK : cuda_error(e, "transport launch");
}

}  // extern "C"
