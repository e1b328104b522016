// query_fp64.cu -- the plain binary64 query pass.  Primitive solids take the ranked pass
// (k_query_rank64, k_query_rank64_short, k_rank_walk): binary32 decides which constraint and which
// crossing give the results, binary64 evaluates those; larger baskets of booleans of solids with at most
// two z-planes likewise (k_query_bool_rank).  The rest is evaluated whole, one thread per track: other and
// short booleans in index order (k_query_fp64); solids with features finer than binary32 resolves in tiles
// ordered by work class when the basket gives every SM a 2048-track tile (k_query_fp64_tiles: the FP64 pipe
// spends the same on a warp instruction whatever its active lanes, so warps of one class run fewer
// instructions), else in index order.  Per track the bits are the same in every one of them.
#include "bool_rank.cuh"
#include "gv_debug.cuh"
#include "gv_internal.h"
#include "solid_fp64.cuh"
#include "rank_fp64.cuh"
#include "work_class.cuh"

namespace gv {

// Copy a descriptor into shared memory with 16-byte loads.
__device__ __forceinline__ void stage_desc(Desc& dst, const Desc* __restrict__ src) {
  const int4* s = reinterpret_cast<const int4*>(src);
  int4* d = reinterpret_cast<int4*>(&dst);
  for (int i = threadIdx.x; i < (int)(sizeof(Desc) / 16); i += blockDim.x) d[i] = s[i];
}

template <int FAMILY>
__global__ void __launch_bounds__(256) k_query_fp64(const Desc* __restrict__ desc, QueryArgs a) {
  __shared__ Desc S;
  stage_desc(S, desc);
  __syncthreads();
  const unsigned want = (a.inside ? f64::kWantCode : 0u) | (a.din ? f64::kWantDin : 0u) |
                        (a.dout ? f64::kWantDout : 0u) | (a.sin ? f64::kWantSin : 0u) |
                        (a.sout ? f64::kWantSout : 0u);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += stride) {
    f64::Track T{a.x[i], a.y[i], a.z[i], 0, 0, 0};
    if (want & (f64::kWantDin | f64::kWantDout)) {
      T.u = a.u[i]; T.v = a.v[i]; T.w = a.w[i];
      GV_DCHECK(dbg_unit(T.u, T.v, T.w), kDbgDirection, i);
    }
    f64::Result R;
    if (FAMILY == 0) f64::box_query(S, T, want, R);
    else if (FAMILY == 1) f64::planar_query(S, T, want, R);
    else if (FAMILY == 4) f64::bool_query(S, T, want, R);
    else f64::pcon_query(S, T, want, R);
    if (a.inside) a.inside[i] = (int8_t)R.code;
    if (a.din) a.din[i] = R.din;
    if (a.dout) a.dout[i] = R.dout;
    if (a.sin) a.sin[i] = R.sin;
    if (a.sout) a.sout[i] = R.sout;
  }
}

// The binary64 pass in tiles ordered by work class: a block takes a tile of 256 * ITEMS
// consecutive tracks, classifies them (f32::track_class, from the high parts; the reads bring the
// tile into the caches), orders the tile's offsets by class in shared memory (a count, a scan
// and a scatter) and evaluates them in that order.
template <int FAMILY, int ITEMS>
__global__ void __launch_bounds__(256) k_query_fp64_tiles(const Desc* __restrict__ desc, QueryArgs a) {
  constexpr int NT = 256, TILE = NT * ITEMS;
  constexpr uint32_t NC = f32::kClasses;
  __shared__ Desc S;
  __shared__ uint16_t ord[TILE];
  __shared__ uint8_t cls[TILE];
  __shared__ unsigned cnt[NC], cur[NC];
  stage_desc(S, desc);
  __syncthreads();
  const unsigned want = (a.inside ? f64::kWantCode : 0u) | (a.din ? f64::kWantDin : 0u) |
                        (a.dout ? f64::kWantDout : 0u) | (a.sin ? f64::kWantSin : 0u) |
                        (a.sout ? f64::kWantSout : 0u);
  const bool dirs = want & (f64::kWantDin | f64::kWantDout);
  const uint2 *X = reinterpret_cast<const uint2*>(a.x), *Y = reinterpret_cast<const uint2*>(a.y),
              *Z = reinterpret_cast<const uint2*>(a.z), *Ux = reinterpret_cast<const uint2*>(a.u),
              *Uy = reinterpret_cast<const uint2*>(a.v), *Uz = reinterpret_cast<const uint2*>(a.w);
  const int tid = threadIdx.x;
  for (int64_t t0 = (int64_t)blockIdx.x * TILE; t0 < a.n; t0 += (int64_t)gridDim.x * TILE) {
    const int len = a.n - t0 < TILE ? (int)(a.n - t0) : TILE;
    if (tid < (int)NC) cnt[tid] = 0u;
    __syncthreads();
    for (int j = tid; j < len; j += NT) {
      const int64_t i = t0 + j;
      bool bad = false;  // a value outside the binary32 range only lands in some class
      const float x = f32::trunc_hi(__ldg(X + i), bad), y = f32::trunc_hi(__ldg(Y + i), bad),
                  z = f32::trunc_hi(__ldg(Z + i), bad);
      float u = 0.f, v = 0.f, w = 0.f;
      if (dirs) {
        u = f32::trunc_hi(__ldg(Ux + i), bad);
        v = f32::trunc_hi(__ldg(Uy + i), bad);
        w = f32::trunc_hi(__ldg(Uz + i), bad);
      }
      const uint32_t c = f32::track_class(S, x, y, z, u, v, w, dirs);
      cls[j] = (uint8_t)c;
      atomicAdd(&cnt[c], 1u);
    }
    __syncthreads();
    if (tid == 0) {
      unsigned run = 0;
      for (uint32_t q = 0; q < NC; q++) {
        cur[q] = run;
        run += cnt[q];
      }
    }
    __syncthreads();
    for (int j = tid; j < len; j += NT) ord[atomicAdd(&cur[cls[j]], 1u)] = (uint16_t)j;
    __syncthreads();
    for (int p = tid; p < len; p += NT) {
      const int64_t i = t0 + ord[p];
      f64::Track T{a.x[i], a.y[i], a.z[i], 0, 0, 0};
      if (dirs) {
        T.u = a.u[i]; T.v = a.v[i]; T.w = a.w[i];
        GV_DCHECK(dbg_unit(T.u, T.v, T.w), kDbgDirection, i);
      }
      f64::Result R;
      if (FAMILY == 0) f64::box_query(S, T, want, R);
      else if (FAMILY == 1) f64::planar_query(S, T, want, R);
      else f64::pcon_query(S, T, want, R);
      if (a.inside) a.inside[i] = (int8_t)R.code;
      if (a.din) a.din[i] = R.din;
      if (a.dout) a.dout[i] = R.dout;
      if (a.sin) a.sin[i] = R.sin;
      if (a.sout) a.sout[i] = R.sout;
    }
    __syncthreads();  // the tile's shared arrays are reused by the next tile
  }
}

// A track whose ranking left its code open.
template <int FAMILY>
static __device__ __noinline__ void query_open(const Desc& S, const QueryArgs& a, int64_t i, unsigned want) {
  f64::Track T{a.x[i], a.y[i], a.z[i], 0, 0, 0};
  const bool dirs = want & (f64::kWantDin | f64::kWantDout);
  if (dirs) { T.u = a.u[i]; T.v = a.v[i]; T.w = a.w[i]; }
  const f32::TrackF F = f32::load_track<(FAMILY >= 2)>(
      reinterpret_cast<const uint2*>(a.x), reinterpret_cast<const uint2*>(a.y), reinterpret_cast<const uint2*>(a.z),
      reinterpret_cast<const uint2*>(a.u), reinterpret_cast<const uint2*>(a.v), reinterpret_cast<const uint2*>(a.w), i, dirs);
  f64::Result R;
  f64::query_refined<FAMILY>(S, T, F, want, R);
  if (a.inside) a.inside[i] = (int8_t)R.code;
  if (a.din) a.din[i] = R.din;
  if (a.dout) a.dout[i] = R.dout;
  if (a.sin) a.sin[i] = R.sin;
  if (a.sout) a.sout[i] = R.sout;
}

// The ranked binary64 pass (rank_fp64.cuh) in tiles of 256 * ITEMS consecutive tracks: a block
// ranks its tile's tracks in binary32 (one verdict word per track in shared memory), orders them by
// the binary64 work their verdict asks for, and evaluates that work in this order, so that the FP64
// pipe sees full warps.  While one resident block evaluates, others rank: the two halves use
// different pipes.  A track without a certain verdict (its code within about 1e-11 mm of the band's
// edges) goes on the block's list, which is evaluated when 256 have gathered and at the end: its code in
// binary64, the rest ranked.
// Measured (GB300, all five queries): cone, 2^20 tracks, 500 -> 179 us; 8-plane polycone, 4 M tracks,
// 6876 -> 1274 us in this kernel alone (before: every candidate in binary64, tiles ordered by class).
// FP64 warp instructions per 32 tracks: cone 226 -> 42, polycone 859 -> 45; issue 41% and FP64 46% busy
// (cone): bound by latency at 24 warps per SM.  Three blocks of 256 threads (80 registers) against two
// (128): cone 179 against 186 us; rows of 256 the other way round.
constexpr int kOpenFlush = 256;
constexpr int kRankThreads = 256, kRankBlocks = 3;
constexpr uint32_t kOpenVerdict = 0xFFFFFFFFu;
// STORED: the verdicts are read from `stored`, where an earlier launch left them.
template <int FAMILY, int ITEMS, bool STORED = false>
__global__ void __launch_bounds__(kRankThreads, ITEMS == 1 ? 512 / kRankThreads : kRankBlocks)
    k_query_rank64(const Desc* __restrict__ desc, QueryArgs a, const uint2* stored) {
  constexpr int NT = kRankThreads, TILE = NT * ITEMS;
  constexpr uint32_t NC = f64::kRankClasses;
  __shared__ Desc S;
  __shared__ uint32_t ver[TILE];
  __shared__ uint16_t ord[TILE];
  __shared__ int64_t open[TILE + kOpenFlush];
  __shared__ unsigned cnt[NC], nopen;
  stage_desc(S, desc);
  const int tid = threadIdx.x;
  const unsigned lane = tid & 31u;
  if (tid == 0) nopen = 0u;
  const unsigned want = (a.inside ? f64::kWantCode : 0u) | (a.din ? f64::kWantDin : 0u) |
                        (a.dout ? f64::kWantDout : 0u) | (a.sin ? f64::kWantSin : 0u) |
                        (a.sout ? f64::kWantSout : 0u);
  const bool dirs = want & (f64::kWantDin | f64::kWantDout);
  const uint2 *X = reinterpret_cast<const uint2*>(a.x), *Y = reinterpret_cast<const uint2*>(a.y),
              *Z = reinterpret_cast<const uint2*>(a.z), *Ux = reinterpret_cast<const uint2*>(a.u),
              *Uy = reinterpret_cast<const uint2*>(a.v), *Uz = reinterpret_cast<const uint2*>(a.w);
  for (int64_t t0 = (int64_t)blockIdx.x * TILE; t0 < a.n; t0 += (int64_t)gridDim.x * TILE) {
    const int len = a.n - t0 < TILE ? (int)(a.n - t0) : TILE;
    if (tid < (int)NC) cnt[tid] = 0u;
    __syncthreads();
    for (int j = tid; j < len; j += NT) {
      const int64_t i = t0 + j;
      uint32_t V;
      if constexpr (STORED) {
        V = stored[i].x;
      } else {
        const f32::TrackF T = f32::load_track<(FAMILY >= 2)>(X, Y, Z, Ux, Uy, Uz, i, dirs);
        GV_DCHECK(!dirs || dbg_unit(a.u[i], a.v[i], a.w[i]), kDbgDirection, i);
        f32::R32 R;
        f64::rank32<FAMILY>(S, T, want, R);
        V = R.flag ? kOpenVerdict : R.rank;
      }
      ver[j] = V;
      if (V == kOpenVerdict) {
        open[atomicAdd(&nopen, 1u)] = i;
      } else {
        atomicAdd(&cnt[f64::rank_class<FAMILY>(f64::Verdict{V})], 1u);
      }
    }
    __syncthreads();
    const unsigned gathered = nopen;
    unsigned ranked = 0;
    if (tid < 32) {  // exclusive sums of the class counts
      const unsigned c = lane < NC ? cnt[lane] : 0u;
      unsigned run = c;
      for (int o = 1; o < 8; o <<= 1) {
        const unsigned v = __shfl_up_sync(0xffffffffu, run, o);
        if ((int)lane >= o) run += v;
      }
      __syncwarp();
      if (lane < NC) cnt[lane] = run - c;
    }
    __syncthreads();
    for (int j = tid; j < len; j += NT)
      if (ver[j] != kOpenVerdict) ord[atomicAdd(&cnt[f64::rank_class<FAMILY>(f64::Verdict{ver[j]})], 1u)] = (uint16_t)j;
    __syncthreads();
    ranked = cnt[NC - 1];
    for (unsigned p = tid; p < ranked; p += NT) {
      const int j = ord[p];
      const int64_t i = t0 + j;
      f64::Track T{a.x[i], a.y[i], a.z[i], 0, 0, 0};
      if (dirs) { T.u = a.u[i]; T.v = a.v[i]; T.w = a.w[i]; }
      f64::Result R;
      f64::query_ranked<FAMILY>(S, T, f64::Verdict{ver[j]}, R);
      if (a.inside) a.inside[i] = (int8_t)R.code;
      if (a.din) a.din[i] = R.din;
      if (a.dout) a.dout[i] = R.dout;
      if (a.sin) a.sin[i] = R.sin;
      if (a.sout) a.sout[i] = R.sout;
    }
    if (gathered >= (unsigned)kOpenFlush) {
      for (unsigned q = tid; q < gathered; q += NT) query_open<FAMILY>(S, a, open[q], want);
      __syncthreads();
      if (tid == 0) nopen = 0u;
    }
    __syncthreads();  // the tile's shared arrays are reused by the next tile
  }
  __syncthreads();
  for (unsigned q = tid; q < nopen; q += NT) query_open<FAMILY>(S, a, open[q], want);
}

// Booleans whose components rank (bool_rank.cuh), in tiles ordered by the binary64 work of the verdicts as
// in k_query_rank64 (ITEMS tracks per thread).  A track without a certain verdict (surface starts of a
// component above all) goes on the block's list, evaluated whole.
// Measured (box minus tube segment, 2^20 tracks, all five queries): 1213 -> 290 us (before: every piece of
// both components in binary64, 594 FP64 warp instructions per 32 tracks); ranked but in index order
// 365 us (139 FP64 warp instructions).  The ranking inlined: 296 us (spills).
// PARTS: every block takes an equal, contiguous part of the basket instead of tiles in turn.  Up to three
// tiles per block this evens out the last round (400000 tracks 151 -> 127 us, 700000 215 -> 187 us); beyond, or
// without distances in short rows, tiles in turn are as even and up to 8% faster.
template <int ITEMS, bool PARTS>
__global__ void __launch_bounds__(256, 2) k_query_bool_rank(const Desc* __restrict__ desc, QueryArgs a) {
  constexpr int TILE = 256 * ITEMS;
  constexpr uint32_t NC = f64::kBoolClasses;
  __shared__ Desc S, A, C;
  __shared__ uint32_t ver[TILE];
  __shared__ uint16_t ord[TILE];
  __shared__ int64_t open[TILE + kOpenFlush];
  __shared__ unsigned cnt[NC], nopen;
  const int tid = threadIdx.x;
  stage_desc(S, desc);
  stage_desc(A, desc->parts);
  stage_desc(C, desc->parts + 1);
  if (tid == 0) nopen = 0u;
  const unsigned want = (a.inside ? f64::kWantCode : 0u) | (a.din ? f64::kWantDin : 0u) |
                        (a.dout ? f64::kWantDout : 0u) | (a.sin ? f64::kWantSin : 0u) |
                        (a.sout ? f64::kWantSout : 0u);
  const bool dirs = want & (f64::kWantDin | f64::kWantDout);
  auto load = [&](int64_t i) {
    f64::Track T{a.x[i], a.y[i], a.z[i], 0, 0, 0};
    if (dirs) { T.u = a.u[i]; T.v = a.v[i]; T.w = a.w[i]; }
    return T;
  };
  auto store = [&](int64_t i, const f64::Result& R) {
    if (a.inside) a.inside[i] = (int8_t)R.code;
    if (a.din) a.din[i] = R.din;
    if (a.dout) a.dout[i] = R.dout;
    if (a.sin) a.sin[i] = R.sin;
    if (a.sout) a.sout[i] = R.sout;
  };
  auto flush = [&](unsigned count) {
    for (unsigned q = tid; q < count; q += 256) {
      f64::Result R;
      f64::bool_query(S, load(open[q]), want, R);
      store(open[q], R);
    }
  };
  // tiles in turn, or an equal, contiguous part of the basket
  const int64_t share = PARTS ? ((a.n + gridDim.x - 1) / gridDim.x + 31) / 32 * 32 : TILE;
  const int64_t end = PARTS ? min((int64_t)(blockIdx.x + 1) * share, a.n) : a.n;
  for (int64_t t0 = (int64_t)blockIdx.x * share; t0 < end; t0 += PARTS ? TILE : (int64_t)gridDim.x * TILE) {  // block-uniform
    const int len = end - t0 < TILE ? (int)(end - t0) : TILE;
    if (tid < (int)NC) cnt[tid] = 0u;
    __syncthreads();
    for (int j = tid; j < len; j += 256) {
      const f64::Track T = load(t0 + j);
      GV_DCHECK(!dirs || dbg_unit(T.u, T.v, T.w), kDbgDirection, t0 + j);
      uint32_t V;
      if (f64::bool_verdict(S, A, C, T, want, V)) {
        atomicAdd(&cnt[f64::bool_class(A, C, f64::BoolVerdict{V})], 1u);
      } else {
        V = kOpenVerdict;
        open[atomicAdd(&nopen, 1u)] = t0 + j;
      }
      ver[j] = V;
    }
    __syncthreads();
    const unsigned gathered = nopen;
    __syncthreads();
    if (tid == 0) {
      unsigned run = 0;
      for (uint32_t q = 0; q < NC; q++) {
        const unsigned c = cnt[q];
        cnt[q] = run;
        run += c;
      }
    }
    __syncthreads();
    for (int j = tid; j < len; j += 256)
      if (ver[j] != kOpenVerdict) ord[atomicAdd(&cnt[f64::bool_class(A, C, f64::BoolVerdict{ver[j]})], 1u)] = (uint16_t)j;
    __syncthreads();
    const int ranked = (int)cnt[NC - 1];
    for (int p = tid; p < ranked; p += 256) {
      const int j = ord[p];
      f64::Result R;
      f64::bool_evaluate(S, A, C, load(t0 + j), f64::BoolVerdict{ver[j]}, R);
      store(t0 + j, R);
    }
    if (gathered >= (unsigned)kOpenFlush) {
      flush(gathered);
      __syncthreads();
      if (tid == 0) nopen = 0u;
    }
    __syncthreads();
  }
  __syncthreads();
  flush(nopen);
}

// Baskets too short to fill the GPU: one track per thread, ranked and evaluated at once.  Latency bounds
// them, and a tile's barriers and second loads only add to it.  Measured (tube DistanceToOut, 50021 tracks):
// 44.6 us evaluating every candidate in binary64, 22.6 us here.
constexpr int kShortThreads = 128;
constexpr int64_t kRankWalkMin = 1 << 19;  // multi-section polycones: two launches from here on
template <int FAMILY>
__global__ void __launch_bounds__(kShortThreads) k_query_rank64_short(const Desc* __restrict__ desc, QueryArgs a) {
  __shared__ Desc S;
  const unsigned want = (a.inside ? f64::kWantCode : 0u) | (a.din ? f64::kWantDin : 0u) |
                        (a.dout ? f64::kWantDout : 0u) | (a.sin ? f64::kWantSin : 0u) |
                        (a.sout ? f64::kWantSout : 0u);
  const bool dirs = want & (f64::kWantDin | f64::kWantDout);
  const int64_t i = (int64_t)blockIdx.x * kShortThreads + threadIdx.x;
  f64::Track T{0, 0, 0, 0, 0, 0};
  if (i < a.n) {
    T.x = a.x[i]; T.y = a.y[i]; T.z = a.z[i];
    if (dirs) { T.u = a.u[i]; T.v = a.v[i]; T.w = a.w[i]; }
  }
  stage_desc(S, desc);
  __syncthreads();
  if (i >= a.n) return;
  GV_DCHECK(!dirs || dbg_unit(T.u, T.v, T.w), kDbgDirection, i);
  const f32::TrackF F = f64::split_track(T, dirs);
  f32::R32 r;
  f64::rank32<FAMILY>(S, F, want, r);
  f64::Result R;
  if (!r.flag) f64::query_ranked<FAMILY>(S, T, f64::Verdict{r.rank}, R);
  else f64::query_refined<FAMILY>(S, T, F, want, R);
  if (a.inside) a.inside[i] = (int8_t)R.code;
  if (a.din) a.din[i] = R.din;
  if (a.dout) a.dout[i] = R.dout;
  if (a.sin) a.sin[i] = R.sin;
  if (a.sout) a.sout[i] = R.sout;
}

// The ranking of multi-section polycones on its own, with lane refill as in the binary32 pass
// (k_query_walk): a warp keeps one track per lane and refills idle lanes from its rows of 32 tracks (the
// warps take rows in turn).  The verdict of track i is left in the low word of out[i].
// Measured (8-plane polycone, 4 M tracks): 957 us with the evaluation, against 1274 us ranking a tile's
// tracks in place, where a warp walks as long as its longest track (12.2 against 13.8 lanes, barriers).
// Below 2^19 tracks the second launch and its traffic cost more than that (300000: 143 against about 100 us
// one track per thread).  Blocks of 256 x 3: 976 us,
// 384 x 2: 962 us.
constexpr int kRankWalkThreads = 320, kRankWalkBlocks = 2;
__global__ void __launch_bounds__(kRankWalkThreads, kRankWalkBlocks) k_rank_walk(const Desc* __restrict__ desc, QueryArgs a,
                                                                                 uint2* out) {
  __shared__ Desc S;
  stage_desc(S, desc);
  __syncthreads();
  const unsigned want = (a.inside ? f64::kWantCode : 0u) | (a.din ? f64::kWantDin : 0u) |
                        (a.dout ? f64::kWantDout : 0u) | (a.sin ? f64::kWantSin : 0u) |
                        (a.sout ? f64::kWantSout : 0u);
  const uint2 *X = reinterpret_cast<const uint2*>(a.x), *Y = reinterpret_cast<const uint2*>(a.y),
              *Z = reinterpret_cast<const uint2*>(a.z), *Ux = reinterpret_cast<const uint2*>(a.u),
              *Uy = reinterpret_cast<const uint2*>(a.v), *Uz = reinterpret_cast<const uint2*>(a.w);
  const unsigned lane = threadIdx.x & 31u, below = (1u << lane) - 1u;
  const int64_t W = (int64_t)gridDim.x * (kRankWalkThreads / 32);
  const int64_t w = (int64_t)blockIdx.x * (kRankWalkThreads / 32) + (threadIdx.x >> 5);
  int64_t next = 0;  // next position in the warp's rows (warp-uniform)
  bool busy = false, more = w * 32 < a.n;
  int64_t i = 0;
  f32::TrackF T;
  f32::R32 R;
  f32::Walk K;
  while (true) {
    const unsigned idle = __ballot_sync(0xffffffffu, !busy);
    if (more && (__popc(idle) >= 16 || idle == 0xffffffffu)) {
      const int64_t seq = next + __popc(idle & below);
      const int64_t j = ((seq >> 5) * W + w) * 32 + (seq & 31);
      next += __popc(idle);
      more = ((next >> 5) * W + w) * 32 < a.n;
      if (!busy && j < a.n) {
        i = j;
        T = f32::load_track<true>(X, Y, Z, Ux, Uy, Uz, i, true);
        GV_DCHECK(dbg_unit(a.u[i], a.v[i], a.w[i]), kDbgDirection, i);
        R.flag = T.bad;
        R.rank = 0u;
        R.code = 1;
        R.din = R.dout = R.sin = R.sout = 0.f;
        R.te = R.se = 0.f;
        K.need_in = K.need_out = K.answered = K.live = false;
        if (!R.flag) busy = f32::pcon_begin<false, false, true>(S, T, want, R, K);
        if (!busy) out[i] = make_uint2(R.flag ? kOpenVerdict : R.rank, 0u);
      }
    }
    if (__ballot_sync(0xffffffffu, busy) == 0u) {
      if (!more) break;
      continue;
    }
    if (busy) {
      f32::pcon_step<false, false, true>(S, T, K);
      if (!K.live) {
        f32::pcon_end<true>(K, R);
        out[i] = make_uint2(R.flag ? kOpenVerdict : R.rank, 0u);
        busy = false;
      }
    }
  }
}

// Multi-section polycones in two launches: the walk leaves its verdicts in a distance result that the
// second launch overwrites.  Not when that array overlaps one that is read (an in-place call): the
// one-launch pass reads and writes each track in turn.
static bool overlaps(const void* p, const void* q, int64_t n) {
  const char *a = static_cast<const char*>(p), *b = static_cast<const char*>(q);
  return a < b + 8 * n && b < a + 8 * n;
}
static double* verdict_array(const QueryArgs& a) {
  double* out = a.dout ? a.dout : a.din;
  const double* in[6] = {a.x, a.y, a.z, a.u, a.v, a.w};
  for (const double* p : in)
    if (overlaps(out, p, a.n)) return nullptr;
  const double* other[4] = {a.din, a.dout, a.sin, a.sout};
  for (const double* p : other)
    if (p && p != out && overlaps(out, p, a.n)) return nullptr;
  if (a.inside && overlaps(out, a.inside, a.n)) return nullptr;
  return out;
}

template <int ITEMS>
static void launch_rank_stored(const gv_solid* s, const QueryArgs& a, const uint2* ver, int64_t cap, cudaStream_t stream) {
  const int64_t tiles = (a.n + kRankThreads * ITEMS - 1) / (kRankThreads * ITEMS);
  k_query_rank64<3, ITEMS, true><<<(unsigned)(tiles < cap ? tiles : cap), kRankThreads, 0, stream>>>(s->d, a, ver);
}
static void launch_rank_walk(const gv_solid* s, const QueryArgs& a, double* out, int sms, cudaStream_t stream) {
  const int64_t blocks = (a.n + kRankWalkThreads - 1) / kRankWalkThreads, cap = (int64_t)sms * kRankWalkBlocks;
  uint2* ver = reinterpret_cast<uint2*>(out);
  k_rank_walk<<<(unsigned)(blocks < cap ? blocks : cap), kRankWalkThreads, 0, stream>>>(s->d, a, ver);
  launch_rank_stored<4>(s, a, ver, (int64_t)sms * 3, stream);
}

template <int FAMILY, int ITEMS>
static void launch_rank64(const gv_solid* s, const QueryArgs& a, int sms, cudaStream_t stream) {
  static const int occ = [] {
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_query_rank64<FAMILY, ITEMS>, kRankThreads, 0) != cudaSuccess ||
        o < 1) {
      cudaGetLastError();
      o = 1;
    }
    return o;
  }();
  const int64_t tiles = (a.n + kRankThreads * ITEMS - 1) / (kRankThreads * ITEMS);
  const int64_t cap = (int64_t)sms * occ;
  k_query_rank64<FAMILY, ITEMS><<<(unsigned)(tiles < cap ? tiles : cap), kRankThreads, 0, stream>>>(s->d, a, nullptr);
}

// Tiles of 2048 tracks when every resident block gets four of them, of 1024 when it gets one; shorter
// baskets one track per thread, except the distances of tubes and cones from 1024 tracks per SM on, which
// gain from ordering already (tile of 256: measured, all five queries, against one track per thread: 50021
// tracks tube 25.9 / 24.9, cone 22.2 / 19.5, polycone 32.4 / 27.2 us; 200000 tracks tube 52.1 / 56.2, cone
// 46.7 / 48.1, box 16.2 / 12.4, trap 31.6 / 28.2 us; without distances 200003 tracks of the cone, codes
// 12.3 / 8.2, safeties 19.7 / 18.1 us).
template <int FAMILY>
static void launch_rank64(const gv_solid* s, const QueryArgs& a, int sms, cudaStream_t stream) {
  constexpr bool kOrdered = FAMILY == 2 || FAMILY == 4;
  const bool tiles = a.n >= (FAMILY == 3 ? kRankWalkMin : (int64_t)sms * 3 * 1024);
  if (tiles && a.n >= (int64_t)sms * 3 * 4 * 2048) {
    launch_rank64<FAMILY, 8>(s, a, sms, stream);
  } else if (tiles) {
    launch_rank64<FAMILY, 4>(s, a, sms, stream);
  } else {
    if constexpr (kOrdered) {
      if ((a.din || a.dout) && a.n >= (int64_t)sms * 1024) {
        launch_rank64<FAMILY, 1>(s, a, sms, stream);
        return;
      }
    }
    k_query_rank64_short<FAMILY><<<(unsigned)((a.n + kShortThreads - 1) / kShortThreads), kShortThreads, 0, stream>>>(s->d, a);
  }
}

template <int FAMILY, int ITEMS>
static int64_t tiles_grid(int64_t tiles, int sms) {
  // resident blocks per SM of the kernel (queried once: it depends only on the kernel and the GPU)
  static const int occ = [] {
    int o = 0;
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_query_fp64_tiles<FAMILY, ITEMS>, 256, 0) != cudaSuccess || o < 1) {
      cudaGetLastError();  // leave no error behind for the launch check
      o = 1;
    }
    return o;
  }();
  return tiles < (int64_t)sms * occ ? tiles : (int64_t)sms * occ;
}

// Booleans rank from more than this many tracks on.  Up to one block of 256 threads per SM a whole evaluation
// takes the time of one chain, and ranking only adds its own: five random booleans of 20000 tracks, all
// queries, ranked / whole 39 / 35, 43 / 43, 64 / 62, 51 / 49, 37 / 33 us; 40000 tracks 39 / 60, 43 / 78, 64 / 110, 53 / 84,
// 39 / 58 us.  Codes and safeties alone are shorter: 80000 tracks, codes 22.4 / 20.5, 22.5 / 18.5, 24.4 / 26.7 us,
// safeties 28.8 / 30.8, 26.3 / 29.8, 34.9 / 43.1 us; 400000 tracks, codes 53 / 64, 53 / 58, 57 / 86 us.
static int64_t bool_rank_min(const QueryArgs& a, int sms) {
  return (int64_t)sms * (a.din || a.dout ? 256 : a.sin || a.sout ? 512 : 1024);
}

cudaError_t launch_query_fp64(const gv_solid* s, const QueryArgs& a, cudaStream_t stream) {
  if (a.n == 0) return cudaSuccess;
  const int threads = 256;
  const int sms = sm_count();
  if (s->h.type != kBool && !(s->h.flags & kFp64Only)) {
    switch (s->h.type) {
      case kBox: launch_rank64<0>(s, a, sms, stream); break;
      case kTrd:
      case kTrap: launch_rank64<1>(s, a, sms, stream); break;
      case kTube: launch_rank64<2>(s, a, sms, stream); break;
      default:
        if (double* out = s->h.nz > 2 && (a.din || a.dout) && a.n >= kRankWalkMin ? verdict_array(a) : nullptr)
          launch_rank_walk(s, a, out, sms, stream);
        else if (s->h.nz > 2) launch_rank64<3>(s, a, sms, stream);
        else launch_rank64<4>(s, a, sms, stream);
        break;
    }
    return cudaGetLastError();
  }
  // tiles of 2048 tracks when the basket gives four of them to every resident block (two per SM),
  // else of 1024 (more tiles, fewer SMs idle in the last round); none below one 2048 tile per SM
  if (s->h.type != kBool && a.n >= (int64_t)sms * 2048) {
    const bool big = a.n >= (int64_t)sms * 2 * 4 * 2048;
    const int64_t tiles = big ? (a.n + 2047) / 2048 : (a.n + 1023) / 1024;
    switch (s->h.type) {
      case kBox:
        if (big) k_query_fp64_tiles<0, 8><<<(unsigned)tiles_grid<0, 8>(tiles, sms), 256, 0, stream>>>(s->d, a);
        else k_query_fp64_tiles<0, 4><<<(unsigned)tiles_grid<0, 4>(tiles, sms), 256, 0, stream>>>(s->d, a);
        break;
      case kTrd:
      case kTrap:
        if (big) k_query_fp64_tiles<1, 8><<<(unsigned)tiles_grid<1, 8>(tiles, sms), 256, 0, stream>>>(s->d, a);
        else k_query_fp64_tiles<1, 4><<<(unsigned)tiles_grid<1, 4>(tiles, sms), 256, 0, stream>>>(s->d, a);
        break;
      default:
        if (big) k_query_fp64_tiles<2, 8><<<(unsigned)tiles_grid<2, 8>(tiles, sms), 256, 0, stream>>>(s->d, a);
        else k_query_fp64_tiles<2, 4><<<(unsigned)tiles_grid<2, 4>(tiles, sms), 256, 0, stream>>>(s->d, a);
        break;
    }
    return cudaGetLastError();
  }
  int64_t blocks = (a.n + threads - 1) / threads;
  const int64_t cap = (int64_t)sms * 8;
  if (blocks > cap) blocks = cap;
  switch (s->h.type) {
    case kBox: k_query_fp64<0><<<(unsigned)blocks, threads, 0, stream>>>(s->d, a); break;
    case kTrd:
    case kTrap: k_query_fp64<1><<<(unsigned)blocks, threads, 0, stream>>>(s->d, a); break;
    case kBool:
      if (a.n > bool_rank_min(a, sms) && f64::bool_ranks(s->ph[0], s->ph[1])) {
        const int64_t resident = (int64_t)sms * 2;
        const unsigned grid = (unsigned)resident;
        if (a.n >= resident * 3072) k_query_bool_rank<4, false><<<grid, 256, 0, stream>>>(s->d, a);
        else if (a.n >= resident * 1024) k_query_bool_rank<4, true><<<grid, 256, 0, stream>>>(s->d, a);
        else if (a.din || a.dout) k_query_bool_rank<1, true><<<grid, 256, 0, stream>>>(s->d, a);
        else k_query_bool_rank<1, false><<<grid, 256, 0, stream>>>(s->d, a);
      } else {
        k_query_fp64<4><<<(unsigned)blocks, threads, 0, stream>>>(s->d, a);
      }
      break;
    default: k_query_fp64<2><<<(unsigned)blocks, threads, 0, stream>>>(s->d, a); break;
  }
  return cudaGetLastError();
}

#ifdef GV_DEBUG
cudaError_t debug_read_query64(unsigned long long out[2], bool clear) { return dbg_read(out, clear); }
#endif

}  // namespace gv
