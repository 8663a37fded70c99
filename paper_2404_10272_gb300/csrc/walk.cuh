// walk.cuh -- the per-ray walk shared by the single-call samplers
// (traverse.cu), the render-only path (render.cu) and the batched sampler
// (batch.cu): the lattice view, its header (closed form and bucket index),
// ray loading, exact point evaluation, region location on a dense or VDB
// grid, the region crossing search, the walk itself (from the start, or
// resumed after its first runs), the warp-cooperative expansion of runs into
// samples (4-byte stores for the one-pass kernel; a per-tile record list and
// 16-byte stores for the emits), the persistent walk kernel with its staged
// tables and its launch, and the scan of per-tile sample counts.  How the walk works
// and why it is exact is explained at the top of traverse.cu.
#pragma once

#include <cstring>
#include <type_traits>

#include "grid.cuh"

namespace hdda {
namespace {

constexpr int kMaxRuns = 16;    // runs per ray kept between the walk and the emit
constexpr unsigned kFull = 0xffffffffu;

// Loads from global memory (read-only path) or shared memory.
template <bool kSm, typename T>
__device__ __forceinline__ T ld(const T* p) {
  if constexpr (kSm) return *p;
  else return __ldg(p);
}

// A table of 4-byte words the walk reads, in shared memory (kSm: by its 32-bit
// shared address, so that no access goes through a generic one) or in global
// memory (read-only path).
template <bool kSm, typename T>
struct Tab {
  static_assert(sizeof(T) == 4, "4-byte entries");
  std::conditional_t<kSm, uint32_t, const T*> p;

  __device__ __forceinline__ T operator[](int i) const {
    if constexpr (kSm) {
      uint32_t v;
      asm("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(p + 4u * (uint32_t)i));
      T t;
      memcpy(&t, &v, 4);
      return t;
    } else {
      return __ldg(p + i);
    }
  }
  __device__ __forceinline__ Tab at(int i) const {
    if constexpr (kSm) return Tab{p + 4u * (uint32_t)i};
    else return Tab{p + i};
  }
};

// ---------------------------------------------------------------------------
// lattice
// ---------------------------------------------------------------------------

__device__ __forceinline__ float lattice_next(float t, const hdda_params& p) {
  const float dt = fminf(fmaxf(__fmul_rn(t, p.cone_angle), p.step), p.max_step);
  return __fadd_rn(t, dt);
}

LatticeDev lattice_view(char* block, int max_k, int K) {
  float* t = reinterpret_cast<float*>(block);
  float* tm = t + max_k + 1;
  int* kidx = reinterpret_cast<int*>(tm + max_k);
  uint32_t* hdr = reinterpret_cast<uint32_t*>(kidx + kKidxMax + 2);
  return LatticeDev{t, tm, kidx, hdr, K};
}

// The lattice header: the bucket index's {key0, shift, NB} and, when the
// lattice has the closed form (constant spacing up to index ks, geometric
// growth by 1 + cone per index from there), the values that estimate an
// index from it: tm_k = tm0 + k dt for k < ks and tm_k = tm_ks (1 + cone)^(k -
// ks) from ks on, both up to the recurrence's rounding.
struct LatHdr {
  uint32_t key0, shift;
  int NB;
  int lin;        // the closed form: 0 none (buckets), 1 constant spacing, 2 then geometric
  float inv_dt, c0;             // 1 / spacing at the start, -tm0 / spacing
  float tm_s, inv_tm_s, ks, A;  // tm_ks (+inf when ks = K), 1 / tm_ks, ks, 1 / log2(1 + cone)
};

__device__ __forceinline__ LatHdr lat_hdr(const LatticeDev& lat) {
  LatHdr h{__ldg(lat.hdr), __ldg(lat.hdr + 1), (int)__ldg(lat.hdr + 2),
           (int)__ldg(lat.hdr + 3), 0.f, 0.f, INFINITY, 0.f, 0.f, 0.f};
  if (h.lin && lat.K > 0) {
    const int ks = (int)__ldg(lat.hdr + 4);
    h.inv_dt = 1.0f / (__ldg(lat.t + 1) - __ldg(lat.t));
    h.c0 = -__ldg(lat.tm) * h.inv_dt;
    h.ks = (float)ks;
    h.A = __uint_as_float(__ldg(lat.hdr + 5));
    if (h.lin == 2 && ks < lat.K) {
      h.tm_s = __ldg(lat.tm + ks);
      h.inv_tm_s = 1.0f / h.tm_s;
    } else {
      h.lin = 1;
    }
  } else {
    h.lin = 0;
  }
  return h;
}

// ---------------------------------------------------------------------------
// the walk
// ---------------------------------------------------------------------------

// A ray in mirrored coordinates: every axis along which it moves backwards is
// negated, so that no coordinate decreases along the ray (negation is exact
// and binary32 rounding symmetric, so |x| of every point stays what it is).
// A region then ends at one upper bound per axis, and leaving it is three
// compares of one kind.
struct Ray {
  float o[3], d[3], inv[3];
  uint32_t nm[3];  // all ones on a mirrored axis, else 0
};

__device__ __forceinline__ bool load_ray(const float* __restrict__ ro,
                                         const float* __restrict__ rd, int64_t r, Ray& ray) {
  bool ok = true;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    const float o = __ldg(ro + 3 * r + c), d = __ldg(rd + 3 * r + c);
    ok &= isfinite(o) && isfinite(d);
    ray.nm[c] = d < 0.f ? ~0u : 0u;  // a zero component counts as positive
    ray.o[c] = d < 0.f ? -o : o;
    ray.d[c] = fabsf(d);
    // estimates only; +inf for a zero component, so that the crossing
    // estimate needs no test for it (see cross)
    ray.inv[c] = d != 0.f ? 1.0f / ray.d[c] : INFINITY;
  }
  return ok;
}

// The tables the walk reads per region, in shared memory (staged) or global
// memory; the rest of the grid stays in the GridDev kernel parameter.
template <bool kSm>
struct Tabs {
  Tab<kSm, float> tm;        // lattice midpoints
  Tab<kSm, int> kidx;        // their bucket index
  Tab<kSm, float> mthr;      // mirrored thresholds
  Tab<kSm, uint32_t> child, tile, prefix, nstate;
};

__device__ __forceinline__ Tabs<false> global_tabs(const GridDev& g, const LatticeDev& lat) {
  return Tabs<false>{{lat.tm}, {lat.kidx}, {g.mthr}, {g.child}, {g.tile}, {g.prefix}, {g.nstate}};
}

// First k with tm_k >= te (K if none), through the bucket index.
template <bool kSm>
__device__ __forceinline__ int first_k_at(const Tabs<kSm>& tb, const LatHdr& h, float te) {
  const uint32_t key = float_key(te);
  const int b = key < h.key0 ? 0 : (int)min((key - h.key0) >> h.shift, (uint32_t)h.NB);
  int lo = tb.kidx[b];
  const int hi = tb.kidx[b + 1];
  while (lo < hi && tb.tm[lo] < te) ++lo;
  return lo;
}

// x = o + tm * d per axis, one rounding per operation.
__device__ __forceinline__ void point_at(const Ray& r, float tm, float x[3]) {
#pragma unroll
  for (int c = 0; c < 3; ++c) x[c] = __fadd_rn(r.o[c], __fmul_rn(tm, r.d[c]));
}

// A region is kept as its upper bound per axis (exclusive, mirrored
// coordinates): the ray has left it once one coordinate reaches its bound.
__device__ __forceinline__ bool outside(const float x[3], const float e[3]) {
  return (x[0] >= e[0]) | (x[1] >= e[1]) | (x[2] >= e[2]);
}

// The lattice index at which tm reaches te, from the lattice's closed form
// (lat_hdr) or the bucket index; off by one at times (the probes correct it).
// Any value, saturated, for a te that is not finite.
template <bool kSm>
__device__ __forceinline__ int estimate_k(const Tabs<kSm>& tb, const LatHdr& h, float te) {
  if (h.lin == 1) return __float2int_ru(fmaf(te, h.inv_dt, h.c0));  // uniform over the launch
  if (h.lin == 2) {
    const float fc = fmaf(te, h.inv_dt, h.c0);                   // constant spacing
    const float fg = fmaf(__log2f(te * h.inv_tm_s), h.A, h.ks);  // geometric growth
    return __float2int_ru(te < h.tm_s ? fc : fg);
  }
  return first_k_at<kSm>(tb, h, te);
}

// First k in (k, kend) whose point is outside the region (kend if none).  The
// point of k is inside.  x receives the point of that k when it is below kend.
template <bool kSm>
__device__ __forceinline__ int cross(const Ray& r, const Tabs<kSm>& tb, const LatHdr& h, int k,
                                     int kend, const float e[3], float x[3]) {
  // estimate: the ray parameter where it meets the first bound.  On an axis
  // the ray does not move along, inv is +inf and the region holds the point,
  // so e - o > 0 there: the term is +inf and sets no bound.
  float te = INFINITY;
#pragma unroll
  for (int c = 0; c < 3; ++c) te = fminf(te, (e[c] - r.o[c]) * r.inv[c]);
  const int ke = max(estimate_k<kSm>(tb, h, te), k + 1);
  // two probes, at the estimate (or the last index) and before it: nearly
  // always the first is outside and the second inside
  const int kp = min(ke, kend - 1), kq = max(kp - 1, k);
  float y[3];
  point_at(r, tb.tm[kp], x);
  point_at(r, tb.tm[kq], y);
  const bool oa = outside(x, e), ob = outside(y, e);
  if (oa & !ob) return kp;
  if (!oa & (ke >= kend)) return kend;
  // the search looks `step` before hi, at most half way
  int lo, hi, step = 1;  // invariant: point lo inside (lo >= k); point hi outside, or hi == kend
  if (ob) {
    lo = k;  // estimate too late
    hi = kq;
  } else {
    for (lo = kp;; step <<= 1) {  // estimate too early: gallop forward
      hi = lo + step;
      if (hi >= kend) { hi = kend; break; }
      point_at(r, tb.tm[hi], y);
      if (outside(y, e)) break;
      lo = hi;
    }
  }
  while (hi - lo > 1) {
    const int mid = hi - min(step, (hi - lo) >> 1);
    point_at(r, tb.tm[mid], y);
    if (outside(y, e)) {
      hi = mid;
      step <<= 1;
    } else {
      lo = mid;
    }
  }
  if (hi < kend) point_at(r, tb.tm[hi], x);
  return hi;
}

// First k in [k0, k1) whose point satisfies `pred` (k1 if none); pred holds
// from some k on.  te estimates where.
template <bool kSm, typename P>
__device__ __forceinline__ int first_true(const Tabs<kSm>& tb, const LatHdr& h, int k0, int k1,
                                          float te, P pred) {
  if (k0 >= k1) return k1;
  int lo = k0 - 1, hi = k1;  // pred fails up to lo and holds from hi on
  int at = min(max(estimate_k<kSm>(tb, h, te), k0), k1 - 1);
  for (int step = 1; hi - lo > 1; step <<= 1) {  // gallop away from the estimate
    if (pred(tb.tm[at])) {
      hi = at;
      at = max(at - step, lo + 1);
      if (lo >= k0) at = lo + ((hi - lo) >> 1);  // both sides known: bisect
    } else {
      lo = at;
      at = min(at + step, hi - 1);
      if (hi < k1) at = lo + ((hi - lo) >> 1);
    }
  }
  return hi;
}

// A box face as a bound in mirrored coordinates: on a mirrored axis, x < v is
// -x >= -(the next value below v).
__device__ __forceinline__ float mirror_bound(float v) {
  const uint32_t u = __float_as_uint(v);
  if ((u & 0x7fffffffu) == 0u) return __uint_as_float(1u);  // below zero: -denorm_min
  return -__uint_as_float((u & 0x80000000u) ? u + 1u : u - 1u);
}

// The lattice indices [.x, .y) whose points lie in a level's box: one
// interval, because no (mirrored) coordinate decreases along the ray.
template <bool kSm>
__device__ __forceinline__ int2 box_span(const LevelDev& B, const Ray& r, const Tabs<kSm>& tb,
                                         const LatHdr& h, int K, int k0) {
  float en[3], ex[3];  // inside: en <= x < ex
  float ti = -INFINITY, tx = INFINITY;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    en[c] = r.nm[c] ? mirror_bound(B.hi[c]) : B.lo[c];
    ex[c] = r.nm[c] ? mirror_bound(B.lo[c]) : B.hi[c];
    ti = fmaxf(ti, (en[c] - r.o[c]) * r.inv[c]);
    tx = fminf(tx, (ex[c] - r.o[c]) * r.inv[c]);
  }
  const int a = first_true<kSm>(tb, h, k0, K, ti, [&](float tm) {
    float x[3];
    point_at(r, tm, x);
    return (x[0] >= en[0]) & (x[1] >= en[1]) & (x[2] >= en[2]);
  });
  const int b = first_true<kSm>(tb, h, a, K, tx, [&](float tm) {
    float x[3];
    point_at(r, tm, x);
    return outside(x, ex);
  });
  return make_int2(a, b);
}

// The stretches of a ray inside one level: lattice indices [k, kend) whose
// points belong to level l (the finest one holding them).  They follow from
// the levels' spans, which are found once per ray; the regions of a stretch
// then need no test of any box.  kOne: the grid has one level, so there is one
// stretch.  A level's constants are mirrored with the ray: voxel index =
// (x - lo) * s either way.
template <int kMode, bool kSm, bool kOne>
struct Stretch {
  float lo[3], s[3];
  Tab<kSm, float> T;  // the level's mirrored thresholds (hdda_internal.cuh), at index 0
  int l;
  int kend;
  int a[kOne ? 1 : kMaxLevels], b[kOne ? 1 : kMaxLevels];

  __device__ __forceinline__ void init(const GridDev& g, const Tabs<kSm>& tb, const Ray& r,
                                       const LatHdr& h, int K, int k0) {
    kend = k0;
    l = 0;
    if constexpr (kOne) {
      const int2 v = box_span<kSm>(g.lv[0], r, tb, h, K, k0);
      a[0] = v.x;
      b[0] = v.y;
      level(g, tb, r);
    } else {
#pragma unroll 1
      for (int i = 0; i < g.L; ++i) {
        const int2 v = box_span<kSm>(g.lv[i], r, tb, h, K, k0);
        a[i] = v.x;
        b[i] = v.y;
      }
    }
  }

  __device__ __forceinline__ void level(const GridDev& g, const Tabs<kSm>& tb, const Ray& r) {
    const LevelDev& V = g.lv[l];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      lo[c] = r.nm[c] ? -V.lo[c] : V.lo[c];
      s[c] = r.nm[c] ? -V.s[c] : V.s[c];
    }
    T = tb.mthr.at(l * 3 * mthr_stride(g.R) + g.R);
  }

  // The stretch at or after k (at its start, moved to k): false if there is none.
  __device__ __forceinline__ bool next(const GridDev& g, const Tabs<kSm>& tb, const Ray& r, int K,
                                       int& k) {
    if constexpr (kOne) {
      if (k >= b[0]) return false;
      k = max(k, a[0]);
      kend = b[0];
      return k < kend;
    } else {
      int at = -1, first = K, until = K;
#pragma unroll 1
      for (int i = 0; i < g.L; ++i) {
        const int ai = a[i], bi = b[i];
        if (ai >= bi || bi <= k) continue;
        if (ai <= k) {
          at = i;
          until = min(until, bi);  // until so far: where a finer level begins
          break;
        }
        until = min(until, ai);
        first = min(first, ai);
      }
      if (at < 0) {  // no level holds k: on to the first that begins later
        if (first >= K) return false;
        k = first;
        until = K;
#pragma unroll 1
        for (int i = 0; i < g.L; ++i) {
          const int ai = a[i], bi = b[i];
          if (ai >= bi || bi <= k) continue;
          if (ai <= k) {
            at = i;
            until = min(until, bi);
            break;
          }
          until = min(until, ai);
        }
      }
      kend = until;
      l = at;
      level(g, tb, r);
      return true;
    }
  }
};

// Classifies x, a point of the stretch's level: returns its occupancy and
// sets e to the upper bounds of the region holding it.
// kSm: the tables in tb point into shared memory.
template <int kMode, bool kSm, bool kOne>
__device__ __forceinline__ bool locate(const GridDev& g, const Tabs<kSm>& tb, const Ray& r,
                                       const Stretch<kMode, kSm, kOne>& st, const float x[3],
                                       float e[3]) {
  const int l = kOne ? 0 : st.l;
  int i[3];
#pragma unroll
  for (int c = 0; c < 3; ++c)  // x lies in the box, so the index is not negative
    i[c] = min(__float2int_rd(__fmul_rn(__fsub_rn(x[c], st.lo[c]), st.s[c])), g.R - 1);
  // Descend to the coarsest uniform region holding x: an aligned cube of `szm`
  // + 1 voxels (cut off at the grid edge).  Every kind ends in the one bound
  // lookup below, so lanes that stop at different depths share it.
  uint32_t szm = 0;
  bool occ;
  do {
    if constexpr (kMode == kModeDense) {
      // R^3 <= 2^30 and L * W <= 2^28: 32-bit offsets (5 % faster than 64-bit)
      const int lin = (i[0] * g.R + i[1]) * g.R + i[2];
      const uint32_t w = __ldg(g.bits + (l * g.W + (lin >> 5)));
      occ = (w >> (lin & 31)) & 1u;
      break;
    }
    if constexpr (kMode == kModeVdbMap) {
      // the refined tree's region, flattened: one 2-byte load.  C^3 * L <= 2^27 * 8
      // entries, so the offset fits 32 bits
      const int C = (g.R + 1) >> 1;
      const int cell = ((l * C + (i[0] >> 1)) * C + (i[1] >> 1)) * C + (i[2] >> 1);
      const uint32_t m = __ldg(g.rmap + cell);
      occ = (m >> (((i[0] & 1) << 2) | ((i[1] & 1) << 1) | (i[2] & 1))) & 1u;
      szm = (1u << (m >> 8)) - 1u;
      break;
    }
    // plain tree.  Node level: L * N^3 <= 8 * 8^3 nodes and L * B^3 * 16 <= 2^28 leaf
    // words, so every offset below fits 32 bits (cheaper address arithmetic than 64-bit)
    const int N = g.N;
    const int ng = l * N * N * N + ((i[0] >> 7) * N + (i[1] >> 7)) * N + (i[2] >> 7);
    const uint32_t st_n = tb.nstate[ng];
    if (st_n != kNodeMixed) {
      szm = kNodeVox - 1;
      occ = st_n == kNodeFull;
      break;
    }
    // block level: empty or tile
    const int cell = (((i[0] >> 3) & 15) * 16 + ((i[1] >> 3) & 15)) * 16 + ((i[2] >> 3) & 15);
    const int w = cell >> 5;
    const uint32_t bit = 1u << (cell & 31);
    const uint32_t cw = tb.child[ng * kNodeWords + w];
    if (!(cw & bit)) {
      szm = kBlockDim - 1;
      occ = (tb.tile[ng * kNodeWords + w] & bit) != 0u;
      break;
    }
    // voxel of a leaf
    const uint32_t leaf = tb.prefix[ng * kNodeWords + w] + __popc(cw & (bit - 1u));
    const int v = ((i[0] & 7) * 8 + (i[1] & 7)) * 8 + (i[2] & 7);
    const uint32_t lw = __ldg(g.leaves + (leaf * (uint32_t)kLeafWords + (uint32_t)(v >> 5)));
    occ = (lw >> (v & 31)) & 1u;
  } while (false);
  const int TS = mthr_stride(g.R);
#pragma unroll
  for (int c = 0; c < 3; ++c)
    e[c] = st.T[c * TS + (int)(((uint32_t)i[c] ^ r.nm[c]) | szm)];
  return occ;
}

// Walks one ray.  Counts its samples and merges occupied regions into runs
// [k_begin, k_end): the first kMaxRuns go to runs[j * stride]; nruns counts
// all.
// kSkip selects the control flow of Algorithm 2 ("DDA skip": cross every
// leading empty region in an inner loop, then take the occupied one)
// instead of Algorithm 1 ("DDA branch": one region per iteration, branching
// on its occupancy).  The regions crossed, and so the samples, are the same.
// kCheck tests that every region holds the point it was found from (raising
// kDevInternal otherwise); the invariant the crossing search rests on.
template <int kMode, bool kSm, bool kSkip, bool kCheck, bool kOne>
__device__ __forceinline__ int64_t walk_levels(const GridDev& g, const Tabs<kSm>& tb,
                                               const LatticeDev& lat, const LatHdr& h,
                                               const Ray& r, uint2* runs, int64_t stride,
                                               int& nruns, unsigned* __restrict__ status) {
  int kept = 0;  // at most 2^24
  nruns = 0;
  if (lat.K <= 0) return 0;
  int rb = -1, re = -1;  // open run
  float x[3];
  int k = 0;
  Stretch<kMode, kSm, kOne> st;
  st.init(g, tb, r, h, lat.K, 0);
  for (;;) {
    bool occ, over = false;
    int kn;
    // One region; in the skip form, every leading empty region first (one
    // copy of locate and cross serves both forms).  cross advances by
    // construction; the skip form still guards its inner loop (no progress:
    // report, end the ray).
    for (;;) {
      if (k >= st.kend) {
        over = !st.next(g, tb, r, lat.K, k);
        if (over) break;
        point_at(r, tb.tm[k], x);
      }
      float e[3];
      occ = locate(g, tb, r, st, x, e);
      if constexpr (kCheck)
        if (outside(x, e)) atomicOr(status, kDevInternal);
      kn = cross<kSm>(r, tb, h, k, st.kend, e, x);
      if constexpr (kSkip)
        if (kn <= k) {
          atomicOr(status, kDevInternal);
          over = true;
          break;
        }
      if (!kSkip || occ) break;
      k = kn;
    }
    if (over) break;
    // an occupied region extends the open run or, not adjacent, opens the next one
    const bool opens = occ & (k != re);
    if (opens & (rb >= 0)) {
      if (nruns < kMaxRuns) runs[nruns * stride] = make_uint2(rb, re);
      ++nruns;
    }
    kept += occ ? kn - k : 0;
    rb = opens ? k : rb;
    re = occ ? kn : re;
    k = kn;
  }
  if (rb >= 0) {
    if (nruns < kMaxRuns) runs[nruns * stride] = make_uint2(rb, re);
    ++nruns;
  }
  return kept;
}

// The walk with the one-level form where it applies (its own copy of the
// code).
template <int kMode, bool kSm, bool kSkip = false, bool kCheck = false>
__device__ __forceinline__ int64_t walk(const GridDev& g, const Tabs<kSm>& tb,
                                        const LatticeDev& lat, const LatHdr& h, const Ray& r,
                                        uint2* runs, int64_t stride, int& nruns,
                                        unsigned* __restrict__ status) {
  if (g.L == 1)  // uniform
    return walk_levels<kMode, kSm, kSkip, kCheck, true>(g, tb, lat, h, r, runs, stride, nruns,
                                                        status);
  return walk_levels<kMode, kSm, kSkip, kCheck, false>(g, tb, lat, h, r, runs, stride, nruns,
                                                       status);
}

// Writes the samples of a ray from lattice index k0 on to `out`, below
// `capacity`, until `left` of them are written or counted (lat.t is a table in
// global memory): the rest of a ray with more runs than were kept, found by a
// second walk.  It starts behind the runs that were, which it need not cross
// again: a single such ray keeps a whole kernel waiting (65,536 rays of which
// 13 have 17 to 19 runs, 2 x 512^3 voxels: the emit took 119 us when they walked
// again from the start, 38 so).  Resuming as walk_from does.
template <int kMode, bool kSm>
__device__ __forceinline__ void emit_from(const GridDev& g, const Tabs<kSm>& tb,
                                          const LatticeDev& lat, const LatHdr& h, const Ray& r,
                                          int k0, int64_t left, int32_t rid, int64_t out,
                                          int64_t capacity, int32_t* __restrict__ ray_idx,
                                          float* __restrict__ t0, float* __restrict__ t1) {
  if (k0 >= lat.K) return;
  float x[3];
  int k = k0;
  Stretch<kMode, kSm, false> st;
  st.init(g, tb, r, h, lat.K, k0);
  while (left > 0) {
    if (k >= st.kend) {
      if (!st.next(g, tb, r, lat.K, k)) break;
      point_at(r, tb.tm[k], x);
    }
    float e[3];
    const bool occ = locate(g, tb, r, st, x, e);
    const int kn = cross<kSm>(r, tb, h, k, st.kend, e, x);
    if (occ) {
      float ta = __ldg(lat.t + k);
      for (int j = k; j < kn && left > 0; ++j, ++out, --left) {
        const float tn = __ldg(lat.t + j + 1);
        if (out < capacity) {
          ray_idx[out] = rid;
          t0[out] = ta;
          t1[out] = tn;
        }
        ta = tn;
      }
    }
    k = kn;
  }
}

// Walks one ray from lattice index k0 and stops after kMaxRuns runs: writes
// them to runs[j * stride], sets nruns, and returns the index where the walk
// resumes (the first k of the next run), or K once the ray is done.  Used
// for rays with more runs than the first pass keeps; resuming at any k gives
// the same samples because every point is classified on its own.  It does
// not check its regions: the first pass crossed the same ones.
template <int kMode, bool kSm>
__device__ __forceinline__ int walk_from(const GridDev& g, const Tabs<kSm>& tb,
                                         const LatticeDev& lat,
                                         const LatHdr& h, const Ray& r, int k0, uint2* runs,
                                         int stride, int& nruns) {
  const int K = lat.K;
  nruns = 0;
  if (k0 >= K) return K;
  int rb = -1, re = -1;  // open run
  float x[3];
  int k = k0;
  Stretch<kMode, kSm, false> st;
  st.init(g, tb, r, h, K, k0);
  for (;;) {
    if (k >= st.kend) {
      if (!st.next(g, tb, r, K, k)) break;
      point_at(r, tb.tm[k], x);
    }
    float e[3];
    const bool occ = locate(g, tb, r, st, x, e);
    const int kn = cross<kSm>(r, tb, h, k, st.kend, e, x);
    if (occ) {
      if (k == re) {
        re = kn;
      } else {
        if (rb >= 0) {
          runs[nruns * stride] = make_uint2(rb, re);
          if (++nruns == kMaxRuns) return k;
        }
        rb = k;
        re = kn;
      }
    }
    k = kn;
  }
  if (rb >= 0) runs[(nruns++) * stride] = make_uint2(rb, re);
  return K;
}

// ---------------------------------------------------------------------------
// expansion of runs into samples
// ---------------------------------------------------------------------------

// One warp writes the samples of its 32 rays.  Lane i holds ray rid0 + i
// with `c` samples from output position `off` (rays in order, so the
// warp's samples are one contiguous range); its runs are runs0[i + j *
// stride], j < kMaxRuns.  Lane j of each 32-sample chunk finds the ray that
// owns its position (binary search over the lanes' offsets) and the run
// inside it.  Rays with more runs than were kept are skipped here; they
// walk again.  Nothing at or past `capacity` is written.
template <bool kSm>
__device__ __forceinline__ void expand_warp(int64_t off, int64_t c, bool overflow,
                                            const uint2* runs0, int64_t stride, int32_t rid0,
                                            const float* __restrict__ t, int64_t capacity,
                                            int32_t* __restrict__ ray_idx,
                                            float* __restrict__ t0, float* __restrict__ t1) {
  const int lane = threadIdx.x & 31;
  const int64_t wbeg = __shfl_sync(kFull, off, 0);
  const int64_t wend = __shfl_sync(kFull, off + c, 31);
  for (int64_t base = wbeg; base < wend; base += 32) {
    const int64_t p = base + lane;
    int own = 0;  // the last lane whose offset is <= p
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      const int64_t v = __shfl_sync(kFull, off, own + s);
      if (v <= p) own += s;
    }
    const int64_t own_off = __shfl_sync(kFull, off, own);
    const int own_ovf = __shfl_sync(kFull, (int)overflow, own);
    if (p < wend && !own_ovf && p < capacity) {
      const uint2* rr = runs0 + own;
      int64_t loc = p - own_off;
      uint2 run = ld<kSm>(rr);
      int j = 0;
      while (loc >= (int64_t)(run.y - run.x)) {
        loc -= run.y - run.x;
        run = ld<kSm>(rr + (++j) * stride);
      }
      const int k = (int)run.x + (int)loc;
      ray_idx[p] = rid0 + own;
      t0[p] = __ldg(t + k);
      t1[p] = __ldg(t + k + 1);
    }
  }
}

// The expansion of the two-pass samplers' emit (separate, fused with the
// walk, or batched), with 16-byte stores.  A warp first lists its tile's
// runs, rays in order and each ray's runs in order, as records {first output
// position relative to the tile's first sample, (first k << 5) | lane}: one
// per run, or, for a ray with more runs than were kept, its last one with
// kRecSkip set, covering all of the ray's samples from that run on (the ray
// walks on from there and writes them itself: emit_from).  A sentinel record with position kRecEnd follows the
// last.  Positions are then expanded four per lane per 128-position block
// (expand_records): a lane finds the record holding its first position, and
// a record covers at least one position, so its four positions lie in at most
// four consecutive records.  A sample's k is its record's first k plus its
// distance from the record's first position.  Positions at or past `lim` (the
// tile's samples, cut off at the buffer's capacity) are not written.
constexpr int kRecMax = 32 * kMaxRuns;   // records of one 32-ray tile
constexpr uint32_t kRecSkip = 1u << 31;
constexpr uint32_t kRecEnd = 0xffffffffu;

// Lane-local part of the listing: writes this lane's records from index
// `first` (the lanes' exclusive scan of their record counts).  `c` is the
// lane's sample count and `q` its first position relative to the tile; run j
// of the lane's ray is runs_r[j * stride].  The runs are read through L2
// (ld.global.cg), not the read-only path, because the fused sampler form
// reads them in the kernel that wrote them.  With more than kMaxRuns runs,
// returns where the last kept one starts: {its first k, its first position};
// else {0, 0}.  Those rays have a loop of their own: with the case decided per
// run in one loop, the emit of an 800 x 800 frame took 140 us instead of 90.
__device__ __forceinline__ uint2 list_runs(uint2* rec, int first, int lane, int nr, int64_t c,
                                           uint32_t q, const uint2* __restrict__ runs_r,
                                           int64_t stride) {
  if (c <= 0) return make_uint2(0u, 0u);
  if (nr > kMaxRuns) {
    for (int j = 0;; ++j) {
      const uint2 v = __ldcg(runs_r + (int64_t)j * stride);
      if (j == kMaxRuns - 1) {
        rec[first + j] = make_uint2(q, kRecSkip | (uint32_t)lane);
        return make_uint2(v.x, q);
      }
      rec[first + j] = make_uint2(q, (v.x << 5) | (uint32_t)lane);
      q += v.y - v.x;
    }
  }
  for (int j0 = 0; j0 < nr; j0 += 4) {
    uint2 v[4];
#pragma unroll
    for (int u = 0; u < 4; ++u)
      if (j0 + u < nr) v[u] = __ldcg(runs_r + (int64_t)(j0 + u) * stride);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      if (j0 + u < nr) {
        rec[first + j0 + u] = make_uint2(q, (v[u].x << 5) | (uint32_t)lane);
        q += v[u].y - v[u].x;
      }
    }
  }
  return make_uint2(0u, 0u);
}

// One record as the expansion uses it: its sample positions q map to
// lattice index kq + q (kq = first k - first position) and to ray rid0 +
// lane; `skip` marks a ray that writes its own samples; `nxt` is the next
// record's first position.
struct RecView {
  int kq;
  int32_t rid;
  bool skip;
  uint32_t nxt;
};

__device__ __forceinline__ RecView rec_view(const uint2* rec, int u, int32_t rid0) {
  const uint2 r = rec[u];
  RecView v;
  v.kq = (int)((r.y & ~kRecSkip) >> 5) - (int)r.x;
  v.rid = rid0 + (int)(r.y & 31u);
  v.skip = (r.y & kRecSkip) != 0u;
  v.nxt = rec[u + 1].x;
  return v;
}

// The four positions q0 .. q0 + 3 of one lane, from record u on, record by
// record (any number of record changes).  Returns in ok[i] whether position
// q0 + i is written here.
__device__ __forceinline__ void expand_four_any(const uint2* rec, int& u, int q0, int lim,
                                                int32_t rid0, const float* __restrict__ t,
                                                int32_t vr[4], float va[4], float vb[4],
                                                bool ok[4]) {
  RecView v = rec_view(rec, u, rid0);
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int q = q0 + i;
    ok[i] = q >= 0 && q < lim;
    vr[i] = 0;
    va[i] = vb[i] = 0.f;
    if (!ok[i]) continue;
    if ((uint32_t)q >= v.nxt) v = rec_view(rec, ++u, rid0);  // a record holds >= 1 position
    ok[i] = !v.skip;
    if (!ok[i]) continue;
    const int k = v.kq + q;
    vr[i] = v.rid;
    va[i] = __ldg(t + k);
    vb[i] = __ldg(t + k + 1);
  }
}

// Expands the records rec[0 .. nrec) (sentinel at rec[nrec]) of one tile
// whose first sample goes to output position wbeg.  vec: ray_idx, t0 and t1
// are 16-byte aligned, so whole 4-position groups take one 16-byte store
// per array.  Each 128-position block starts from `ufirst`, a record at or
// before all of its positions (the record of the previous block's last
// position): lane j reads the first position of record ufirst + j, and a
// five-step shuffle search gives each lane the last of those 32 records
// starting at or before its first position; a lane whose position lies
// beyond them (a block of more than 32 records) binary-searches the rest.
// A lane's four positions then take their lattice index, ray and skip flag
// from that record or the next one by selects; only a lane whose positions
// reach a third record steps through them one by one.  Of several warps that
// share the tile, the one with number `part` of 2^shift writes an equal part of
// the blocks (kSplit).
template <bool kSplit = false>
__device__ __forceinline__ void expand_records(const uint2* rec, int nrec, int lim, int64_t wbeg,
                                               int32_t rid0, const float* __restrict__ t,
                                               bool vec, int32_t* __restrict__ ray_idx,
                                               float* __restrict__ t0, float* __restrict__ t1,
                                               int part = 0, int shift = 0) {
  if (nrec <= 0 || lim <= 0) return;
  const int lane = threadIdx.x & 31;
  int ufirst = 0;  // rec[0] starts at position 0
  int base = -(int)(wbeg & 3), end = lim;
  if constexpr (kSplit) {
    const int64_t blocks = ((int64_t)lim - base + 127) >> 7;
    end = (int)min((int64_t)lim, 128 * ((blocks * (part + 1)) >> shift) + base);
    base += (int)(128 * ((blocks * part) >> shift));
  }
  for (; base < end; base += 128) {
    const int q0 = base + 4 * lane;
    const int qs = max(q0, 0);
    const uint32_t pj = rec[min(ufirst + lane, nrec)].x;  // the sentinel past the end
    int j = 0;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      const uint32_t pv = __shfl_sync(kFull, pj, j + s);
      if (pv <= (uint32_t)qs) j += s;
    }
    int u = ufirst + j;
    if (j == 31 && u < nrec) {  // the record may lie further on: binary search
      int hi = nrec;  // rec[u] <= qs < rec[hi] (the sentinel)
      while (hi - u > 1) {
        const int mid = (u + hi) >> 1;
        if (rec[mid].x <= (uint32_t)qs) u = mid;
        else hi = mid;
      }
    }
    int32_t vr[4];
    float va[4], vb[4];
    bool ok[4] = {false, false, false, false};
    if (qs < lim) {
      // The lane's positions lie in record u and, past its end, in record u + 1
      // (without branches), unless they reach a third record (short runs).
      const RecView a = rec_view(rec, u, rid0);
      const RecView b = rec_view(rec, min(u + 1, nrec - 1), rid0);  // used only past a.nxt
      if ((uint32_t)(q0 + 3) >= b.nxt && a.nxt <= (uint32_t)(q0 + 3)) {
        expand_four_any(rec, u, q0, lim, rid0, t, vr, va, vb, ok);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int q = q0 + i;
          const bool in_a = (uint32_t)q < a.nxt;
          const int k = (in_a ? a.kq : b.kq) + q;
          vr[i] = in_a ? a.rid : b.rid;
          ok[i] = q >= 0 && q < lim && !(in_a ? a.skip : b.skip);
          va[i] = ok[i] ? __ldg(t + k) : 0.f;
          vb[i] = ok[i] ? __ldg(t + k + 1) : 0.f;
        }
        if (a.nxt <= (uint32_t)(q0 + 3)) ++u;  // the record of the lane's last position
      }
      const int64_t p0 = wbeg + q0;
      if (vec && (ok[0] & ok[1] & ok[2] & ok[3])) {
        *reinterpret_cast<int4*>(ray_idx + p0) = make_int4(vr[0], vr[1], vr[2], vr[3]);
        *reinterpret_cast<float4*>(t0 + p0) = make_float4(va[0], va[1], va[2], va[3]);
        *reinterpret_cast<float4*>(t1 + p0) = make_float4(vb[0], vb[1], vb[2], vb[3]);
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (!ok[i]) continue;
          ray_idx[p0 + i] = vr[i];
          t0[p0 + i] = va[i];
          t1[p0 + i] = vb[i];
        }
      }
    }
    ufirst = __shfl_sync(kFull, u, 31);  // the record of this block's last position
  }
}

// ---------------------------------------------------------------------------
// pass 1 of the two-pass samplers and of the render-only path: the walk
// (persistent warps, staged tables)
// ---------------------------------------------------------------------------

// 32 warps, one CTA per SM: the tables are staged once per SM (3 % faster than
// two CTAs of 512 on the object frame, no register spills)
constexpr int kWalkBS = 1024;

// Shared-memory bytes that stage the walk's tables (0 = they do not fit).
struct StageLayout {
  size_t tm, kidx, thr, child, tile, prefix, nstate, bytes;
};

__host__ __device__ inline StageLayout stage_layout(int K, int L, int R, int64_t nodes, int mode) {
  StageLayout s{};
  size_t o = 0;
  s.tm = o; o += sizeof(float) * (size_t)K;
  s.kidx = o; o += sizeof(int) * (size_t)(kKidxMax + 2);
  s.thr = o; o += sizeof(float) * (size_t)L * 3 * mthr_stride(R);
  s.child = s.tile = s.prefix = s.nstate = o;
  if (mode == kModeVdb) {
    s.child = o; o += 4 * (size_t)nodes * kNodeWords;
    s.tile = o; o += 4 * (size_t)nodes * kNodeWords;
    s.prefix = o; o += 4 * (size_t)nodes * kNodeWords;
    s.nstate = o; o += 4 * (size_t)nodes;
  }
  s.bytes = (o + 15) & ~(size_t)15;
  return s;
}

// leaves the L1 half of the SM's 256 KB
constexpr size_t kMaxStageBytes = 128 * 1024;
constexpr size_t kMaxCtaSmem = 227 * 1024;  // what one CTA can have on sm_103a

template <typename T>
__device__ __forceinline__ void stage_copy(T* dst, const T* __restrict__ src, int64_t count) {
  for (int64_t i = threadIdx.x; i < count; i += blockDim.x) dst[i] = __ldg(src + i);
}

// The walk's tables: copied into shared memory at `smem` (stage_layout, kSm;
// synchronises the block) or where they are.
template <int kMode, bool kSm>
__device__ __forceinline__ Tabs<kSm> walk_tables(unsigned char* smem, const GridDev& g,
                                                 const LatticeDev& lat, const LatHdr& h) {
  if constexpr (!kSm) {
    return global_tabs(g, lat);
  } else {
    const int64_t nodes = (int64_t)g.L * g.N * g.N * g.N;
    const StageLayout sl = stage_layout(lat.K, g.L, g.R, nodes, kMode);
    stage_copy(reinterpret_cast<float*>(smem + sl.tm), lat.tm, lat.K);
    if (!h.lin)  // the closed form does without the buckets
      stage_copy(reinterpret_cast<int*>(smem + sl.kidx), lat.kidx, (int64_t)h.NB + 2);
    stage_copy(reinterpret_cast<float*>(smem + sl.thr), g.mthr,
               (int64_t)g.L * 3 * mthr_stride(g.R));
    if constexpr (kMode == kModeVdb) {
      stage_copy(reinterpret_cast<uint32_t*>(smem + sl.child), g.child, nodes * kNodeWords);
      stage_copy(reinterpret_cast<uint32_t*>(smem + sl.tile), g.tile, nodes * kNodeWords);
      stage_copy(reinterpret_cast<uint32_t*>(smem + sl.prefix), g.prefix, nodes * kNodeWords);
      stage_copy(reinterpret_cast<uint32_t*>(smem + sl.nstate), g.nstate, nodes);
    }
    __syncthreads();
    uint32_t b = (uint32_t)__cvta_generic_to_shared(smem);
    asm volatile("" : "+r"(b)::"memory");  // the loads depend on it: none moves above the barrier
    return Tabs<true>{{b + (uint32_t)sl.tm},    {b + (uint32_t)sl.kidx},
                      {b + (uint32_t)sl.thr},   {b + (uint32_t)sl.child},
                      {b + (uint32_t)sl.tile},  {b + (uint32_t)sl.prefix},
                      {b + (uint32_t)sl.nstate}};
  }
}

// Adds v samples to 32-ray tile t: its sum and, when kept, the sums of its
// groups of 32 and of 1024 tiles (all zeroed by the caller).
__device__ __forceinline__ void add_tile_sum(int64_t t, int64_t v, int64_t* tile_sum,
                                             unsigned long long* sums32,
                                             unsigned long long* sums1024) {
  atomicAdd(reinterpret_cast<unsigned long long*>(tile_sum) + t, (unsigned long long)v);
  if (sums32) {
    atomicAdd(sums32 + (t >> 5), (unsigned long long)v);
    atomicAdd(sums1024 + (t >> 10), (unsigned long long)v);
  }
}

// Pass 1.  Persistent: each warp takes work tiles in order until none is
// left, so a warp never waits for another.  A work tile is 32 consecutive
// rays, or, when the rays are the pixels of a `width`-wide image row by row
// (width > 0), a block of 8 x 4 pixels, whose rays start and end their
// regions at more similar depths.  Writes counts[r], nruns[r] (saturated at
// 255) and the first kMaxRuns runs at runs[r + j * n], and, unless tile_sum
// is null, each 32-ray tile's sample total at tile_sum[r / 32]: stored in
// index order, added atomically in block order (then zeroed by the caller).
template <int kMode, bool kSm, bool kSkip, bool kCheck>
__global__ void __launch_bounds__(kWalkBS) walk_kernel(
    const float* __restrict__ ro, const float* __restrict__ rd, int64_t n, GridDev g,
    LatticeDev lat, int32_t* __restrict__ counts, uint8_t* __restrict__ nruns_out,
    uint2* __restrict__ runs, int64_t* __restrict__ tile_sum, unsigned* __restrict__ tile_counter,
    unsigned* __restrict__ status, unsigned long long* __restrict__ sums32,
    unsigned long long* __restrict__ sums1024, int32_t width) {
  extern __shared__ __align__(16) unsigned char smem[];
  const LatHdr h = lat_hdr(lat);
  const Tabs<kSm> tb = walk_tables<kMode, kSm>(smem, g, lat, h);
  // work tiles, and block columns: 8 x 4 blocks over ceil(n / width) rows.
  // Kept in shared memory, not in registers across the walk.
  __shared__ unsigned s_tiles[2];
  if (threadIdx.x == 0) {
    const unsigned bc = width > 0 ? ((unsigned)width + 7) / 8 : 0;
    s_tiles[0] = width > 0 ? bc * (unsigned)(((n + width - 1) / width + 3) / 4)
                           : (unsigned)((n + 31) / 32);
    s_tiles[1] = bc;
  }
  __syncthreads();
  const int lane = threadIdx.x & 31;
  for (;;) {
    unsigned tile = 0;
    if (lane == 0) tile = atomicAdd(tile_counter, 1u);
    tile = __shfl_sync(kFull, tile, 0);
    if (tile >= s_tiles[0]) break;
    int64_t r;
    bool ok;
    if (width > 0) {
      const unsigned bcols = s_tiles[1];
      const unsigned by = tile / bcols, x = (tile - by * bcols) * 8 + (lane & 7);
      r = (int64_t)(by * 4 + (lane >> 3)) * width + x;
      ok = x < (unsigned)width && r < n;
    } else {
      r = (int64_t)tile * 32 + lane;
      ok = r < n;
    }
    int64_t c = 0;
    if (ok) {
      Ray ray;
      int nr = 0;
      if (load_ray(ro, rd, r, ray))
        c = walk<kMode, kSm, kSkip, kCheck>(g, tb, lat, h, ray, runs + r, n, nr, status);
      counts[r] = (int32_t)c;
      nruns_out[r] = (uint8_t)min(nr, 255);
    }
    if (!tile_sum) continue;
    if (width > 0) {
      // the 8 lanes of a block row hold consecutive rays, so at most two
      // 32-ray tiles: the row leader's and the next.  A row whose leader is
      // out of range has no ray in range.
      const int64_t t = r >> 5, ta = __shfl_sync(kFull, t, lane & ~7);
      int64_t a = t == ta ? c : 0, b = c - a;
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        a += __shfl_xor_sync(kFull, a, o);
        b += __shfl_xor_sync(kFull, b, o);
      }
      if ((lane & 7) == 0) {
        if (a) add_tile_sum(ta, a, tile_sum, sums32, sums1024);
        if (b) add_tile_sum(ta + 1, b, tile_sum, sums32, sums1024);
      }
      continue;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(kFull, c, o);
    if (lane == 0) {
      const int64_t t = r >> 5;  // lane 0's ray opens the tile
      tile_sum[t] = c;
      if (sums32) {  // the group sums tile_offset reads (zeroed by the caller)
        atomicAdd(sums32 + (t >> 5), (unsigned long long)c);
        atomicAdd(sums1024 + (t >> 10), (unsigned long long)c);
      }
    }
  }
}

// The first output position of tile t: the sum of every earlier tile's
// samples, from the sums the walk kept per 1024 tiles and per 32 tiles and
// the tile sums themselves (at most 31 + 31 entries of the last two, and
// t / 1024 of the first, read by the warp's lanes at once).  Called by a
// whole warp; every lane returns the offset.
__device__ __forceinline__ int64_t tile_offset(int64_t t, const int64_t* __restrict__ tile_sum,
                                               const unsigned long long* __restrict__ sums32,
                                               const unsigned long long* __restrict__ sums1024) {
  const int lane = threadIdx.x & 31;
  int64_t v = 0;
  const int64_t g2 = t >> 10;  // whole 1024-tile groups before t
  for (int64_t j = lane; j < g2; j += 32) v += (int64_t)__ldg(sums1024 + j);
  const int64_t g1 = (g2 << 5) + lane;  // 32-tile groups of t's 1024-tile group before t's
  if (g1 < (t >> 5)) v += (int64_t)__ldg(sums32 + g1);
  const int64_t j0 = ((t >> 5) << 5) + lane;  // tiles of t's 32-tile group before t
  if (j0 < t) v += __ldg(tile_sum + j0);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(kFull, v, o);
  return v;
}

// ---------------------------------------------------------------------------
// host-side launch of the walk
// ---------------------------------------------------------------------------

// The walk a grid takes: dense DDA, or HDDA with or without refinement.
int walk_mode(const hdda_grid* grid) {
  if (grid->kind == HDDA_GRID_DENSE) return kModeDense;
  return grid->refine ? kModeVdbMap : kModeVdb;
}

struct WalkArgs {
  const float* ro;
  const float* rd;
  int64_t n;
  GridDev g;
  LatticeDev lat;
  int32_t* counts;
  uint8_t* nruns;
  uint2* runs;
  int64_t* tile_sum;
  unsigned* counter;
  unsigned* status;
  unsigned long long* sums32 = nullptr;    // optional group sums for tile_offset
  unsigned long long* sums1024 = nullptr;
  int32_t width = 0;                       // image width: walk in 8 x 4 pixel blocks
};

template <int kMode, bool kSm, bool kSkip>
int launch_walk(const WalkArgs& w, size_t smem, cudaStream_t s) {
  // the checked instantiation only while region checks are on
  auto kern = w.g.check ? walk_kernel<kMode, kSm, kSkip, true> : walk_kernel<kMode, kSm, kSkip, false>;
  if (smem > 48 * 1024)
    HDDA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)smem));
  int dev = 0;
  HDDA_CUDA_TRY(cudaGetDevice(&dev));
  // one resident wave, but no more CTAs than one per eight 32-ray tiles: a small call
  // is still spread over several SMs (its warps take tiles from the shared counter)
  // without every SM staging the tables for warps that find no tile (30 us on the
  // 96x96 frame, 288 tiles; one CTA per tile or per 32 tiles was 6 and 14 % slower
  // when the walk took 75 us).
  const int64_t want = ((w.n + 31) / 32 + 7) / 8;
  const int64_t full = sm_count(dev);  // one CTA of 1024 fits (57 registers a thread)
  const unsigned grid = (unsigned)(want < full ? want : full);
  kern<<<grid, kWalkBS, smem, s>>>(w.ro, w.rd, w.n, w.g, w.lat, w.counts, w.nruns, w.runs,
                                   w.tile_sum, w.counter, w.status, w.sums32, w.sums1024,
                                   w.width);
  HDDA_CUDA_TRY(cudaGetLastError());
  return HDDA_OK;
}

template <int kMode>
int launch_walk_mode(const WalkArgs& w, size_t stage_bytes, bool skip, cudaStream_t s) {
  if (skip)
    return stage_bytes <= kMaxStageBytes ? launch_walk<kMode, true, true>(w, stage_bytes, s)
                                         : launch_walk<kMode, false, true>(w, 0, s);
  return stage_bytes <= kMaxStageBytes ? launch_walk<kMode, true, false>(w, stage_bytes, s)
                                       : launch_walk<kMode, false, false>(w, 0, s);
}

const char* walk_name(int mode) {
  return mode == kModeDense ? "dense_walk" : mode == kModeVdb ? "hdda_walk_plain" : "hdda_walk";
}

// ---------------------------------------------------------------------------
// scan of per-tile sample counts
// ---------------------------------------------------------------------------

// Exclusive scan of the per-tile sums by one CTA of 1024 threads.  The sums
// go through shared memory in chunks of 4096 (coalesced loads and stores);
// each thread scans 4 consecutive entries, a CTA scan joins the threads and
// a carry joins the chunks.  Writes the total and offsets[n] too.
constexpr int kScanThreads = 1024;
constexpr int kScanPer = 4;

__global__ void __launch_bounds__(kScanThreads) tile_scan_kernel(
    const int64_t* __restrict__ tile_sum, int64_t T, int64_t* __restrict__ tile_prefix,
    int64_t* __restrict__ total, int64_t* __restrict__ offsets_end) {
  __shared__ int64_t buf[kScanThreads * kScanPer];
  __shared__ int64_t wt[33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int64_t carry = 0;
  for (int64_t c0 = 0; c0 < T; c0 += kScanThreads * kScanPer) {
    const int64_t m = min((int64_t)kScanThreads * kScanPer, T - c0);
    for (int i = threadIdx.x; i < kScanThreads * kScanPer; i += kScanThreads)
      buf[i] = i < m ? tile_sum[c0 + i] : 0;
    __syncthreads();
    int64_t v[kScanPer];
    int64_t sum = 0;
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) {
      v[j] = buf[threadIdx.x * kScanPer + j];
      sum += v[j];
    }
    int64_t inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += y;
    }
    if (lane == 31) wt[warp] = inc;
    __syncthreads();
    if (warp == 0) {
      const int64_t t = wt[lane];
      int64_t ti = t;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(kFull, ti, o);
        if (lane >= o) ti += y;
      }
      wt[lane] = ti - t;
      if (lane == 31) wt[32] = ti;
    }
    __syncthreads();
    int64_t run = carry + wt[warp] + inc - sum;
#pragma unroll
    for (int j = 0; j < kScanPer; ++j) {
      buf[threadIdx.x * kScanPer + j] = run;
      run += v[j];
    }
    carry += wt[32];
    __syncthreads();
    for (int i = threadIdx.x; i < m; i += kScanThreads) tile_prefix[c0 + i] = buf[i];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *total = carry;
    *offsets_end = carry;
  }
}


// The same scan in parallel, for at most kMaxSupers * kSuperTiles tiles:
// CTA b adds up every tile sum before its own kSuperTiles tiles (at most
// (kMaxSupers - 1) loads per thread, eight in flight) and scans its own;
// no CTA waits for another.
constexpr int kSuperTiles = 1024;
constexpr int kMaxSupers = 64;

__global__ void __launch_bounds__(kSuperTiles) tile_scan_par_kernel(
    const int64_t* __restrict__ tile_sum, int64_t T, int64_t* __restrict__ tile_prefix,
    int64_t* __restrict__ total, int64_t* __restrict__ offsets_end) {
  __shared__ int64_t wt[33];
  __shared__ int64_t ws[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int b = blockIdx.x;
  int64_t before = 0;
#pragma unroll 8
  for (int j = 0; j < b; ++j) before += tile_sum[(int64_t)j * kSuperTiles + threadIdx.x];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) before += __shfl_xor_sync(kFull, before, o);
  if (lane == 0) ws[warp] = before;
  const int64_t i = (int64_t)b * kSuperTiles + threadIdx.x;
  const int64_t x = i < T ? tile_sum[i] : 0;
  int64_t inc = x;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int64_t y = __shfl_up_sync(kFull, inc, o);
    if (lane >= o) inc += y;
  }
  if (lane == 31) wt[warp] = inc;
  __syncthreads();
  if (warp == 0) {
    const int64_t t = wt[lane];
    int64_t ti = t;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(kFull, ti, o);
      if (lane >= o) ti += y;
    }
    wt[lane] = ti - t;
    if (lane == 31) wt[32] = ti;
  }
  __syncthreads();
  int64_t base = 0;
#pragma unroll 8
  for (int w = 0; w < kSuperTiles / 32; ++w) base += ws[w];
  if (i < T) tile_prefix[i] = base + wt[warp] + inc - x;
  if (b == (int)gridDim.x - 1 && threadIdx.x == 0) {
    *total = base + wt[32];
    *offsets_end = base + wt[32];
  }
}

}  // namespace
}  // namespace hdda
