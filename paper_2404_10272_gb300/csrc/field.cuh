// field.cuh -- the Gaussian-blob field and the front-to-back accumulation
// shared by the compositor over stored samples (composite.cu) and the
// render-only path that expands runs on the fly (render.cu).
//
// Sec. 1: the densities and colours at a ray's sampled points are
// accumulated into its pixel, front to back.  The blob field stands in for
// the trained radiance field: sigma(x) = sum_g a_g exp(-|x - mu_g|^2 /
// (2 s_g^2)), colour = the sigma-weighted mean of the blobs' colours.
//
// Along one ray a blob is a Gaussian of the ray parameter alone: with t* the
// parameter of the ray's point nearest to mu and p its distance,
//     a exp(-|x(t) - mu|^2 / (2 s^2)) = 2^(log2 a - c p^2 - (k (t - t*))^2),
//     c = log2(e) / (2 s^2),  k = sqrt(c) |d|,
// so a sample costs two fused multiply-adds and one exp2 per blob before its
// four sums, where the distance in space took seven operations.  The three
// numbers per (ray, blob) are computed once per ray (setup_ray).
//
// Work split: a warp is four groups of eight lanes.  A group works on one
// ray at a time, 32 samples per step ("chunk"), four consecutive ones per
// lane; a group that has finished its ray takes the next ray of the warp's
// task, so the groups stay busy whatever the rays' lengths.
// Rays never share a chunk, hence one record per blob and chunk serves all
// of a group's samples, a 32-sample stretch of one ray meets few blobs it
// does not need, the colour sums stay in registers until the ray ends, and a
// scan over eight lanes (three steps) turns the samples' optical depths into
// transmittances.
//
// Blob culling, in two stages.  setup_ray keeps the blobs within reach
// (kCullSigmas standard deviations, plus a margin for binary32 rounding) of
// the ray's line; cull_chunk keeps those whose reach along the ray meets the
// chunk's parameter range.  So no blob within kCullSigmas s of a sample is
// dropped; a dropped one weighs below a * exp(-kCullSigmas^2 / 2) = a *
// e^-24.5, about 2e-11 of its amplitude.  Amplitudes must be non-negative
// (their logarithm is taken).
//
// What bounds it: instruction issue and latency (67 % of cycles issue at 24
// warps per SM).  36 % of the instructions are the blob loop, the rest is per
// chunk (listing, range, opacities, scan) and per ray (records).  Against two
// samples per lane of whichever rays come next, with distances in space and
// colours scanned per chunk, the compositor went from 432 to 308 us on an 800 x
// 800 object frame of 64 blobs and from 864 to 658 on a 1245 x 825 unbounded one.
// Tried, at 64 blobs when they took 297 and 1460 (another camera): four lanes per
// ray with eight samples each (a quarter fewer instructions, but 14 warps per SM:
// 20 % slower), 16 lanes' worth of registers saved by loading behind the blob
// loop (12 % slower), 7 CTAs per SM (spills, 15 % slower), CTAs of 8 to 16 tasks
// that their warps take in turn (5 to 10 % slower), groups refilled only when
// several are idle (0 to 5 % slower).  The layout's offsets as a kernel parameter
// instead of sums of its sizes: fewer spills, 3 % slower.
//
// Rounding.  Ray parameters are taken relative to a base parameter near the
// blobs (make_ray_rec), where the base point is rounded once, so t* and p carry
// the rounding of coordinates near the blobs, not of the origin's.  Every
// product-sum is an explicit fused multiply-add, so the arithmetic does not
// depend on the translation unit's contraction flags.
#pragma once

#include <cmath>

#include "hdda_internal.cuh"

namespace hdda {
namespace {

constexpr int kMaxGauss = 256;
constexpr float kCullSigmas = 7.f;
constexpr unsigned kFieldFull = 0xffffffffu;
constexpr int kGroupLanes = 8;                       // lanes that share a ray
constexpr int kGroups = 32 / kGroupLanes;            // rays a warp has in work
constexpr int kPerLane = 4;                          // consecutive samples of a lane
constexpr int kPairs = kPerLane / 2;
constexpr unsigned kLeaders = 0xffffffffu / ((1u << kGroupLanes) - 1u);  // the groups' first lanes
constexpr int kChunk = kGroupLanes * kPerLane;       // samples of one ray per step
constexpr float kLog2e = 1.4426950408889634f;

// The blobs as setup_ray reads them, two per lane, w lanes at a time (w = 32; 8 for
// kFew): pair p holds blobs b = (p / w) * 2 w + p % w and b + w in four arrays over
// the pairs (16 bytes per lane and load, consecutive lanes consecutive): {-mu_x,
// -mu_y}, {-mu_z, c}, {log2 a, sqrt(c)} and sqrt(c) (kCullSigmas s + margin),
// each as both blobs' values.
__host__ __device__ inline int field_pairs(int G) { return (G + 63) / 64 * 32; }
constexpr uint32_t kPairBytes = 3 * sizeof(float4) + sizeof(float2);

// A ray as setup_ray reads it: base point and base parameter, direction e = s d
// and 1 / |e|^2 (dir_scale); beside it a RayLen.
struct RayRec {
  float4 base;  // o + tb d, tb
  float4 dir;   // e, 1 / |e|^2
};

// What else a ray keeps.
struct __align__(16) RayLen {
  float len, margin;  // |e|; the rounding margin of distances to its line
  float half;         // 1 / (2 s): from half a parameter along e to one along d
  union {
    float T;          // a faint ray's transmittance (faint_chunk)
    int next_w;       // render.cu: the samples of the ray's next round
  };
};

// Dynamic shared memory of a compositing CTA of `warps` warps over G blobs,
// tasks of R rays per warp: the blobs in pairs; [G + 1] colours (the last one black,
// for padding) and the mean of the blobs' centres; then per warp [R] RayRec,
// [R] RayLen and, per group, room for `cap`
// records {k / 2, b = -k t*, c p^2 - log2 a, half-width | blob index} (and an
// empty one behind them, for padding), as many list entries {offset of a
// record, offset of its colour}, and `ring` factors of a faint ray.
//
// Up to kAllBlobs blobs every one has a record in every group.  A larger field
// would leave too few warps on an SM that way; there a group has room for about
// half of them (99 % of the rays of an object or an unbounded frame are within
// reach of less), and a ray within reach of more takes each chunk in passes
// (FieldWarp::more, kMany).  Shared memory then lets at most five CTAs on an SM
// from 160 blobs on, so the kernels have the registers of five (96): at 80 they
// spilled 110 to 160 bytes.  With room for 5/8 and 80 registers, and so (us): 128
// blobs, object frame 550 and 477, unbounded 1125 and 943; 200 blobs 996 and 741,
// 2088 and 1486; 256 blobs 1235 and 1016, 2608 and 2085.  (Distances in space,
// without records, took 661 and 1161, 1002 and 1689, 1356 and 2403.)
constexpr int kAllBlobs = 64;

// Up to kFewBlobs blobs the compositor's groups each set up their own ray (kFew).
constexpr int kFewBlobs = 32;

enum FieldForm { kFew, kSome, kMany };

struct FieldLayout {
  uint32_t col, warp0, per_warp, len, recs, list, ring, group, bytes;
  int cap;
};

// `ring`: factors of faint rays kept per group.
template <int kRoom64>
__host__ __device__ inline FieldLayout field_layout(int G, int warps, int R, int ring) {
  FieldLayout L;
  L.cap = G <= kAllBlobs ? G : (kRoom64 * G / 64 > kAllBlobs ? kRoom64 * G / 64 : kAllBlobs);
  L.col = (uint32_t)field_pairs(G) * kPairBytes;
  L.warp0 = L.col + ((uint32_t)G + 2u) * sizeof(float4);
  L.len = (uint32_t)R * sizeof(RayRec);
  L.recs = L.len + (uint32_t)R * sizeof(RayLen);
  L.list = ((uint32_t)L.cap + 1u) * sizeof(float4);
  L.ring = L.list + (((uint32_t)L.cap + 1u) & ~1u) * sizeof(uint2);  // lists are padded to even
  L.group = L.ring + (uint32_t)ring * sizeof(float);
  L.per_warp = L.recs + kGroups * L.group;
  L.bytes = L.warp0 + (uint32_t)warps * L.per_warp;
  return L;
}

// Stages `G` blobs of 8 floats {mu[3], s, a, rgb[3]} (block-wide; the caller
// synchronises the block afterwards).
template <int kForm>
__device__ __forceinline__ void stage_blobs(unsigned char* smem, const FieldLayout& L,
                                            const float* __restrict__ field, int G) {
  float* tab = reinterpret_cast<float*>(smem);
  const int np = field_pairs(G);
  float4* col = reinterpret_cast<float4*>(smem + L.col);
  for (int i = threadIdx.x; i < G; i += blockDim.x) {
    const float* f = field + 8 * i;
    const float s = f[3], c = kLog2e / (2.f * s * s), rc = sqrtf(c);
    const float reach = kCullSigmas * s;
    const float mu_max = fmaxf(fabsf(f[0]), fmaxf(fabsf(f[1]), fabsf(f[2])));
    constexpr int w = kForm == kFew ? kGroupLanes : 32;
    const int p = i / (2 * w) * w + i % w, h = i / w & 1;  // the pair, its blob
    float *xy = tab + 4 * p + h, *zc = xy + 4 * np, *ak = zc + 4 * np;
    xy[0] = -f[0];
    xy[2] = -f[1];
    zc[0] = -f[2];
    zc[2] = c;
    ak[0] = log2f(f[4]);
    ak[2] = rc;
    tab[12 * np + 2 * p + h] = rc * (reach + 2e-5f * (1.f + mu_max + reach));
    col[i] = make_float4(f[5], f[6], f[7], 0.f);
  }
  if (threadIdx.x >= blockDim.x - 32) {  // the mean of the centres: a warp without blobs up to 96
    const int lane = threadIdx.x & 31;
    float m[3] = {0.f, 0.f, 0.f};
    for (int i = lane; i < G; i += 32)
#pragma unroll
      for (int k = 0; k < 3; ++k) m[k] += field[8 * i + k];
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m[k] += __shfl_xor_sync(kFieldFull, m[k], o);
    if (lane == 0) {
      const float s = 1.f / (float)max(G, 1);
      col[G] = make_float4(0.f, 0.f, 0.f, 0.f);
      col[G + 1] = make_float4(s * m[0], s * m[1], s * m[2], 0.f);
    }
  }
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

__device__ __forceinline__ float2 splat(float v) { return make_float2(v, v); }

// (1 - exp(-tau)) / tau for |tau| < 1/2: the Taylor series sum_k (-tau)^k /
// (k+1)!, k = 0..7, in Horner form (the first term left out, (tau/2)^8 / 9! <
// 1.1e-8, is far below binary32 rounding), which keeps small opacities
// accurate to a few ulp.
__device__ __forceinline__ float2 opacity_series2(float2 tau) {
  const float2 x = make_float2(-tau.x, -tau.y);
  float2 p = splat(1.f / 40320.f);  // 1/8!
  p = __ffma2_rn(p, x, splat(1.f / 5040.f));
  p = __ffma2_rn(p, x, splat(1.f / 720.f));
  p = __ffma2_rn(p, x, splat(1.f / 120.f));
  p = __ffma2_rn(p, x, splat(1.f / 24.f));
  p = __ffma2_rn(p, x, splat(1.f / 6.f));
  p = __ffma2_rn(p, x, splat(0.5f));
  return __ffma2_rn(p, x, splat(1.f));
}

// One group's ray in work (the same values on the group's lanes except the
// lane's colour sums).
struct RayAcc {
  float S;            // optical depth so far, times log2(e)
  float T;            // faint ray: transmittance so far (faint_product)
  float2 r, g, b;     // this lane's colour sums (two halves, added at the end)
};

__device__ __forceinline__ void acc_clear(RayAcc& a) {
  a.S = 0.f;
  a.T = 1.f;
  a.r = a.g = a.b = splat(0.f);
}

// A power of two that brings a direction of extreme length to one whose square
// is a normal number; 1 for lengths from 1e-15 to 1e15.
__device__ __forceinline__ float dir_scale(const float d[3]) {
  const float m = fmaxf(fabsf(d[0]), fmaxf(fabsf(d[1]), fabsf(d[2])));
  if (!(m > 0.f) || (m > 1e-15f && m < 1e15f)) return 1.f;
  const int x = min(max((int)(__float_as_uint(m) >> 23) - 127, -126), 126);
  return __uint_as_float((uint32_t)(127 - x) << 23);
}

// Fills the RayRec and RayLen of one ray (one lane per ray) whose samples lie
// between ta and te.
//
// The base parameter is where the ray passes nearest to the blobs' mean centre.
// Parameters and distances are exact to the rounding of numbers of the size of
// their difference from the base, and most of a field's weight lies near its
// middle, while a ray's samples may reach far beyond it (a four-level cascade:
// with the middle of the samples as the base the error against binary64 was up
// to 1.7 times as large).
__device__ __forceinline__ void make_ray_rec(RayRec* rr, RayLen* rl, const unsigned char* smem,
                                             const FieldLayout& L, int G, const float o[3],
                                             const float d[3], float ta, float te) {
  const float4 m = reinterpret_cast<const float4*>(smem + L.col)[G + 1];
  const float s = dir_scale(d);
  const float e[3] = {d[0] * s, d[1] * s, d[2] * s};
  const float w = fmaf(m.x - o[0], e[0], fmaf(m.y - o[1], e[1], (m.z - o[2]) * e[2]));
  const float ee = fmaf(e[0], e[0], fmaf(e[1], e[1], e[2] * e[2]));
  float tb = fminf(fmaxf(__fdividef(w, ee) * s, fminf(ta, te)), fmaxf(ta, te));
  if (!(fabsf(tb) < INFINITY)) tb = 0.f;
  float b[3];
  float om = 0.f, bm = 0.f;
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    b[c] = fmaf(tb, d[c], o[c]);
    om = fmaxf(om, fabsf(o[c]));
    bm = fmaxf(bm, fabsf(b[c]));
  }
  const bool moves = ee > 0.f;
  rr->base = make_float4(b[0], b[1], b[2], tb);
  rr->dir = make_float4(e[0], e[1], e[2], moves ? 1.f / ee : 0.f);
  rl->len = moves ? sqrtf(ee) : 0.f;
  rl->margin = 2e-5f * (om + bm);
  rl->half = 0.5f / s;
  rl->T = 1.f;
}

// sqrt(x), approximately, rounded up and its low 8 bits replaced by a blob's
// index: at least 2^8 units in the last place are added, the square root's own
// error is a few.
__device__ __forceinline__ float half_width(float x, int q) {
  float h;
  asm("sqrt.approx.f32 %0, %1;" : "=f"(h) : "f"(x));
  h = fminf(h, 1e30f);
  return __uint_as_float(((__float_as_uint(h) + 0x1ffu) & ~0xffu) | (uint32_t)q);
}

// The blobs within reach of the ray's line, as records in `rec`; returns
// their number.  With kMany: from blob q0 (a multiple of 64) on, as many whole
// steps of 64 blobs as `cap` records hold, q0 advancing past the blobs looked
// at.  Called by the whole warp, two blobs per lane and step in packed
// arithmetic (the ray's samples need not ascend, so the line is not cut off at
// its first and last one: cutting it measured no faster either).  t* is found,
// the vector to the blob taken there, and both are refined once from that
// vector, so their rounding is that of the distance, not of the span from the
// base point.  A blob per lane took 304 us on the object frame, 1482 on the
// unbounded one and 1907 on a 1080p render-only one; two take 292, 1455, 1819.
// With kFew every group's eight lanes work on its own ray, where `on`.
template <int kForm>
__device__ __forceinline__ int setup_ray(const unsigned char* smem, int G, const RayRec* rr,
                                         const RayLen* rl, float4* rec, int cap, int& q0,
                                         bool on = true) {
  constexpr int w = kForm == kFew ? kGroupLanes : 32;  // lanes on the ray
  const float4* tab = reinterpret_cast<const float4*>(smem);
  const int lane = threadIdx.x & (w - 1), first = (threadIdx.x & 31) - lane, np = field_pairs(G);
  const unsigned mine = (kFieldFull >> (32 - w)) << first;
  const float4 B = rr->base, D = rr->dir;
  const float4 len = *reinterpret_cast<const float4*>(rl);  // |e|, margin, 1 / (2 s)
  const float2 dx = splat(D.x), dy = splat(D.y), dz = splat(D.z), nw = splat(-D.w);
  int n = 0;
  for (; q0 < G; q0 += 2 * w) {
    const int p = (q0 >> 1) + lane;
    const float4 XY = tab[p], ZC = tab[np + p], AK = tab[2 * np + p];
    const float2 reach = reinterpret_cast<const float2*>(tab + 3 * np)[p];
    const float2 c = make_float2(ZC.z, ZC.w), rc = make_float2(AK.z, AK.w);
    const float2 wx = __fadd2_rn(splat(B.x), make_float2(XY.x, XY.y));
    const float2 wy = __fadd2_rn(splat(B.y), make_float2(XY.z, XY.w));
    const float2 wz = __fadd2_rn(splat(B.z), make_float2(ZC.x, ZC.y));
    float2 ts = __fmul2_rn(nw, __ffma2_rn(wx, dx, __ffma2_rn(wy, dy, __fmul2_rn(wz, dz))));
    float2 qx = __ffma2_rn(ts, dx, wx), qy = __ffma2_rn(ts, dy, wy), qz = __ffma2_rn(ts, dz, wz);
    const float2 de = __fmul2_rn(nw, __ffma2_rn(qx, dx, __ffma2_rn(qy, dy, __fmul2_rn(qz, dz))));
    ts = __fadd2_rn(ts, de);
    qx = __ffma2_rn(de, dx, qx);
    qy = __ffma2_rn(de, dy, qy);
    qz = __ffma2_rn(de, dz, qz);
    const float2 cp2 = __fmul2_rn(c, __ffma2_rn(qx, qx, __ffma2_rn(qy, qy, __fmul2_rn(qz, qz))));
    const float2 hl = __ffma2_rn(rc, splat(len.y), reach);
    const float2 lim2 = __ffma2_rn(hl, hl, make_float2(-cp2.x, -cp2.y));
    const float2 k = __fmul2_rn(rc, splat(len.x));
    const float2 hk = __fmul2_rn(splat(len.z), k), b = __fmul2_rn(make_float2(-k.x, -k.y), ts);
    const float2 e = __fadd2_rn(cp2, make_float2(-AK.x, -AK.y));
    const int q = q0 + lane;
    const bool near0 = on && lim2.x >= 0.f && q < G, near1 = on && lim2.y >= 0.f && q + w < G;
    const unsigned ball0 = __ballot_sync(kFieldFull, near0) & mine;
    const unsigned ball1 = __ballot_sync(kFieldFull, near1) & mine;
    const int n0 = __popc(ball0), kept = n0 + __popc(ball1);
    if (kForm == kMany && n + kept > cap) break;  // uniform; one step always fits
    const unsigned below = (1u << (threadIdx.x & 31)) - 1u;
    if (near0)
      rec[n + __popc(ball0 & below)] = make_float4(hk.x, b.x, e.x, half_width(lim2.x, q));
    if (near1)
      rec[n + n0 + __popc(ball1 & below)] = make_float4(hk.y, b.y, e.y, half_width(lim2.y, q + w));
    n += kept;
  }
  return n;
}

// The four sums over the blobs, for each of the lane's samples: density and
// density-weighted colour.
struct BlobSums {
  float2 s[kPairs], r[kPairs], g[kPairs], b[kPairs];
};

// Adds the listed blobs at the lane's samples, given as doubled relative
// parameters t = (t0 - tb) + (t1 - tb).
__device__ __forceinline__ void sum_blobs(const unsigned char* smem, uint32_t list, int len,
                                          const float2 t[kPairs], BlobSums& S) {
  for (int i = 0; i < len; i += 2) {
    const uint4 e = *reinterpret_cast<const uint4*>(smem + list + 8u * i);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const float4 R = *reinterpret_cast<const float4*>(smem + (j ? e.z : e.x));
      const float4 C = *reinterpret_cast<const float4*>(smem + (j ? e.w : e.y));
#pragma unroll
      for (int h = 0; h < kPairs; ++h) {
        const float2 u = __ffma2_rn(t[h], splat(R.x), splat(R.y));
        const float2 v = __ffma2_rn(u, u, splat(R.z));
        const float2 w = make_float2(ex2_approx(-v.x), ex2_approx(-v.y));
        S.s[h] = __fadd2_rn(S.s[h], w);
        S.r[h] = __ffma2_rn(w, splat(C.x), S.r[h]);
        S.g[h] = __ffma2_rn(w, splat(C.y), S.g[h]);
        S.b[h] = __ffma2_rn(w, splat(C.z), S.b[h]);
      }
    }
  }
}

// A warp's groups over one task: where their shared memory is, and each
// group's blob records (the same values on the group's lanes).
template <int kForm>
struct FieldWarp {
  unsigned char* smem;
  uint32_t recs;  // the group's records
  int nc;         // their number
  int next;       // kMany: blobs below it are in the records or were; below G: there are more
  int most;       // the largest nc of the warp's groups

  static __device__ __forceinline__ uint32_t rays_at(const FieldLayout& L) {
    return L.warp0 + (threadIdx.x >> 5) * L.per_warp;
  }

  __device__ __forceinline__ RayRec* rays(const FieldLayout& L) const {
    return reinterpret_cast<RayRec*>(smem + rays_at(L));
  }

  __device__ __forceinline__ RayLen* lens(const FieldLayout& L) const {
    return reinterpret_cast<RayLen*>(smem + rays_at(L) + L.len);
  }

  __device__ __forceinline__ void init(unsigned char* smem_, const FieldLayout& L) {
    smem = smem_;
    const int lane = threadIdx.x & 31;
    recs = rays_at(L) + L.recs + (uint32_t)(lane / kGroupLanes) * L.group;
    // the group's last record is empty, for padding
    if ((lane & (kGroupLanes - 1)) == 0)
      *reinterpret_cast<float4*>(smem + recs + L.list - sizeof(float4)) =
          make_float4(0.f, 0.f, INFINITY, 0.f);
    release();
    most = 0;
  }

  // The group has no ray.
  __device__ __forceinline__ void release() {
    nc = 0;
    if constexpr (kForm == kMany) next = kMaxGauss;
  }

  // The records of group g for ray i of the task, from blob q0 on.
  __device__ __forceinline__ void setup(const FieldLayout& L, int G, int g, int i, int q0 = 0) {
    const uint32_t rec = rays_at(L) + L.recs + (uint32_t)g * L.group;
    const int m = setup_ray<kForm>(smem, G, rays(L) + i, lens(L) + i,
                                   reinterpret_cast<float4*>(smem + rec), L.cap, q0);
    if ((int)(threadIdx.x & 31) / kGroupLanes == g) {
      nc = m;
      if constexpr (kForm == kMany) next = q0;
    }
  }

  // kFew: the records of every group whose ray, `ray` of the task, is new (`on`).
  // Rays of a few samples often end together: 640,000 of two samples took 214 us
  // over 16 blobs and 226 over 32 with the whole warp on one group after the
  // other, 171 and 199 so (of 20 samples over 32 blobs 306 either way).
  __device__ __forceinline__ void setup_own(const FieldLayout& L, int G, bool on, int ray) {
    const int i = max(ray, 0);
    int q0 = 0;
    const int m = setup_ray<kForm>(smem, G, rays(L) + i, lens(L) + i,
                                   reinterpret_cast<float4*>(smem + recs), L.cap, q0, on);
    if (on) nc = m;
  }

  // After setups: they are visible, `most` is up to date.
  __device__ __forceinline__ void ready() {
    most = (int)__reduce_max_sync(kFieldFull, (unsigned)nc);
    __syncwarp();
  }

  // Lists the group's blobs whose reach meets the parameter range [lo, hi]
  // (doubled and relative to the base) and pads every group's list with empty
  // records to the longest one's length, rounded up to even, which it returns;
  // `kept` receives the group's own.
  __device__ __forceinline__ int cull(const FieldLayout& L, int G, float lo, float hi, int& kept) {
    const int lane = threadIdx.x & 31, gl = lane & (kGroupLanes - 1);
    const unsigned mine = ((1u << kGroupLanes) - 1u) << (lane & ~(kGroupLanes - 1));
    const unsigned below = mine & ((1u << lane) - 1u);
    uint2* out = reinterpret_cast<uint2*>(smem + recs + L.list);
    const uint32_t col = L.col;
    int m = 0;
    uint32_t at = recs + 16u * gl;
    for (int i0 = 0; i0 < most; i0 += kGroupLanes, at += 16u * kGroupLanes) {
      bool near = false;
      float h = 0.f;
      if (i0 + gl < nc) {
        const float4 R = *reinterpret_cast<const float4*>(smem + at);
        h = R.w;
        near = fmaf(lo, R.x, R.y) <= h && fmaf(hi, R.x, R.y) >= -h;
      }
      const unsigned ball = __ballot_sync(kFieldFull, near);
      if (near)
        out[m + __popc(ball & below)] = make_uint2(at, col + 16u * (__float_as_uint(h) & 0xffu));
      m += __popc(ball & mine);
    }
    kept = m;
    const int len = ((int)__reduce_max_sync(kFieldFull, (unsigned)m) + 1) & ~1;
    const int least = (int)__reduce_min_sync(kFieldFull, (unsigned)m);
    for (int p0 = least; p0 < len; p0 += kGroupLanes) {  // uniform
      const int p = p0 + gl;
      if (p >= m && p < len)
        out[p] = make_uint2(recs + L.list - (uint32_t)sizeof(float4), col + 16u * (uint32_t)G);
    }
    __syncwarp();
    return len;
  }

  // kMany: the blobs that did not fit the groups' records, for the chunk in
  // work; then the records start over.  `ray` is the group's ray in the task.
  __device__ __forceinline__ void more(const FieldLayout& L, int G, int ray, float lo, float hi,
                                       const float2 t[kPairs], BlobSums& S, int& kept) {
    const int lane = threadIdx.x & 31, nc0 = nc;
    const unsigned multi = __ballot_sync(kFieldFull, next < G);
    for (unsigned todo = multi; todo;) {  // uniform
      if (!((todo >> lane) & 1u)) nc = 0;
      again(L, G, todo, ray, false);
      int m;
      const int len = cull(L, G, lo, hi, m);
      kept += m;
      sum_blobs(smem, recs + L.list, len, t, S);
      todo = __ballot_sync(kFieldFull, ((todo >> lane) & 1u) && next < G);
    }
    if (!multi) return;
    if (!((multi >> lane) & 1u)) nc = nc0;
    again(L, G, multi, ray, true);
  }

  // Sets up the groups in `lanes` for their next blobs, or from the first one.
  __device__ __forceinline__ void again(const FieldLayout& L, int G, unsigned lanes, int ray,
                                        bool restart) {
    __syncwarp();  // the records may be overwritten
    for (unsigned l = lanes & kLeaders; l; l &= l - 1) {
      const int f = __ffs(l) - 1;
      const int i = __shfl_sync(kFieldFull, ray, f), q0 = __shfl_sync(kFieldFull, next, f);
      setup(L, G, f / kGroupLanes, i, restart ? 0 : q0);
    }
    ready();
  }
};

__device__ __forceinline__ void sums_clear(BlobSums& S) {
#pragma unroll
  for (int h = 0; h < kPairs; ++h) S.s[h] = S.r[h] = S.g[h] = S.b[h] = splat(0.f);
}

// The limit, in optical depth times log2(e), below which a ray is faint: its
// transmittance is above 0.98.
//
// A ray's transmittance comes from the sum of its optical depths, chunk by
// chunk: a product of (1 - alpha) rounds every factor to a multiple of 6e-8 and
// every product again.  Error against binary64 (2-norm, relative) as a product
// and as a sum: 1.9e-7 and 1.1e-7 on object frames, 6.1e-7 and 2.7e-7 on
// unbounded ones.  Only the lane's own four samples are a product: with an
// exponential for each, the compositor was 7 % slower for the same error.
// A faint ray's opacity is the exception: it is 1 minus a product of (1 -
// alpha) in a fixed order, that of faint_chunk for stored samples and up to
// kAllBlobs blobs, else that of faint_product, chunk after chunk.  The roundings
// above are up to 2e-4 of so small an opacity, and another order, or the sum,
// would move frames that programs have stored by as much; the products keep them.
constexpr float kFaintDepth = 0.029146346f;  // -log2(0.98)
constexpr float kNoDepth = 1.f / (1 << 26);  // below it every 1 - alpha of a ray is 1

// Accumulates a chunk's samples of lengths dt = t1 - t0 (0 for padding) front
// to back: adds to the group's optical depth and to the lane's colour sums.
// f receives the samples' 1 - alpha.  Returns whether the group's ray (`ray` >=
// 0) is still faint.
__device__ __forceinline__ bool shade_chunk(BlobSums& B, const float2 dt[kPairs], int ray,
                                            RayAcc& acc, float2 f[kPairs]) {
  const int gl = threadIdx.x & (kGroupLanes - 1);
  float2(&tau)[kPairs] = B.s;  // densities, now optical depths
  const float2(&cr)[kPairs] = B.r, (&cg)[kPairs] = B.g, (&cb)[kPairs] = B.b;
#pragma unroll
  for (int h = 0; h < kPairs; ++h) tau[h] = __fmul2_rn(tau[h], dt[h]);
  // depth before the lane's first sample: the ray's so far, the lanes before
  float inc = kLog2e * ((tau[0].x + tau[0].y) + (tau[1].x + tau[1].y));
#pragma unroll
  for (int o = 1; o < kGroupLanes; o <<= 1) {
    const float y = __shfl_up_sync(kFieldFull, inc, o, kGroupLanes);
    if (gl >= o) inc += y;
  }
  float before = __shfl_up_sync(kFieldFull, inc, 1, kGroupLanes);
  before = gl ? acc.S + before : acc.S;
  acc.S += __shfl_sync(kFieldFull, inc, kGroupLanes - 1, kGroupLanes);
  // opacities, and the opacity per density
  float2 al[kPairs], op[kPairs];
  float tm = 0.f;
#pragma unroll
  for (int h = 0; h < kPairs; ++h) {
    const float2 p = opacity_series2(tau[h]);
    al[h] = __fmul2_rn(tau[h], p);
    op[h] = __fmul2_rn(dt[h], p);
    tm = fmaxf(tm, fmaxf(fabsf(tau[h].x), fabsf(tau[h].y)));
  }
  if (!(tm < 0.5f)) {  // 1 - exp2: its absolute error of a few 1e-8 is small against >= 0.39
#pragma unroll
    for (int h = 0; h < kPairs; ++h) {
      // (1 - exp(-tau)) / sigma = (1 - exp(-tau)) dt / tau
      if (!(fabsf(tau[h].x) < 0.5f)) {
        al[h].x = 1.f - ex2_approx(-kLog2e * tau[h].x);
        op[h].x = __fdividef(al[h].x * dt[h].x, tau[h].x);
      }
      if (!(fabsf(tau[h].y) < 0.5f)) {
        al[h].y = 1.f - ex2_approx(-kLog2e * tau[h].y);
        op[h].y = __fdividef(al[h].y * dt[h].y, tau[h].y);
      }
    }
  }
  // transmittance before each sample: of the depth before the lane, times the
  // lane's earlier samples' 1 - alpha
  float run = ex2_approx(-before);
#pragma unroll
  for (int h = 0; h < kPairs; ++h) {
    f[h] = __ffma2_rn(al[h], splat(-1.f), splat(1.f));
    const float mid = run * f[h].x;
    const float2 g = __fmul2_rn(op[h], make_float2(run, mid));
    run = mid * f[h].y;
    acc.r = __ffma2_rn(g, cr[h], acc.r);
    acc.g = __ffma2_rn(g, cg[h], acc.g);
    acc.b = __ffma2_rn(g, cb[h], acc.b);
  }
  return ray >= 0 && acc.S < kFaintDepth;
}

// A finished ray's opacity, from its optical depth or, faint, its transmittance T.
__device__ __forceinline__ float ray_opacity(float S, float T) {
  return 1.f - (S < kFaintDepth ? T : ex2_approx(-S));
}

// The transmittance of faint rays (`faint` on the group's lanes) behind a chunk,
// in the chunk's order: the lane's four factors in turn, then a tree over the
// group's lanes.  Called by the whole warp.
__device__ __forceinline__ void faint_product(const float2 f[kPairs], bool faint, RayAcc& acc) {
  if (!__any_sync(kFieldFull, faint && !(fabsf(acc.S) < kNoDepth))) return;
  float m = f[0].x * f[0].y;
#pragma unroll
  for (int h = 1; h < kPairs; ++h) {
    m *= f[h].x;
    m *= f[h].y;
  }
#pragma unroll
  for (int o = 1; o < kGroupLanes; o <<= 1) m *= __shfl_xor_sync(kFieldFull, m, o);
  acc.T *= m;
}

// The product for stored samples and up to kAllBlobs blobs: the samples of four
// rays (ray / 4), each 64 in a row, are a segment; a segment's samples of one
// ray are a balanced tree over the pairs of places, counted back from the last
// whole pair, times a last single sample; segments multiply in order.  Between
// chunks the factors wait in a ring of 96 per group in shared memory.  The
// limit: with 0.998 three of 81 random unbounded frames differ by 2.1e-5
// (2-norm, relative) from the same product order throughout, with 0.98 none by more
// than 7.5e-6.
constexpr int kFaintRays = 4;
constexpr int kRing = 96;  // a segment and a chunk beyond it

// One chunk of every group, called by the whole warp: `f` the lane's factors (1
// for padding), `q` its first position (a multiple of 4), `on` whether the
// group's ray, `ray` of positions [beg, end), is faint, `S` its depth behind
// the chunk; lane i's `my_beg` is the first position of ray i.  The product so
// far stays in rl->T (it takes no register of the blob loop's).
__device__ __forceinline__ void faint_chunk(float* ring, RayLen* rl, const float2 f[kPairs],
                                            bool on, int ray, int q, int beg, int end, int my_beg,
                                            float S) {
  static_assert(kPairs == 2, "one 16-byte store per lane");
  const int gl = threadIdx.x & (kGroupLanes - 1);
  if (on)
    *reinterpret_cast<float4*>(ring + (unsigned)q % kRing) =
        make_float4(f[0].x, f[0].y, f[1].x, f[1].y);
  on = on && !(fabsf(S) < kNoDepth);
  // where every factor so far is 1 (few blobs, rays that miss them) no product is needed
  // (unbounded frame without blobs: 458 -> 349 us, with four 519 -> 406)
  if (!__any_sync(kFieldFull, on)) return;
  const int task = __shfl_sync(kFieldFull, my_beg, ray & ~(kFaintRays - 1));
  __syncwarp();
  const int base = q - kPerLane * gl;  // the chunk's positions
  const int to = min(base + kChunk, end);
  int at = max(beg, base);  // a position of the segment in work
  float F = rl->T;
  __syncwarp();
#pragma unroll 1
  for (int turn = 0; turn < 2; ++turn) {  // a chunk ends two segments at most
    const int c0 = task + ((at - task) & ~63);  // its 64 places
    const int s0 = max(c0, beg), s1 = min(c0 + 64, end);
    const bool full = on && at < to && s1 <= to;  // it ends in this chunk
    if (!__any_sync(kFieldFull, full)) break;
    const int n = (s1 - c0) & ~1;  // places up to the last whole pair
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int p = c0 + n - 2 - 2 * (4 * gl + i);  // the pair's first position
      v[i] = 1.f;
      if (full && p + 1 >= s0) {
        const float y = ring[(unsigned)(p + 1) % kRing];
        v[i] = p >= s0 ? ring[(unsigned)p % kRing] * y : y;
      }
    }
    float m = (v[0] * v[1]) * (v[2] * v[3]);
#pragma unroll
    for (int o = 1; o < kGroupLanes; o <<= 1) m *= __shfl_xor_sync(kFieldFull, m, o);
    if (full) {
      F *= m;
      if ((s1 - c0) & 1) F *= ring[(unsigned)(s1 - 1) % kRing];
      at = s1;  // on to the next segment
    }
  }
  if (on) rl->T = F;  // the same value from the group's lanes
  __syncwarp();       // the ring may be overwritten
}

// A chunk's doubled relative parameters and lengths from its interval ends,
// and the group's range of the former.  `rel` is the lane's first position
// in the ray (negative before its first sample) and `count` the ray's
// samples: positions outside [0, count) become padding (length 0, a parameter
// within the range).  kAscend: the ray's samples ascend and the group's first
// one is one of them, so its first and last one bound the range.
template <bool kAscend>
__device__ __forceinline__ void chunk_params(const float2 a[kPairs], const float2 b[kPairs],
                                             float tb, int rel, int count, float2 t[kPairs],
                                             float2 dt[kPairs], float& lo, float& hi) {
  const float2 B = splat(-tb);
#pragma unroll
  for (int h = 0; h < kPairs; ++h) {
    t[h] = __fadd2_rn(__fadd2_rn(a[h], B), __fadd2_rn(b[h], B));
    dt[h] = make_float2(b[h].x - a[h].x, b[h].y - a[h].y);
  }
  if constexpr (kAscend) lo = __shfl_sync(kFieldFull, t[0].x, 0, kGroupLanes);
  const bool part = rel < 0 || rel + kPerLane > count;
  const bool any = __any_sync(kFieldFull, part);
  if (any) {  // uniform
    const float pad = kAscend ? lo : NAN;  // NaN: left out of the range
#pragma unroll
    for (int h = 0; h < kPairs; ++h) {
      const bool i0 = (unsigned)(rel + 2 * h) < (unsigned)count;
      const bool i1 = (unsigned)(rel + 2 * h + 1) < (unsigned)count;
      t[h] = make_float2(i0 ? t[h].x : pad, i1 ? t[h].y : pad);
      dt[h] = make_float2(i0 ? dt[h].x : 0.f, i1 ? dt[h].y : 0.f);
    }
  }
  hi = fmaxf(t[0].x, t[0].y);
#pragma unroll
  for (int h = 1; h < kPairs; ++h) hi = fmaxf(hi, fmaxf(t[h].x, t[h].y));
  if constexpr (kAscend) {
    const int last = count - 1 - rel + kPerLane * (threadIdx.x & (kGroupLanes - 1));
    hi = __shfl_sync(kFieldFull, hi, min(last, kChunk - 1) / kPerLane, kGroupLanes);
  } else {
    lo = fminf(t[0].x, t[0].y);
#pragma unroll
    for (int h = 1; h < kPairs; ++h) lo = fminf(lo, fminf(t[h].x, t[h].y));
#pragma unroll
    for (int o = 1; o < kGroupLanes; o <<= 1) {
      lo = fminf(lo, __shfl_xor_sync(kFieldFull, lo, o));
      hi = fmaxf(hi, __shfl_xor_sync(kFieldFull, hi, o));
    }
    if (any) {
#pragma unroll
      for (int h = 0; h < kPairs; ++h) t[h] = make_float2(fmaxf(t[h].x, lo), fmaxf(t[h].y, lo));
    }
  }
}

// Writes the pixels of the groups whose ray is done (called by the whole
// warp): the colour sums are added up over the group's eight lanes, each pair
// of lanes ending with one channel.
// `T` is the transmittance of a faint ray.
__device__ __forceinline__ void finish_rays(const RayAcc& acc, float T, bool done, float* px) {
  static_assert(kGroupLanes == 8, "two lanes per channel");
  const int gl = threadIdx.x & (kGroupLanes - 1);
  const float r = acc.r.x + acc.r.y, g = acc.g.x + acc.g.y, b = acc.b.x + acc.b.y;
  const bool up = gl & 4, odd = gl & 2;
  // lanes 0-3 keep r and g, lanes 4-7 b; then lanes 0, 1 r, lanes 2, 3 g, lanes 4, 5 b
  float u = (up ? b : r) + __shfl_xor_sync(kFieldFull, up ? r : b, 4);
  const float v = (up ? 0.f : g) + __shfl_xor_sync(kFieldFull, up ? g : 0.f, 4);
  u = (odd ? v : u) + __shfl_xor_sync(kFieldFull, odd ? u : v, 2);
  u += __shfl_xor_sync(kFieldFull, u, 1);
  if (gl == 6) u = ray_opacity(acc.S, T);
  if (done && !(gl & 1)) px[gl >> 1] = u;
}

// Rays per warp task: tasks of 8 keep the four groups of a warp evenly busy
// (object frame of 640,000 rays: 285 us; 4 rays 300, 16 rays 294, 32 rays 344
// us); a small call is spread over the chip (9,216 rays, sampling included: 96
// us by 4 rays, 106 us by 8; 47,311 rays, render only: 107 and 118 us).
inline int field_task_rays(int64_t n) { return n >= 65536 ? 8 : 4; }

}  // namespace
}  // namespace hdda
