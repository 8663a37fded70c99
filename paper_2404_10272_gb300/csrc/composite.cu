// composite.cu -- front-to-back compositing of stored samples over a
// Gaussian-blob field (Sec. 1: the sampled points' densities and colours are
// accumulated into the pixel).  The blob field, its culling and the
// per-chunk accumulation are in field.cuh.
//
// Work split: a warp owns R consecutive rays (field_task_rays) and works on
// four of them at a time, one per group of eight lanes.  A ray's samples are
// a contiguous range of the CSR arrays; a group reads it 32 samples at a
// time, four consecutive ones per lane, from a position rounded down to a
// multiple of four so that a lane's values are 16-byte loads (plain loads
// when the arrays are not aligned, or at their very end).
#include "field.cuh"

namespace hdda {
namespace {

constexpr int kWarpsPerCta = 4;  // CTAs per SM: 6 by registers (80); up to 32 blobs 7 (72: object
                                 // frame over 16 blobs 228 -> 220 us); over 64, see kAllBlobs
// Records per group in 64ths of a field of many blobs.  Not 32: with that the form for up to 64
// blobs, which does not use it, is compiled with 28 bytes of spills instead of 4 and is 3 % slower
// (object frame 307 and 317 us); here 32 and 33 are equally fast.
constexpr int kRoom64 = 33;

// Blob evaluations (sample x kept blob), counted only while profiling.
__device__ unsigned long long g_blob_evals;

// The lane's values at positions q .. q + kPerLane - 1 of both arrays (kVec:
// the arrays and q are 16-byte aligned), where they belong to the ray [beg,
// end); `lim` bounds the arrays.
template <bool kVec>
__device__ __forceinline__ void load_lane(const float* __restrict__ t0, const float* __restrict__ t1,
                                          int q, int beg, int end, int lim, float2 a[kPairs],
                                          float2 b[kPairs]) {
  if (kVec && q + kPerLane <= lim) {
#pragma unroll
    for (int h = 0; h < kPairs; h += 2) {
      if (q + 2 * h < end) {
        const float4 x = __ldg(reinterpret_cast<const float4*>(t0 + q + 2 * h));
        const float4 y = __ldg(reinterpret_cast<const float4*>(t1 + q + 2 * h));
        a[h] = make_float2(x.x, x.y);
        a[h + 1] = make_float2(x.z, x.w);
        b[h] = make_float2(y.x, y.y);
        b[h + 1] = make_float2(y.z, y.w);
      }
    }
  } else {
#pragma unroll
    for (int h = 0; h < kPairs; ++h) {
      const int p = q + 2 * h;
      if (p >= beg && p < end) {
        a[h].x = __ldg(t0 + p);
        b[h].x = __ldg(t1 + p);
      }
      if (p + 1 >= beg && p + 1 < end) {
        a[h].y = __ldg(t0 + p + 1);
        b[h].y = __ldg(t1 + p + 1);
      }
    }
  }
}

template <bool kVec, int kForm>
__global__ void __launch_bounds__(kWarpsPerCta * 32, kForm == kMany ? 5 : kForm == kFew ? 7 : 6) composite_kernel(
    const float* __restrict__ ro, const float* __restrict__ rd, int64_t n, int R,
    const int64_t* __restrict__ offsets, const float* __restrict__ t0,
    const float* __restrict__ t1, const float* __restrict__ field, int G,
    float* __restrict__ rgba, bool count_evals) {
  extern __shared__ __align__(16) unsigned char smem[];  // field_layout
  const FieldLayout L = field_layout<kRoom64>(G, kWarpsPerCta, R, kForm == kMany ? 0 : kRing);
  stage_blobs<kForm>(smem, L, field, G);
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int grp = lane / kGroupLanes, gl = lane & (kGroupLanes - 1);
  const int64_t first = ((int64_t)blockIdx.x * kWarpsPerCta + wib) * R;
  if (first >= n) return;  // uniform per warp; no block barrier follows
  FieldWarp<kForm> fw;
  fw.init(smem, L);

  // lane i < R holds ray i's range, relative to the warp's first position
  // rounded down to a multiple of four (a task's samples fit in 32 bits)
  const int64_t r = first + lane;
  const bool has_ray = lane < R && r < n;
  const int64_t sb = has_ray ? __ldg(offsets + r) : 0, se = has_ray ? __ldg(offsets + r + 1) : 0;
  const int64_t wbase = __shfl_sync(kFieldFull, sb, 0) & ~(int64_t)3;
  const int my_beg = (int)(sb - wbase), my_end = (int)(se - wbase);
  const int lim = (int)min(__ldg(offsets + n) - wbase, (int64_t)INT32_MAX);
  t0 += wbase;
  t1 += wbase;
  const bool nonempty = has_ray && se > sb;
  if (nonempty) {
    const float ta = __ldg(t0 + my_beg), te = __ldg(t1 + my_end - 1);
    float o[3], d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      o[c] = __ldg(ro + 3 * r + c);
      d[c] = __ldg(rd + 3 * r + c);
    }
    make_ray_rec(fw.rays(L) + lane, fw.lens(L) + lane, smem, L, G, o, d, ta, te);
  } else if (has_ray) {
    reinterpret_cast<float4*>(rgba)[r] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  unsigned pending = __ballot_sync(kFieldFull, nonempty);  // rays not yet taken by a group
  __syncwarp();  // the ray records are visible

  // the group's ray: its index in the task (-1: none), its range, the lane's
  // position, its records
  int ray = -1, beg = 0, end = 0, q = 0;
  float tb = 0.f;
  unsigned evals = 0;  // of the ray in work
  RayAcc acc;
  acc_clear(acc);
  float2 a[kPairs], b[kPairs];  // the next chunk's t0, t1
#pragma unroll
  for (int h = 0; h < kPairs; ++h) a[h] = b[h] = splat(0.f);
  rgba += 4 * first;
  for (;;) {
    unsigned idle = __ballot_sync(kFieldFull, ray < 0) & kLeaders;  // groups without a ray
    if (idle) {  // uniform
      if (!pending && idle == kLeaders) break;
      const bool was_idle = ray < 0;
      while (idle && pending) {
        const int g = (__ffs(idle) - 1) / kGroupLanes, i = __ffs(pending) - 1;
        idle &= idle - 1;
        pending &= pending - 1;
        const int rb = __shfl_sync(kFieldFull, my_beg, i), re = __shfl_sync(kFieldFull, my_end, i);
        if (grp == g) {
          ray = i;
          beg = rb;
          end = re;
          q = (rb & ~3) + kPerLane * gl;
          load_lane<kVec>(t0, t1, q, beg, end, lim, a, b);
          tb = fw.rays(L)[i].base.w;
        }
        if constexpr (kForm != kFew) fw.setup(L, G, g, i);
      }
      if constexpr (kForm == kFew) fw.setup_own(L, G, was_idle && ray >= 0, ray);
      fw.ready();
    }
    float2 t[kPairs], dt[kPairs];
    float lo, hi;
    chunk_params<false>(a, b, tb, q - beg, end - beg, t, dt, lo, hi);
    int kept;
    const int len = fw.cull(L, G, lo, hi, kept);
    q += kChunk;
    load_lane<kVec>(t0, t1, q, beg, end, lim, a, b);  // the next chunk's, ahead of the blob loop
    BlobSums sums;
    sums_clear(sums);
    sum_blobs(smem, fw.recs + L.list, len, t, sums);
    if constexpr (kForm == kMany) fw.more(L, G, ray, lo, hi, t, sums, kept);
    if (count_evals && ray >= 0 && gl == 0)
      evals += (unsigned)kept * (unsigned)(min(q, end) - max(q - kChunk, beg));
    RayLen* const rl = fw.lens(L) + max(ray, 0);
    float2 f[kPairs];
    const bool faint = shade_chunk(sums, dt, ray, acc, f);
    if constexpr (kForm == kMany) {
      faint_product(f, faint, acc);
    } else if (__any_sync(kFieldFull, faint)) {
      faint_chunk(reinterpret_cast<float*>(smem + fw.recs + L.ring), rl, f, faint, ray, q - kChunk,
                  beg, end, my_beg, acc.S);
    }
    const bool done = ray >= 0 && q - kPerLane * gl >= end;
    if (__any_sync(kFieldFull, done)) {
      finish_rays(acc, kForm == kMany ? acc.T : rl->T, done, rgba + 4 * ray);
      if (done) {
        ray = -1;
        beg = end = 0;
        fw.release();
        acc_clear(acc);
        if (count_evals && gl == 0) atomicAdd(&g_blob_evals, (unsigned long long)evals);
        evals = 0;
      }
    }
    __syncwarp();  // the group's lists and records may be overwritten
  }
}

}  // namespace

unsigned long long composite_take_blob_evals() {
  unsigned long long v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_blob_evals, sizeof(v)) != cudaSuccess) return 0;
  cudaMemcpyToSymbol(g_blob_evals, &zero, sizeof(zero));
  return v;
}

}  // namespace hdda

extern "C" int hdda_composite(const float* rays_o, const float* rays_d, int64_t n_rays,
                              const int64_t* offsets, const float* t0, const float* t1,
                              const float* field, int n_gauss, float* rgba_out,
                              hdda_stream_t stream) {
  using namespace hdda;
  clear_error();
  if (n_rays < 0) return set_error(HDDA_ERR_INVALID_ARG, "n_rays < 0");
  if (n_gauss < 0 || n_gauss > kMaxGauss)
    return set_error(HDDA_ERR_INVALID_ARG, "n_gauss=%d outside 0..%d", n_gauss, kMaxGauss);
  if (n_rays == 0) return HDDA_OK;
  if (!rays_o || !rays_d || !offsets || !rgba_out || (n_gauss > 0 && !field))
    return set_error(HDDA_ERR_INVALID_ARG, "NULL pointer");
  if (reinterpret_cast<uintptr_t>(rgba_out) % 16 != 0)
    return set_error(HDDA_ERR_INVALID_ARG, "rgba_out must be 16-byte aligned");
  // over up to 16 blobs a task is over soon: of twice as many rays its start weighs less (640,000
  // rays of 20 samples over 16 blobs 253 -> 222 us, over 32 298 -> 267, but an object frame over 32
  // 248 -> 262)
  const int R = field_task_rays(n_rays) * (n_gauss <= 16 && n_rays >= 65536 ? 2 : 1);
  const int64_t warps = (n_rays + R - 1) / R;
  const int64_t blocks = (warps + kWarpsPerCta - 1) / kWarpsPerCta;
  if (blocks > INT32_MAX) return set_error(HDDA_ERR_INVALID_ARG, "too many rays");
  const unsigned grid = (unsigned)blocks;
  const FieldLayout L = field_layout<kRoom64>(n_gauss, kWarpsPerCta, R, n_gauss <= kAllBlobs ? kRing : 0);
  const bool vec = ((reinterpret_cast<uintptr_t>(t0) | reinterpret_cast<uintptr_t>(t1)) & 15) == 0;
  const auto kern = n_gauss <= kFewBlobs
                        ? (vec ? composite_kernel<true, kFew> : composite_kernel<false, kFew>)
                    : n_gauss <= kAllBlobs
                        ? (vec ? composite_kernel<true, kSome> : composite_kernel<false, kSome>)
                        : (vec ? composite_kernel<true, kMany> : composite_kernel<false, kMany>);
  if (L.bytes > 48 * 1024)
    HDDA_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)L.bytes));
  KernelTimer kt("composite", (cudaStream_t)stream);
  kern<<<grid, kWarpsPerCta * 32, L.bytes, (cudaStream_t)stream>>>(
      rays_o, rays_d, n_rays, R, offsets, t0, t1, field, n_gauss, rgba_out, counters_on());
  kt.stop();
  HDDA_CUDA_TRY(cudaGetLastError());
  return HDDA_OK;
}
