// render.cu -- the render-only path: the sampler and the compositor joined
// at the level of runs, so that no sample is ever written to memory (the
// fused sampler + field evaluation; Sec. 1's accumulation applied to the
// intervals Algorithm 1 keeps).
//
// Pass 1 is the samplers' walk (walk_kernel, walk.cuh): each ray's merged
// occupied runs of lattice indices [k_begin, k_end), the first kMaxRuns of
// them, and its number of runs.  Pass 2 (render_kernel) gives each warp R
// consecutive rays (field_task_rays), four of them in work at a time, one
// per group of eight lanes, 32 samples per step (field.cuh).  Every lattice
// index k of a run is the sample (t_k, t_{k+1}), read from the lattice table
// all rays share.  The task's runs are staged in shared memory with their
// first sample positions in the ray, so that a lane finds the run of its
// four consecutive samples by a binary search; usually they lie in one run
// and are five consecutive lattice entries.  No global scan, no sample
// arrays, no host read-back.
//
// A ray with more than kMaxRuns runs is finished in rounds: after the runs
// it has are composited, it walks again from the end of the last one
// (walk_from) and the next kMaxRuns runs are composited with its
// transmittance and colour carried over, so samples are still accumulated front to
// back.  Whenever a group has to walk on, the warp's other groups with runs left walk
// too, into runs of their own: 200,000 rays of 64 runs took 2.46 ms with each
// group walking when it came to it, 1.62 so (1.50 in warps that walked all their
// rays at once).
//
// The same kernel with kStore also writes what the samplers' emit writes:
// the CSR offsets (each task's 32-ray tile prefix from the tile scan plus a
// warp scan of the tile's counts) and every sample at its CSR position (the
// ray's offset, plus its samples of earlier rounds, plus its position in
// this round), so one pass both stores the samples and composites them
// (hdda_traverse_composite).
#include "field.cuh"
#include "walk.cuh"

namespace hdda {
namespace {

constexpr int kRenderWarps = 4;
constexpr int kRoom64 = 32;  // records per group in 64ths of a field of many blobs
constexpr uint32_t kNoRun = 0x7fffffffu;
constexpr unsigned kWalked = 1u, kOther = 2u;
constexpr int kRunStride = kMaxRuns + 1;  // per ray: odd, so the groups' searches hit other banks

// Blob evaluations (sample x kept blob), counted only while profiling.
__device__ unsigned long long g_render_evals;

// Outputs of the storing form (kStore): the samplers' CSR arrays.
struct StoreArgs {
  const int64_t* tile_prefix;  // exclusive prefix of the 32-ray tiles' sample counts
  const int32_t* counts;       // samples per ray
  int64_t* offsets;            // [n + 1], clamped to capacity
  int32_t* ray_idx;
  float* t0;
  float* t1;
  int64_t capacity;
  unsigned* status;            // kDevCapacity when the samples do not fit
};

// Turns a ray's `nr` runs [k_begin, k_end) into {k_begin - first position,
// first position}, positions counted within the ray's round (unused slots
// start at kNoRun, as does the one after the last), and returns the number of
// samples.
__device__ __forceinline__ int number_runs(uint2* sr, int nr) {
  int pos = 0;
  for (int j = 0; j < kRunStride; ++j) {
    const uint2 v = sr[j];
    if (j < nr) {
      sr[j] = make_uint2(v.x - (uint32_t)pos, (uint32_t)pos);
      pos += (int)(v.y - v.x);
    } else {
      sr[j] = make_uint2(0u, kNoRun);
    }
  }
  return pos;
}

template <int kMode, bool kStore, int kForm>
__global__ void __launch_bounds__(kRenderWarps * 32, kForm == kMany ? 5 : 6) render_kernel(
    const float* __restrict__ ro, const float* __restrict__ rd, int64_t n, int R, GridDev g,
    LatticeDev lat, const uint8_t* __restrict__ nruns,
    const uint2* __restrict__ runs, const float* __restrict__ field, int G,
    float* __restrict__ rgba, bool count_evals, StoreArgs out) {
  // field_layout, then per warp [R + kGroups][kRunStride] runs: the rays' and, per group, those
  // of its ray's next round
  extern __shared__ __align__(16) unsigned char smem[];
  const FieldLayout L = field_layout<kRoom64>(G, kRenderWarps, R, 0);
  stage_blobs<kForm>(smem, L, field, G);
  __syncthreads();
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  const int grp = lane / kGroupLanes, gl = lane & (kGroupLanes - 1);
  const int64_t task = (int64_t)blockIdx.x * kRenderWarps + wib, first = task * R;
  if (first >= n) return;  // uniform per warp; no block barrier follows
  FieldWarp<kForm> fw;
  fw.init(smem, L);
  uint2* sr = reinterpret_cast<uint2*>(smem + L.bytes) + wib * (R + kGroups) * kRunStride;

  // lane i < R holds ray i's number of runs, samples of this round and resume index
  const int64_t r = first + lane;
  const bool has_ray = lane < R && r < n;
  const int nr_all = has_ray ? (int)__ldg(nruns + r) : 0;  // saturated at 255; 0 when not finite
  const int nr = min(nr_all, kMaxRuns);
  for (int u0 = 0; u0 < R * kMaxRuns; u0 += 32) {  // R is a multiple of 4: at least two slots
    const int u = u0 + lane, i = u & (R - 1), j = u / R;
    if (j < __shfl_sync(kFull, nr, i)) sr[i * kRunStride + j] = __ldg(runs + (int64_t)j * n + first + i);
  }
  __syncwarp();
  int my_w = 0, my_next = lat.K;
  if (nr > 0) {
    const uint32_t ka = sr[lane * kRunStride].x, kb = sr[lane * kRunStride + nr - 1].y;
    if (nr_all > kMaxRuns) my_next = (int)kb;
    const float ta = __ldg(lat.t + ka), te = __ldg(lat.t + kb);
    float o[3], d[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      o[c] = __ldg(ro + 3 * r + c);
      d[c] = __ldg(rd + 3 * r + c);
    }
    make_ray_rec(fw.rays(L) + lane, fw.lens(L) + lane, smem, L, G, o, d, ta, te);
    my_w = number_runs(sr + lane * kRunStride, nr);
  } else if (has_ray) {
    reinterpret_cast<float4*>(rgba)[r] = make_float4(0.f, 0.f, 0.f, 0.f);
  }
  unsigned pending = __ballot_sync(kFull, nr > 0);  // rays not yet taken by a group
  // storing form: the ray's CSR offset
  int64_t my_gofs = 0;
  if constexpr (kStore) {
    const int per_tile = 32 / R;  // R divides 32
    const int64_t tile = task / per_tile;
    const int64_t tr = tile * 32 + lane;
    const int64_t c = tr < n ? (int64_t)__ldg(out.counts + tr) : 0;
    int64_t inc = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int64_t y = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += y;
    }
    const int64_t ex = __ldg(out.tile_prefix + tile) + inc - c;
    const int slot = (int)(task % per_tile) * R + (lane & (R - 1));
    my_gofs = __shfl_sync(kFull, ex, slot);
    const int64_t mine = __shfl_sync(kFull, c, slot);
    // capacity 0 counts only: offsets unclamped, no samples, no status
    const bool clamp = out.capacity > 0;
    if (has_ray) {
      out.offsets[r] = clamp ? min(my_gofs, out.capacity) : my_gofs;
      if (r == n - 1)
        out.offsets[n] = clamp ? min(my_gofs + mine, out.capacity) : my_gofs + mine;
    }
    if (__any_sync(kFull, clamp && has_ray && my_gofs + mine > out.capacity) && lane == 0)
      atomicOr(out.status, kDevCapacity);
  }
  __syncwarp();

  // the group's ray: its index in the task (-1: none), samples of this round,
  // the lane's position, resume index, records
  int ray = -1, W = 0, q = 0, k_next = 0;
  unsigned ahead = 0;  // kWalked: the next round is there; kOther: this one is in the group's runs
  float tb = 0.f;
  int64_t gofs = 0;
  RayAcc acc;
  acc_clear(acc);
  rgba += 4 * first;
  for (;;) {
    unsigned idle = __ballot_sync(kFull, ray < 0) & kLeaders;  // one bit per group
    if (idle) {  // uniform
      if (!pending && idle == kLeaders) break;
      while (idle && pending) {
        const int gi = (__ffs(idle) - 1) / kGroupLanes, i = __ffs(pending) - 1;
        idle &= idle - 1;
        pending &= pending - 1;
        const int w = __shfl_sync(kFull, my_w, i), kn = __shfl_sync(kFull, my_next, i);
        int64_t go = 0;
        if constexpr (kStore) go = __shfl_sync(kFull, my_gofs, i);
        if (grp == gi) {
          ray = i;
          W = w;
          k_next = kn;
          q = kPerLane * gl;
          tb = fw.rays(L)[i].base.w;
          gofs = go;
        }
        fw.setup(L, G, gi, i);
      }
      fw.ready();
    }
    // this chunk's samples
    float2 a[kPairs], b[kPairs];
#pragma unroll
    for (int h = 0; h < kPairs; ++h) a[h] = b[h] = splat(tb);
    if (ray >= 0 && q < W) {
      const uint2* mr = sr + (ahead & kOther ? R + grp : ray) * kRunStride;
      int j = 0;  // the last run that starts at or before q
#pragma unroll
      for (int s = kMaxRuns / 2; s > 0; s >>= 1)
        if (mr[j + s].y <= (uint32_t)q) j += s;
      uint32_t kq = mr[j].x;
      uint32_t nxt = mr[j + 1].y;
      if ((uint32_t)(q + kPerLane) <= nxt && q + kPerLane <= W) {
        const float* t = lat.t + (int)(kq + (uint32_t)q);
        float x = __ldg(t);
#pragma unroll
        for (int h = 0; h < kPairs; ++h) {
          const float y = __ldg(t + 2 * h + 1), z = __ldg(t + 2 * h + 2);
          a[h] = make_float2(x, y);
          b[h] = make_float2(y, z);
          x = z;
        }
      } else {
#pragma unroll
        for (int i = 0; i < kPerLane; ++i) {
          if (q + i >= W) continue;
          if ((uint32_t)(q + i) >= nxt) {  // a run holds at least one sample
            kq = mr[++j].x;
            nxt = mr[j + 1].y;
          }
          const float* t = lat.t + (int)(kq + (uint32_t)(q + i));
          (i & 1 ? a[i / 2].y : a[i / 2].x) = __ldg(t);
          (i & 1 ? b[i / 2].y : b[i / 2].x) = __ldg(t + 1);
        }
      }
      if constexpr (kStore) {
#pragma unroll
        for (int i = 0; i < kPerLane; ++i) {
          const int64_t qo = gofs + q + i;
          if (q + i < W && qo < out.capacity) {
            out.ray_idx[qo] = (int32_t)(first + ray);
            out.t0[qo] = i & 1 ? a[i / 2].y : a[i / 2].x;
            out.t1[qo] = i & 1 ? b[i / 2].y : b[i / 2].x;
          }
        }
      }
    }
    float2 t[kPairs], dt[kPairs];
    float lo, hi;
    chunk_params<true>(a, b, tb, q, W, t, dt, lo, hi);
    int kept;
    const int len = fw.cull(L, G, lo, hi, kept);
    BlobSums sums;
    sums_clear(sums);
    sum_blobs(smem, fw.recs + L.list, len, t, sums);
    if constexpr (kForm == kMany) fw.more(L, G, ray, lo, hi, t, sums, kept);
    if (count_evals && ray >= 0 && gl == 0)
      atomicAdd(&g_render_evals, (unsigned long long)(kept * min(kChunk, W - q)));
    float2 f[kPairs];
    const bool faint = shade_chunk(sums, dt, ray, acc, f);
    faint_product(f, faint, acc);
    q += kChunk;
    const bool round_over = ray >= 0 && q - kPerLane * gl >= W;
    bool done = round_over && k_next >= lat.K;
    const bool more = round_over && !done;  // another round of runs
    if (__any_sync(kFull, more)) {
      RayLen* const rl = fw.lens(L) + max(ray, 0);  // its T is free here
      if (__any_sync(kFull, more && !(ahead & kWalked))) {
        // One lane per ray walks on, for every group with runs left and not only for the one
        // that needs them now: a walk is a chain that keeps the warp waiting.
        const bool go = ray >= 0 && k_next < lat.K && !(ahead & kWalked);
        if (go) ahead |= kWalked;
        if (go && gl == 0) {
          uint2* mr = sr + (ahead & kOther ? ray : R + grp) * kRunStride;
          Ray ry;
          load_ray(ro, rd, first + ray, ry);
          const LatHdr h = lat_hdr(lat);
          int nr2 = 0;
          const int kn = walk_from<kMode, false>(g, global_tabs(g, lat), lat, h, ry, k_next, mr, 1, nr2);
          rl->next_w = number_runs(mr, nr2);
          mr[kMaxRuns].x = (uint32_t)kn;  // where it resumes: that slot holds no run
        }
        __syncwarp();
      }
      if (more) {
        gofs += W;
        W = rl->next_w;
        ahead ^= kWalked | kOther;
        k_next = (int)sr[(ahead & kOther ? R + grp : ray) * kRunStride + kMaxRuns].x;
        q = kPerLane * gl;
        done = W == 0;
      }
    }
    if (__any_sync(kFull, done)) {
      finish_rays(acc, acc.T, done, rgba + 4 * ray);
      if (done) {
        ray = -1;
        W = 0;
        ahead = 0;
        fw.release();
        acc_clear(acc);
      }
    }
    __syncwarp();  // the group's lists, records and runs may be overwritten
  }
}

const char* render_name(int mode) {
  return mode == kModeDense ? "dense_render" : mode == kModeVdb ? "hdda_render_plain"
                                                                 : "hdda_render";
}

template <int kMode, bool kStore>
int launch_field(const WalkArgs& w, const uint8_t* nr, const uint2* runs, const float* field,
                 int G, float* rgba, const StoreArgs& out, cudaStream_t s) {
  const int R = field_task_rays(w.n);
  const int64_t warps = (w.n + R - 1) / R;
  const unsigned nb = (unsigned)((warps + kRenderWarps - 1) / kRenderWarps);
  const size_t smem = field_layout<kRoom64>(G, kRenderWarps, R, 0).bytes +
                      (size_t)kRenderWarps * (R + kGroups) * kRunStride * sizeof(uint2);
  const auto kern =
      G <= kAllBlobs ? render_kernel<kMode, kStore, kSome> : render_kernel<kMode, kStore, kMany>;
  if (smem > 48 * 1024)
    HDDA_CUDA_TRY(
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  kern<<<nb, kRenderWarps * 32, smem, s>>>(w.ro, w.rd, w.n, R, w.g, w.lat, nr, runs, field, G,
                                           rgba, counters_on(), out);
  return HDDA_OK;
}

size_t a256(size_t x) { return (x + 255) & ~(size_t)255; }

// Scratch: [0, 256) header {walk counter u32, status u32}, then counts, run
// counts and runs (the render kernel needs no tile sums: the walk skips them).
size_t render_scratch_bytes(int64_t n) {
  return 256 + a256(4 * (size_t)n) + a256((size_t)n) + a256(sizeof(uint2) * kMaxRuns * (size_t)n);
}

// Pinned host word for the synchronous status read.
struct HostWord {
  unsigned* p = nullptr;
  ~HostWord() { if (p) cudaFreeHost(p); }
};
thread_local HostWord t_word;

int launch_render(const float* ro, const float* rd, int64_t n, const hdda_grid* grid,
                  const LatticeDev& lat, int32_t width, const float* field, int G, float* rgba,
                  unsigned* dev_status, char* scratch, cudaStream_t s) {
  unsigned* counter = reinterpret_cast<unsigned*>(scratch);
  unsigned* status = dev_status ? dev_status : counter + 1;
  char* p = scratch + 256;
  int32_t* counts = reinterpret_cast<int32_t*>(p);
  p += a256(4 * (size_t)n);
  uint8_t* nr = reinterpret_cast<uint8_t*>(p);
  p += a256((size_t)n);
  uint2* runs = reinterpret_cast<uint2*>(p);
  HDDA_CUDA_TRY(cudaMemsetAsync(scratch, 0, 256, s));
  const int mode = walk_mode(grid);
  WalkArgs w{ro, rd, n, grid->view(), lat, counts, nr, runs, nullptr, counter, status};
  w.width = (int32_t)(width < n ? width : n);
  const size_t stage = stage_layout(lat.K, w.g.L, w.g.R, grid->nodes_total(), mode).bytes;
  {
    KernelTimer kt(walk_name(mode), s);
    const bool skip = grid->walk_variant == HDDA_WALK_SKIP;
    const int st = mode == kModeDense ? launch_walk_mode<kModeDense>(w, stage, skip, s)
                   : mode == kModeVdb ? launch_walk_mode<kModeVdb>(w, stage, skip, s)
                                      : launch_walk_mode<kModeVdbMap>(w, stage, skip, s);
    if (st != HDDA_OK) return st;
  }
  {
    KernelTimer kt(render_name(mode), s);
    const StoreArgs none{};
    const int st = mode == kModeDense
                       ? launch_field<kModeDense, false>(w, nr, runs, field, G, rgba, none, s)
                   : mode == kModeVdb
                       ? launch_field<kModeVdb, false>(w, nr, runs, field, G, rgba, none, s)
                       : launch_field<kModeVdbMap, false>(w, nr, runs, field, G, rgba, none, s);
    if (st != HDDA_OK) return st;
  }
  HDDA_CUDA_TRY(cudaGetLastError());
  return HDDA_OK;
}

// Scratch of the storing form: the header, tile sums and prefixes, counts,
// run counts and runs.
size_t sample_composite_scratch_bytes(int64_t n) {
  const int64_t T = (n + 31) / 32;
  return 256 + 2 * a256(8 * (size_t)T) + a256(4 * (size_t)n) + a256((size_t)n) +
         a256(sizeof(uint2) * kMaxRuns * (size_t)n);
}

const char* sample_composite_name(int mode) {
  return mode == kModeDense ? "dense_sample_composite"
         : mode == kModeVdb ? "hdda_sample_composite_plain"
                            : "hdda_sample_composite";
}

// Walk, tile scan, then the storing render kernel: the samplers' outputs and
// the frame in one pass over the samples.
int launch_sample_composite(const float* ro, const float* rd, int64_t n, const hdda_grid* grid,
                            const LatticeDev& lat, int32_t width, const float* field, int G,
                            float* rgba,
                            int64_t* offsets, int32_t* ray_idx, float* t0, float* t1,
                            int64_t capacity, unsigned* status, char* scratch, cudaStream_t s) {
  const int64_t T = (n + 31) / 32;
  unsigned* counter = reinterpret_cast<unsigned*>(scratch);
  int64_t* total = reinterpret_cast<int64_t*>(scratch + 8);
  char* p = scratch + 256;
  int64_t* tile_sum = reinterpret_cast<int64_t*>(p);
  p += a256(8 * (size_t)T);
  int64_t* tile_prefix = reinterpret_cast<int64_t*>(p);
  p += a256(8 * (size_t)T);
  int32_t* counts = reinterpret_cast<int32_t*>(p);
  p += a256(4 * (size_t)n);
  uint8_t* nr = reinterpret_cast<uint8_t*>(p);
  p += a256((size_t)n);
  uint2* runs = reinterpret_cast<uint2*>(p);
  // a walk in pixel blocks adds the tile sums up atomically: clear them too
  WalkArgs w{ro, rd, n, grid->view(), lat, counts, nr, runs, tile_sum, counter, status};
  w.width = (int32_t)(width < n ? width : n);
  HDDA_CUDA_TRY(cudaMemsetAsync(scratch, 0, w.width > 0 ? 256 + 8 * (size_t)T : 256, s));
  const int mode = walk_mode(grid);
  const size_t stage = stage_layout(lat.K, w.g.L, w.g.R, grid->nodes_total(), mode).bytes;
  {
    KernelTimer kt(walk_name(mode), s);
    const bool skip = grid->walk_variant == HDDA_WALK_SKIP;
    const int st = mode == kModeDense ? launch_walk_mode<kModeDense>(w, stage, skip, s)
                   : mode == kModeVdb ? launch_walk_mode<kModeVdb>(w, stage, skip, s)
                                      : launch_walk_mode<kModeVdbMap>(w, stage, skip, s);
    if (st != HDDA_OK) return st;
  }
  {
    KernelTimer kt("tile_scan", s);
    if (T <= (int64_t)kMaxSupers * kSuperTiles)
      tile_scan_par_kernel<<<(unsigned)((T + kSuperTiles - 1) / kSuperTiles), kSuperTiles, 0, s>>>(
          tile_sum, T, tile_prefix, total, offsets + n);
    else
      tile_scan_kernel<<<1, kScanThreads, 0, s>>>(tile_sum, T, tile_prefix, total, offsets + n);
  }
  HDDA_CUDA_TRY(cudaGetLastError());
  {
    KernelTimer kt(sample_composite_name(mode), s);
    const StoreArgs out{tile_prefix, counts, offsets, ray_idx, t0, t1, capacity, status};
    const int st = mode == kModeDense
                       ? launch_field<kModeDense, true>(w, nr, runs, field, G, rgba, out, s)
                   : mode == kModeVdb
                       ? launch_field<kModeVdb, true>(w, nr, runs, field, G, rgba, out, s)
                       : launch_field<kModeVdbMap, true>(w, nr, runs, field, G, rgba, out, s);
    if (st != HDDA_OK) return st;
  }
  HDDA_CUDA_TRY(cudaGetLastError());
  return HDDA_OK;
}

}  // namespace

unsigned long long render_take_blob_evals() {
  unsigned long long v = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&v, g_render_evals, sizeof(v)) != cudaSuccess) return 0;
  cudaMemcpyToSymbol(g_render_evals, &zero, sizeof(zero));
  return v;
}

}  // namespace hdda

extern "C" int hdda_render(const float* rays_o, const float* rays_d, int64_t n_rays,
                           const hdda_grid* grid, const hdda_params* params, const float* field,
                           int n_gauss, float* rgba_out, uint32_t* dev_status,
                           hdda_stream_t stream) {
  using namespace hdda;
  clear_error();
  cudaStream_t s = (cudaStream_t)stream;
  if (!grid) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  if (n_rays < 0 || n_rays > INT32_MAX)
    return set_error(HDDA_ERR_INVALID_ARG, "n_rays=%lld", (long long)n_rays);
  if (n_gauss < 0 || n_gauss > kMaxGauss)
    return set_error(HDDA_ERR_INVALID_ARG, "n_gauss=%d outside 0..%d", n_gauss, kMaxGauss);
  if (n_rays > 0 && (!rays_o || !rays_d || !rgba_out))
    return set_error(HDDA_ERR_INVALID_ARG, "NULL pointer");
  if (n_gauss > 0 && !field) return set_error(HDDA_ERR_INVALID_ARG, "field is NULL");
  if (reinterpret_cast<uintptr_t>(rgba_out) % 16 != 0)
    return set_error(HDDA_ERR_INVALID_ARG, "rgba_out must be 16-byte aligned");
  if (reinterpret_cast<uintptr_t>(dev_status) % 4 != 0)
    return set_error(HDDA_ERR_INVALID_ARG, "dev_status must be 4-byte aligned");
  int dev = 0;
  HDDA_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != grid->device)
    return set_error(HDDA_ERR_INVALID_ARG, "grid lives on device %d, current is %d",
                     grid->device, dev);
  LatticeDev lat;
  int st = lattice_for(params, s, &lat);
  if (st != HDDA_OK) return st;
  if (n_rays == 0) return HDDA_OK;
  unsigned* hw = nullptr;
  if (!dev_status) {
    if (!t_word.p) HDDA_CUDA_TRY(cudaMallocHost(&t_word.p, sizeof(unsigned)));
    hw = t_word.p;
  }
  char* scratch = nullptr;
  HDDA_CUDA_TRY(scratch_alloc(&scratch, render_scratch_bytes(n_rays), s));
  st = launch_render(rays_o, rays_d, n_rays, grid, lat, params->image_width, field, n_gauss,
                     rgba_out, dev_status, scratch, s);
  if (st == HDDA_OK && !dev_status) {
    cudaError_t e = cudaMemcpyAsync(hw, scratch + 4, sizeof(unsigned), cudaMemcpyDeviceToHost, s);
    if (e != cudaSuccess) st = cuda_error(e, "cudaMemcpyAsync(status)");
  }
  st = scratch_free(scratch, s, st);
  if (st != HDDA_OK || dev_status) return st;
  HDDA_CUDA_TRY(cudaStreamSynchronize(s));
  if (*hw & kDevInternal) return set_error(HDDA_ERR_INTERNAL, "region check failed on the device");
  return HDDA_OK;
}

extern "C" int hdda_traverse_composite(const float* rays_o, const float* rays_d, int64_t n_rays,
                                       const hdda_grid* grid, const hdda_params* params,
                                       int64_t* offsets, int32_t* ray_idx, float* t0, float* t1,
                                       int64_t capacity, const float* field, int n_gauss,
                                       float* rgba_out, uint32_t* dev_status,
                                       hdda_stream_t stream) {
  using namespace hdda;
  clear_error();
  cudaStream_t s = (cudaStream_t)stream;
  if (!grid) return set_error(HDDA_ERR_INVALID_ARG, "grid is NULL");
  if (!params) return set_error(HDDA_ERR_INVALID_ARG, "params is NULL");
  if (n_rays < 0 || n_rays > INT32_MAX)
    return set_error(HDDA_ERR_INVALID_ARG, "n_rays=%lld", (long long)n_rays);
  if (n_gauss < 0 || n_gauss > kMaxGauss)
    return set_error(HDDA_ERR_INVALID_ARG, "n_gauss=%d outside 0..%d", n_gauss, kMaxGauss);
  if (!offsets) return set_error(HDDA_ERR_INVALID_ARG, "offsets is NULL");
  if (capacity < 0) return set_error(HDDA_ERR_INVALID_ARG, "capacity < 0");
  if (capacity > 0 && (!ray_idx || !t0 || !t1))
    return set_error(HDDA_ERR_INVALID_ARG, "sample arrays NULL");
  if (n_rays > 0 && (!rays_o || !rays_d || !rgba_out))
    return set_error(HDDA_ERR_INVALID_ARG, "NULL pointer");
  if (n_gauss > 0 && !field) return set_error(HDDA_ERR_INVALID_ARG, "field is NULL");
  if (reinterpret_cast<uintptr_t>(rgba_out) % 16 != 0)
    return set_error(HDDA_ERR_INVALID_ARG, "rgba_out must be 16-byte aligned");
  if (!dev_status) return set_error(HDDA_ERR_INVALID_ARG, "dev_status is NULL");
  if (reinterpret_cast<uintptr_t>(dev_status) % 4 != 0)
    return set_error(HDDA_ERR_INVALID_ARG, "dev_status must be 4-byte aligned");
  int dev = 0;
  HDDA_CUDA_TRY(cudaGetDevice(&dev));
  if (dev != grid->device)
    return set_error(HDDA_ERR_INVALID_ARG, "grid lives on device %d, current is %d",
                     grid->device, dev);
  LatticeDev lat;
  int st = lattice_for(params, s, &lat);
  if (st != HDDA_OK) return st;
  if (n_rays == 0) {
    HDDA_CUDA_TRY(cudaMemsetAsync(offsets, 0, sizeof(int64_t), s));
    return HDDA_OK;
  }
  char* scratch = nullptr;
  HDDA_CUDA_TRY(scratch_alloc(&scratch, sample_composite_scratch_bytes(n_rays), s));
  st = launch_sample_composite(rays_o, rays_d, n_rays, grid, lat, params->image_width, field,
                               n_gauss, rgba_out, offsets, ray_idx, t0, t1, capacity, dev_status,
                               scratch, s);
  return scratch_free(scratch, s, st);
}
