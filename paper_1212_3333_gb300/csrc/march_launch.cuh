// Template launcher shared by the per-storage translation units.
#pragma once
#include <algorithm>
#include <type_traits>

#include "ctx.h"
#include "march.cuh"
#include "march_deferred.cuh"
#include "march_persist.cuh"
#include "march_split.cuh"
#include "march_wave.cuh"

namespace amr {

// A block may use 48 KB of shared memory, its static arrays (`fixed`) included, unless the
// kernel's dynamic part is allowed to be larger.
template <typename K>
cudaError_t allow_smem(K kernel, size_t smem, size_t fixed) {
  if (smem + fixed <= 48 * 1024) return cudaSuccess;
  return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
}

// Allows the launch its shared memory and fits the carveout: the smallest split that still
// holds as many blocks per SM as the registers allow, so that the rest of the SM's 256 KB serves
// as L1 cache for the bricks (measured on C2, Phong, per-ray loop at 2048^2 / deferred at 1024^2,
// Gsamples/s: driver's choice 81.1 / 46.4, this split 81.8 / 47.7; more L1 matters - the per-ray
// loop with 28 KB of unused shared memory per block ran at 77.6).  Returns the resident blocks
// per SM.
template <typename K>
cudaError_t fit_carveout(K kernel, size_t smem, int threads, int& occ) {
  int dev = 0, max_smem = 0, reserved = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess) e = allow_smem(kernel, smem, fa.sharedSizeBytes);
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&max_smem, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
  if (e == cudaSuccess)
    e = cudaDeviceGetAttribute(&reserved, cudaDevAttrReservedSharedMemoryPerBlock, dev);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                             cudaSharedmemCarveoutMaxShared);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, threads, smem);
  if (e != cudaSuccess || occ <= 0 || max_smem <= 0) return e;
  // a block's shared memory: the dynamic part, the kernel's static arrays, the reserve
  const long long need = (long long)occ * ((long long)smem + (long long)fa.sharedSizeBytes + reserved);
  const int pct = (int)std::min(100LL, (need * 100 + max_smem - 1) / max_smem);
  return cudaFuncSetAttribute(kernel, cudaFuncAttributePreferredSharedMemoryCarveout, pct);
}

template <typename K>
cudaError_t launch_one(K kernel, dim3 grid, dim3 block, size_t smem, cudaStream_t s,
                       const RenderArgs& a) {
  int occ = 0;
  const cudaError_t e = fit_carveout(kernel, smem, (int)(block.x * block.y * block.z), occ);
  if (e != cudaSuccess) return e;
  kernel<<<grid, block, smem, s>>>(a);
  return cudaGetLastError();
}

// Persistent launch of the refill schedule: the queue head is zeroed, then as many blocks
// as fit on the device start, at most one warp per 8x4 pixel tile.
template <typename K>
cudaError_t launch_persist(K kernel, size_t smem, cudaStream_t s, const RenderArgs& a) {
  cudaError_t e = cudaMemsetAsync(a.counters + kQueueCounter, 0, sizeof(unsigned long long), s);
  cudaFuncAttributes fa;
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, kernel);
  if (e == cudaSuccess) e = allow_smem(kernel, smem, fa.sharedSizeBytes);
  int dev = 0, sms = 0, occ = 0;
  if (e == cudaSuccess) e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kernel, 128, smem);
  if (e != cudaSuccess) return e;
  const long long tiles = (long long)((a.ray.width + 7) / 8) * ((a.ray.rows + 3) / 4);
  const long long grid = std::max(1LL, std::min((long long)sms * std::max(occ, 1), (tiles + 3) / 4));
  kernel<<<(unsigned)grid, dim3(8, 16), smem, s>>>(a, a.samples_per_iter);
  return cudaGetLastError();
}

inline long long tiles_of(const RenderArgs& a) {
  return (long long)((a.ray.width + 7) / 8) * ((a.ray.rows + 3) / 4);
}
inline long long tiles_of(const BatchArgs& b) { return b.n_items; }
inline const RenderArgs& args_of(const RenderArgs& a) { return a; }
inline const RenderArgs& args_of(const BatchArgs& b) { return b.A; }

// Persistent launch: as many 128-thread blocks as are resident at once, at most `per_tile`
// of them per tile, and at least a warp per tile while they last.
template <typename K, typename Args>
cudaError_t launch_stride(K kernel, size_t smem, cudaStream_t s, const Args& a, int per_tile) {
  int dev = 0, sms = 0, occ = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e == cudaSuccess) e = fit_carveout(kernel, smem, 128, occ);
  if (e != cudaSuccess) return e;
  const long long want = per_tile > 0 ? tiles_of(a) * per_tile : (tiles_of(a) + 3) / 4;
  const long long grid = std::max(1LL, std::min((long long)sms * std::max(occ, 1), want));
  kernel<<<(unsigned)grid, dim3(8, 16), smem, s>>>(a);
  return cudaGetLastError();
}

// The same for the tile-queue kernels (march_kernel, deferred_kernel), whose queue head is
// zeroed first (every launch owns its queue, also when a caller renders a frame in several
// bands on one set of counters); at most one warp per tile.
template <typename K, typename Args>
cudaError_t launch_tiles(K kernel, size_t smem, cudaStream_t s, const Args& a) {
  cudaError_t e = cudaMemsetAsync(args_of(a).counters + kQueueCounter, 0, sizeof(unsigned long long), s);
  return e == cudaSuccess ? launch_stride(kernel, smem, s, a, 0) : e;
}

template <int ST>
constexpr bool kLinearStorage = ST != ST_TEXOBJ && ST != ST_ATLAS_TEX3D;

// Deferred shading in one kernel, of all tiles or of those the split march left: the per-ray
// loop for single images of kLargePixels pixels and more, whose rays stay together (2048^2, ms,
// deferred / per ray: 77 leaves 3.7 / 2.7, 3,998 leaves ramp 11.0 / 9.7, half of the cells opaque
// 31.2 / 25.6, 30,164 leaves 85.8 / 85.4; but ramp 17.9 / 19.0, which the split march takes).
template <int ST, int SHADE, typename Args>
cudaError_t launch_one_kernel(cudaStream_t s, const Args& a) {
  const size_t base = StagedTf<Args>::bytes(a);
  if constexpr (std::is_same<Args, RenderArgs>::value && kLinearStorage<ST> &&
                (SHADE & kShadeShadow) == 0 && AMR_WARP_TILE_W == 8)
    if (tiles_of(a) * 32 >= kLargePixels) return launch_tiles(march_kernel<ST, 1, SHADE>, base, s, a);
  return launch_tiles(deferred_kernel<ST, SHADE, Args>, base + 4 * sizeof(DeferArea), s, a);
}

// One band of the split march (b carries its workspace), in rounds that each fill the
// workspace at most once, then the tiles that were left.
template <int ST, int SHADE, typename Args>
cudaError_t launch_rounds(int rounds, cudaStream_t s, const Args& b) {
  const TaskSpace& ts = args_of(b).ts;
  const size_t base = StagedTf<Args>::bytes(b);
  cudaError_t e = cudaMemsetAsync(ts.heads, 0, kHeads * sizeof(unsigned), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(ts.tile, 0xff, (size_t)tiles_of(b) * sizeof(int2), s);
  for (int r = 0; e == cudaSuccess && r < rounds; ++r) {
    if (r > 0) e = cudaMemsetAsync(ts.heads, 0, kRoundHeads * sizeof(unsigned), s);
    if (e == cudaSuccess)
      e = launch_stride(split_march_kernel<ST, SHADE, Args>, base + 4 * sizeof(CandArea<true>), s, b, 1);
    if (e == cudaSuccess && fault_injected("shade_launch")) e = cudaErrorLaunchFailure;
    if (e == cudaSuccess) e = launch_stride(split_shade_kernel<ST, SHADE, Args>, base, s, b, 4);
    if (e == cudaSuccess) e = launch_stride(split_outer_kernel<ST, SHADE, Args>, base, s, b, 4);
    if (e == cudaSuccess) e = launch_stride(split_sum_kernel<Args>, 0, s, b, 4);
  }
  if (e != cudaSuccess) return e;
  return launch_one_kernel<ST, SHADE>(s, b);
}

// Deferred shading of one image: the split march in bands of rows that the workspace has tile
// records for, or without a workspace the one-kernel march.
template <int ST, int SHADE>
cudaError_t launch_shaded(const TaskPlan& plan, cudaStream_t s, const RenderArgs& a) {
  if constexpr (kLinearStorage<ST>) {
    const long long tiles_x = (a.ray.width + 7) / 8;
    const int band = 4 * (int)std::min(plan.tiles / tiles_x, 1LL << 20);  // rows
    if (band > 0) {
      cudaError_t e = cudaSuccess;
      for (int row = 0; e == cudaSuccess && row < a.ray.rows; row += band) {
        RenderArgs b = a;
        b.ts = plan.ts;
        b.ray.row0 = a.ray.row0 + row;
        b.ray.rows = std::min(band, a.ray.rows - row);
        b.out = a.out + (size_t)row * a.ray.width;
        b.dense_below = plan.dense_below;
        e = launch_rounds<ST, SHADE>(plan.rounds(tiles_of(b)), s, b);
      }
      return e;
    }
  }
  return launch_one_kernel<ST, SHADE>(s, a);
}

// Level-of-detail pruning from so many pixels on leaves few and long segments, as in a tree of few
// leaves: the one-kernel marches are faster.  (ms, split / one kernel: 30,164 leaves 2048^2 at 4
// pixels 16.6 / 18.7, at 10 5.7 / 4.8, 1024^2 at 10 0.92 / 0.82; 32,198 leaves 1024^2 at 4 5.9 / 7.8, at 10
// 2.8 / 2.2.)
inline bool pruned_far(const RenderArgs& a) {
  return a.ray.lod_scale * a.ray.height >= 8.0 * 2.0 * a.ray.tan_half_fov_y;
}

// Unshaded frames with stencil-maximum bricks: the split march for images whose few warps wait
// for fetches, on hierarchies with enough leaves to make those dear; the per-ray loop elsewhere.
// Measured (ms, split / per ray, ramp and every sample opaque): 77 leaves 256^2 0.163 / 0.143, 0.226
// / 0.179; 1,175 leaves 640 x 479 0.66 / 0.65, 1.16 / 1.01; 3,998 leaves 640 x 479 0.69 / 0.72, 1.36 / 1.28,
// 800 x 600 0.82 / 0.77, 1.81 / 1.41; 30,164 leaves 640 x 479 1.23 / 1.60, 3.25 / 3.91, 800 x 600 1.50 /
// 1.76, 4.36 / 4.45, 1024^2 3.05 / 2.63, 9.9 / 7.9.
template <int ST>
cudaError_t launch_plain_max(size_t tf_bytes, cudaStream_t s, const RenderArgs& a) {
  const long long most = a.ray.n_leaves >= 10000 ? 600000 : a.ray.n_leaves >= 2500 ? 350000 : 0;
  if ((long long)a.ray.width * a.ray.rows > most || pruned_far(a))
    return launch_tiles(march_kernel<ST, 1, kShadeMaxBit>, tf_bytes, s, a);
  return launch_tiles(split_march_kernel<ST, kShadeMaxBit>,
                      ((tf_bytes + 15) & ~(size_t)15) + 4 * sizeof(CandArea<false>), s, a);
}

template <int ST>
amr_status launch_storage(amr_ctx* c, const RenderArgs& a, int interp, int shade, int schedule,
                          cudaStream_t s) {
  const dim3 block(8, 16);
  const dim3 grid((unsigned)((a.ray.width + 7) / 8), (unsigned)((a.ray.rows + 15) / 16));
  const size_t tf_bytes = (size_t)a.tf_n * sizeof(float4) + (size_t)(a.tf_n + 1) * sizeof(int);
  if (grid.x == 0 || grid.y == 0) return AMR_OK;
  // the stencil-maximum opacity test: pointer storages, trilinear, schedules 0 and 3
  constexpr bool kPtr = ST == ST_PTR || ST == ST_PTR_F16 || ST == ST_PTR_BF16;
  const bool mx = kPtr && (shade & kShadeMaxBit) != 0 && interp == 1 &&
                  !(shade & kShadeShadow) && (schedule == 0 || schedule == 3);
  shade &= ~kShadeMaxBit;
  TaskPlan plan;
  // (not for texture storages, where it measured slower at 1900 x 1800: 37.1 against 31.8 ms;
  // nor for a caller that brings its own counters and may not allocate)
  if (kLinearStorage<ST> && schedule == 3 && a.counters == c->dev.counters &&
      ((shade & kShadeShadow) != 0 || !pruned_far(a)))
    plan = plan_tasks(c, tiles_of(a), (shade & kShadeShadow) != 0 ? TaskUse::shadow : TaskUse::image, s);
  cudaError_t e;
  if (shade & kShadeShadow) {
    // secondary rays to the point light: per-ray schedule (a lane marches its samples'
    // light rays) or deferred shading (the warp marches each queued sample's light ray
    // together); trilinear, FP32 linear storages
    if constexpr (ST == ST_PTR || ST == ST_ATLAS_LINEAR) {
      const int base = shade & 3;
      if (interp != 1 || (schedule != 0 && schedule != 3) || (schedule == 3 && base == 0))
        return fail(c, AMR_ERR_ARG,
                    "secondary rays render trilinear with schedule 0, or 3 with shade = 1");
      if (schedule == 3) {
        if (base == 1) e = launch_shaded<ST, 1 | kShadeShadow>(plan, s, a);
        else e = launch_shaded<ST, 2 | kShadeShadow>(plan, s, a);
      } else {
        const size_t smem = tf_bytes;
        if (base == 0) e = launch_tiles(march_kernel<ST, 1, kShadeShadow>, smem, s, a);
        else if (base == 1) e = launch_tiles(march_kernel<ST, 1, 1 | kShadeShadow>, smem, s, a);
        else e = launch_tiles(march_kernel<ST, 1, 2 | kShadeShadow>, smem, s, a);
      }
    } else {
      return fail(c, AMR_ERR_ARG, "secondary rays need the ptr or atlas_linear storage, FP32 cells");
    }
  } else if (schedule == 3) {
    // warp-synchronous march with deferred shading (trilinear, Phong)
    if (interp != 1 || (shade != 1 && shade != 2))
      return fail(c, AMR_ERR_ARG, "deferred shading renders trilinear with shade = 1");
    if constexpr (kPtr) {
      if (mx) {
        if (shade == 1) e = launch_shaded<ST, 1 | kShadeMaxBit>(plan, s, a);
        else e = launch_shaded<ST, 2 | kShadeMaxBit>(plan, s, a);
        goto launched;
      }
    }
    if (shade == 1) e = launch_shaded<ST, 1>(plan, s, a);
    else e = launch_shaded<ST, 2>(plan, s, a);
  } else if (schedule == 2) {
    // persistent warps with ray refill (trilinear)
    if (interp != 1) return fail(c, AMR_ERR_ARG, "the refill schedule renders trilinear");
    const size_t smem = tf_bytes;
    if (shade == 0) e = launch_persist(persist_kernel<ST, 1, 0>, smem, s, a);
    else if (shade == 1) e = launch_persist(persist_kernel<ST, 1, 1>, smem, s, a);
    else e = launch_persist(persist_kernel<ST, 1, 2>, smem, s, a);
  } else if constexpr (ST >= ST_PTR_F16) {
    // 16-bit cells: trilinear, per-ray schedule
    if (interp != 1 || schedule != 0)
      return fail(c, AMR_ERR_ARG, "16-bit storage renders trilinear with schedule 0, 2 or 3");
    const size_t smem = tf_bytes;
    if constexpr (kPtr) {
      if (mx) {
        if (shade == 0) e = launch_plain_max<ST>(smem, s, a);
        else if (shade == 1) e = launch_tiles(march_kernel<ST, 1, 1 | kShadeMaxBit>, smem, s, a);
        else e = launch_tiles(march_kernel<ST, 1, 2 | kShadeMaxBit>, smem, s, a);
        goto launched;
      }
    }
    if (shade == 0) e = launch_tiles(march_kernel<ST, 1, 0>, smem, s, a);
    else if (shade == 1) e = launch_tiles(march_kernel<ST, 1, 1>, smem, s, a);
    else e = launch_tiles(march_kernel<ST, 1, 2>, smem, s, a);
  } else if (schedule == 0 && ST == ST_TEXOBJ) {
    // per-patch textures: one block per 8x16 tile (see march_kernel)
    const size_t smem = tf_bytes;
    if (interp == 1 && shade == 0) e = launch_one(march_kernel<ST, 1, 0, false>, grid, block, smem, s, a);
    else if (interp == 1 && shade == 1) e = launch_one(march_kernel<ST, 1, 1, false>, grid, block, smem, s, a);
    else if (interp == 1 && shade == 2) e = launch_one(march_kernel<ST, 1, 2, false>, grid, block, smem, s, a);
    else if (interp == 0 && shade == 0) e = launch_one(march_kernel<ST, 0, 0, false>, grid, block, smem, s, a);
    else e = launch_one(march_kernel<ST, 0, 1, false>, grid, block, smem, s, a);
  } else if (schedule == 0) {
    const size_t smem = tf_bytes;
    if constexpr (kPtr) {
      if (mx) {
        if (shade == 0) e = launch_plain_max<ST>(smem, s, a);
        else if (shade == 1) e = launch_tiles(march_kernel<ST, 1, 1 | kShadeMaxBit>, smem, s, a);
        else e = launch_tiles(march_kernel<ST, 1, 2 | kShadeMaxBit>, smem, s, a);
        goto launched;
      }
    }
    if (interp == 1 && shade == 0) e = launch_tiles(march_kernel<ST, 1, 0>, smem, s, a);
    else if (interp == 1 && shade == 1) e = launch_tiles(march_kernel<ST, 1, 1>, smem, s, a);
    else if (interp == 1 && shade == 2) e = launch_tiles(march_kernel<ST, 1, 2>, smem, s, a);
    else if (interp == 0 && shade == 0) e = launch_tiles(march_kernel<ST, 0, 0>, smem, s, a);
    else e = launch_tiles(march_kernel<ST, 0, 1>, smem, s, a);
  } else {
    const size_t smem = ((tf_bytes + 15) & ~(size_t)15) + 4 * sizeof(WarpArea);
    if (interp == 1 && shade == 0) e = launch_one(wave_kernel<ST, 1, 0>, grid, block, smem, s, a);
    else if (interp == 1 && shade == 1) e = launch_one(wave_kernel<ST, 1, 1>, grid, block, smem, s, a);
    else if (interp == 1 && shade == 2) e = launch_one(wave_kernel<ST, 1, 2>, grid, block, smem, s, a);
    else if (interp == 0 && shade == 0) e = launch_one(wave_kernel<ST, 0, 0>, grid, block, smem, s, a);
    else e = launch_one(wave_kernel<ST, 0, 1>, grid, block, smem, s, a);
  }
launched:
  if (e != cudaSuccess)
    return fail(c, AMR_ERR_CUDA, std::string("march launch: ") + cudaGetErrorString(e));
  return AMR_OK;
}

amr_status launch_ptr(amr_ctx* c, const RenderArgs& a, int interp, int shade, int schedule,
                      cudaStream_t s);
amr_status launch_texobj(amr_ctx* c, const RenderArgs& a, int interp, int shade, int schedule,
                         cudaStream_t s);
amr_status launch_atlas_linear(amr_ctx* c, const RenderArgs& a, int interp, int shade,
                               int schedule, cudaStream_t s);
amr_status launch_atlas_tex3d(amr_ctx* c, const RenderArgs& a, int interp, int shade,
                              int schedule, cudaStream_t s);
amr_status launch_16bit(amr_ctx* c, const RenderArgs& a, int storage, int interp, int shade,
                        int schedule, cudaStream_t s);

}  // namespace amr
