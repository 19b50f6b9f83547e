// Warp-synchronous frame march with deferred shading (schedule 3).
//
// Under the per-ray loop (march_kernel) the opaque samples of a warp - a few percent of
// all samples - branch into gradient shading a handful of lanes at a time, and when a
// gradient neighbour lies beyond the leaf (a cross-leaf lookup through the tree) the whole
// warp waits for that chain of dependent loads.  Here every lane marches its own pixel as
// before, but the warp moves through one loop in step:
//   fetch  - lanes whose segment ended find their next non-empty segment;
//   sample - lanes with samples left take up to samples_per_iter samples: value, transfer
//            function, opacity and the accumulated alpha (so early ray termination is
//            decided at once); an opaque sample is queued with what its shading needs;
//   shade  - once 32 samples are queued (and at the end), each lane shades one of them
//            (gradient, Phong; with secondary rays the warp first marches each queued
//            sample's light ray together) and every lane then adds its own samples'
//            colours in sample order.
// The colour sum of a pixel sees the same terms in the same order as in the per-ray loop,
// so the image is bit-identical to it; only the moments at which the sums are taken
// change.  (With secondary rays each light ray's transmittance is a product taken in
// another order - 32 samples per round - so those images agree to rounding, not bits.)
#pragma once
#include <type_traits>

#include "march.cuh"

namespace amr {

// An opaque sample waiting for its colour: position and segment, value (its transfer-function
// colour is looked up again) and compositing weight w = (1 - A) alpha.  11 words (odd, so a
// warp writing one task per lane hits distinct banks).
struct ShadeTask {
  float beta[3];  // brick coordinates
  float v;
  float w;
  float margin;   // bound on the FP32 position error (brick units)
  int leaf;       // packed leaf id and pruning bound
  int pid0, pid1, n;
  int k_lane;     // sample number (bits 0..22) and the lane whose ray it belongs to (23..27)
};

// Ring of queued samples: at most 31 wait before a step adds up to 32.
constexpr int kDeferRing = 64;
struct DeferArea {
  ShadeTask task[kDeferRing];
  float3 col[32];
};

// resident blocks per SM the register budget allows for (measured on C2, Phong, 2048^2 /
// 1024^2 / 512^2 Gsamples/s: 3 blocks 61.3 / 46.1 / 28.9, 4 blocks 55.9 / 41.9 / 24.9)
#ifndef AMR_MIN_BLOCKS_DEFERRED
#define AMR_MIN_BLOCKS_DEFERRED 3
#endif

// The sample of task t in finest-cell units (as composite_sample computes it).
__device__ __forceinline__ float3 task_point(const RenderArgs& A, const ShadeTask& t) {
  const DLeaf& lf = A.leaves[leaf_of(t.leaf)];
  const float sc = (float)A.lv[lf.level].sc;
  return make_float3((t.beta[0] - 0.5f + (float)lf.blo[0]) * sc,
                     (t.beta[1] - 0.5f + (float)lf.blo[1]) * sc,
                     (t.beta[2] - 0.5f + (float)lf.blo[2]) * sc);
}

// Colour of queued sample t of pixel (px, py), headlight direction (Lx, Ly, Lz): what
// composite_sample computes for an opaque sample; T is its transmittance to the light when
// SHADOW is set.
template <int ST, int GB, bool SHADOW = false>
__device__ __forceinline__ float3 shade_task(const RenderArgs& A, const RayArgs& R,
                                             const float4* s_tf, const ShadeTask& t, int px,
                                             int py, float Lx, float Ly, float Lz, float T) {
  const DLeaf lf = A.leaves[leaf_of(t.leaf)];
  const DLevel& lv = A.lv[lf.level];
  SegState s;
  s.brick = leaf_brick(A.patches, lf);
  s.level = lf.level;
  s.leaf = t.leaf;
  leaf_bounds(lf, lv, s.brick, lod_of(t.leaf), s.leaf_lo, s.bl, s.bh);
  s.margin = t.margin;
  s.pid0 = t.pid0;
  s.pid1 = t.pid1;
  s.n = t.n;
  s.px = px;
  s.py = py;
  const float beta[3] = {t.beta[0], t.beta[1], t.beta[2]};
  float gr[3];
  gradient<ST, 1, GB>(A, R, s, beta, t.k_lane & ((1 << kTaskSampleBits) - 1), lv, gr);
  const float4 c = tf_lookup(s_tf, A.tf_n, t.v, A.vmin, A.inv_range);
  float cr = c.x, cg = c.y, cb = c.z;
  phong(A, lv, gr, Lx, Ly, Lz, cr, cg, cb);
  if constexpr (SHADOW) {
    const float I = fmaf(1.0f - A.light_ambient, T, A.light_ambient);
    cr *= I;
    cg *= I;
    cb *= I;
  }
  return make_float3(cr, cg, cb);
}

// The march of pixel (i, j) of view R by one lane of a warp whose 32 lanes all call this
// together (lanes without a pixel pass active = false); Q is the warp's queue area.
// Returns premultiplied RGBA (zero for inactive lanes); adds to nsamp and status.
// samples whose stencil maxima (with stencil-maximum bricks) or values (without) the
// deferred loop loads together
#ifndef AMR_DEFER_GROUP
#define AMR_DEFER_GROUP 8
#endif
#ifndef AMR_DEFER_VALUES
#define AMR_DEFER_VALUES 2
#endif

template <int ST, int SHADE>
__device__ __forceinline__ float4 march_deferred(const RenderArgs& A, const RayArgs& R, int i,
                                                 int j, bool active, const float4* s_tf,
                                                 const int* s_nz, float clear_below,
                                                 DeferArea& Q, unsigned& nsamp,
                                                 unsigned long long& status) {
  constexpr bool MX = (SHADE & kShadeMaxBit) != 0;  // the stencil-maximum test
  const unsigned FULL = 0xffffffffu;
  const int lane = (int)(threadIdx.x + blockDim.x * threadIdx.y) & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  RayF rf;
  float Lx = 0.f, Ly = 0.f, Lz = 0.f;
  bool live = false;
  {
    RayX rx;
    if (active && make_ray(R, i, j, rx)) {
      make_frame(R, rx, rf);
      const float inv_dn = 1.0f / rf.dn;
      Lx = -rf.Dd[0] * (float)R.hf[0] * inv_dn;
      Ly = -rf.Dd[1] * (float)R.hf[1] * inv_dn;
      Lz = -rf.Dd[2] * (float)R.hf[2] * inv_dn;
      live = true;
    }
  }
  float C0 = 0.f, C1 = 0.f, C2 = 0.f, Acc = 0.f;
  int pid0 = kPidIn, seg = 0, prev = -1;
  float tau0 = 0.f, e0 = 0.f;
  uint32_t start = 0;
  SegSetup g;
  MaxWalk<ST> walk;
  g.s.n = 0;
  int k = 0;
  int queued = 0, head = 0;      // warp-uniform: tasks in the ring, and the first one's slot
  unsigned long long mine = 0;   // bit p: the p-th queued task is this lane's

  // shade the first `count` queued tasks (one per lane), then each lane adds its own colours
  // in order; with secondary rays the whole warp first marches each task's light ray together
  auto drain = [&](int count) {
    __syncwarp();
    float T = 1.0f;
    if constexpr ((SHADE & kShadeShadow) != 0) {
      for (int q = 0; q < count; ++q) {
        const float3 x = task_point(A, Q.task[(head + q) & (kDeferRing - 1)]);
        const float Tq = warp_shadow_transmittance<ST>(A, R, s_tf, x.x, x.y, x.z);
        if (lane == q) T = Tq;
      }
    }
    const ShadeTask& t = Q.task[(head + lane) & (kDeferRing - 1)];
    const int owner = lane < count ? t.k_lane >> kTaskSampleBits : lane;
    const int px = __shfl_sync(FULL, i, owner), py = __shfl_sync(FULL, j, owner);
    const float tx = __shfl_sync(FULL, Lx, owner), ty = __shfl_sync(FULL, Ly, owner),
                tz = __shfl_sync(FULL, Lz, owner);
    if (lane < count)
      Q.col[lane] = shade_task<ST, (SHADE & 3) == 2, (SHADE & kShadeShadow) != 0>(
          A, R, s_tf, t, px, py, tx, ty, tz, T);
    __syncwarp();
    for (unsigned m = (unsigned)mine & (0xffffffffu >> (32 - count)); m != 0; m &= m - 1) {
      const int q = __ffs(m) - 1;
      const float w = Q.task[(head + q) & (kDeferRing - 1)].w;
      const float3 c = Q.col[q];
      C0 = fmaf(w, c.x, C0);
      C1 = fmaf(w, c.y, C1);
      C2 = fmaf(w, c.z, C2);
    }
    __syncwarp();
    queued -= count;
    head += count;
    mine >>= count;
  };

  // Every pass either fetches segments for at least one lane or takes samples, and each
  // ray has finitely many of both, so the loop ends with every lane's ray finished.
  for (;;) {
    const bool flush = !__any_sync(FULL, live);  // every ray has ended: only the ring is left
    if (flush && queued == 0) break;
    // lanes whose segment ended fetch their next non-empty one (measured on C2: fetching
    // as soon as any lane needs beats waiting for a quarter or half of them)
    const bool need = live && k >= g.s.n;
    if (need) {
      for (;;) {
        if (pid0 == kPidOut) {
          live = false;
          break;
        }
        if (seg >= A.max_segments) {
          status |= kStatusCapacity;
          live = false;
          break;
        }
        ++seg;
        int pid1 = kPidOut;
        float tau1 = rf.tau_out, e1 = exit_bound(rf);
        const int lmin = lod_min_level(R, A.lv, rf, i, j, pid0, tau0, e0);
        const int lid = next_leaf<kLdexp<1, SHADE>>(A.nodes, A.leaves, A.face_node, A.node_box, R, i, j, rf,
                                  start, prev, pid0, tau0, e0, pid1, tau1, e1, lmin);
        if (lid < 0) {
          status |= kStatusDevice;
          live = false;
          break;
        }
        prev = lid;
        const DLeaf lf = A.leaves[lid];
        const DLevel& lv = A.lv[lf.level];
        int n = segment_count(R, i, j, rf, pid0, tau0, e0, pid1, tau1, e1, lv);
        if (n > kMaxSamplesPerSegment) {
          status |= kStatusCapacity;
          n = kMaxSamplesPerSegment;
        }
        if (A.skip && tf_transparent(s_nz, A.tf_n, lf.vmin, lf.vmax, A.vmin, A.inv_range)) {
          pid0 = pid1;
          tau0 = tau1;
          e0 = e1;
          continue;
        }
        setup_segment(A, rf, lf, lv, lid, pid0, pid1, tau0, e0, tau1, e1, n, i, j, g, lmin);
        if constexpr (MX) walk.start(A, g);
        k = 0;
        pid0 = pid1;  // where the next segment starts
        tau0 = tau1;
        e0 = e1;
        break;
      }
    }
    // A lane takes its next G samples at a time: a mask of those that may be opaque (by
    // their stencil maxima, or by their values), then, in step with the other lanes, each
    // sample of the mask in order.  Most masks are empty, so the warp-wide steps are few.
    constexpr int G = MX ? AMR_DEFER_GROUP : AMR_DEFER_VALUES;
    for (int step = 0; step < A.samples_per_iter; step += G) {
      const int kb = k;
      const int cnt = live ? min(min(G, A.samples_per_iter - step), g.s.n - k) : 0;
      unsigned mask = 0;
      float val[MX ? 1 : G];
      if (cnt > 0) {
        if constexpr (MX) {
          if (walk.inside) mask = walk.template opaque_mask<G>(kb, g.s.n, clear_below);
          else mask = 0xffffffffu;
        } else {
#pragma unroll
          for (int q = 0; q < G; ++q) {
            const float kk = (float)min(kb + q, g.s.n - 1);
            val[q] = trilinear<ST>(A, g.s.brick, fmaf(kk, g.db[0], g.b0[0]),
                                   fmaf(kk, g.db[1], g.b0[1]), fmaf(kk, g.db[2], g.b0[2]));
          }
#pragma unroll
          for (int q = 0; q < G; ++q) mask |= val[q] < clear_below ? 0u : 1u << q;
        }
        mask &= (1u << cnt) - 1u;
        k += cnt;
        nsamp += cnt;
      }
      for (;;) {
        const bool some = __any_sync(FULL, mask != 0);
        if (some) {
          bool opaque = false;
          int kk = 0;
          float beta[3], v = 0.f, w = 0.f;
          if (mask != 0) {
            const int q = __ffs(mask) - 1;
            mask &= mask - 1;
            kk = kb + q;
#pragma unroll
            for (int a = 0; a < 3; ++a) beta[a] = fmaf((float)kk, g.db[a], g.b0[a]);
            if constexpr (MX) {
              v = trilinear<ST>(A, g.s.brick, beta[0], beta[1], beta[2]);
            } else {
              v = val[0];
#pragma unroll
              for (int e = 1; e < G; ++e) v = q == e ? val[e] : v;
            }
            const float a_tf = tf_alpha(s_tf, A.tf_n, v, A.vmin, A.inv_range);
            if (a_tf > 0.0f) {
              const float alpha = -expm1f(-A.kappa * a_tf * g.delta);
              w = (1.0f - Acc) * alpha;
              Acc += w;
              opaque = true;
              if (Acc >= A.ert_thresh) {  // early ray termination
                nsamp -= (unsigned)(kb + cnt - 1 - kk);
                live = false;
                mask = 0;
              }
            }
          }
          const unsigned om = __ballot_sync(FULL, opaque);
          if (opaque) {
            const int q = queued + __popc(om & lt_mask);
            ShadeTask& t = Q.task[(head + q) & (kDeferRing - 1)];
            t.beta[0] = beta[0];
            t.beta[1] = beta[1];
            t.beta[2] = beta[2];
            t.v = v;
            t.w = w;
            t.margin = g.s.margin;
            t.leaf = g.s.leaf;
            t.pid0 = g.s.pid0;
            t.pid1 = g.s.pid1;
            t.n = g.s.n;
            t.k_lane = kk | (lane << kTaskSampleBits);
            mine |= 1ull << q;
          }
          queued += __popc(om);
        }
        if (queued >= 32 || (flush && queued != 0)) drain(min(queued, 32));
        else if (!some) break;
      }
      if (flush) break;
    }
  }
  return make_float4(C0, C1, C2, Acc);
}

// An 8x4-pixel tile of a launch: of its one image, or of one of a batch's views.
struct TileAt {
  int tile, tiles_x;  // in its image
  int tf;             // transfer function (batches)
  int view;
  float4* out;
  int width, rows;

  __device__ __forceinline__ void pixel(int lane, int& i, int& jr) const {
    i = (tile % tiles_x) * 8 + (lane & 7);
    jr = (tile / tiles_x) * 4 + (lane >> 3);
  }
  __device__ __forceinline__ size_t at(int i, int jr) const { return (size_t)jr * width + i; }
};

__device__ __forceinline__ const RenderArgs& render_args(const RenderArgs& A) { return A; }
__device__ __forceinline__ const RenderArgs& render_args(const BatchArgs& B) { return B.A; }

__device__ __forceinline__ int count_tiles(const RenderArgs& A) {
  return ((A.ray.width + 7) / 8) * ((A.ray.rows + 3) / 4);
}
__device__ __forceinline__ int count_tiles(const BatchArgs& B) { return B.n_items; }

__device__ __forceinline__ TileAt tile_at(const RenderArgs& A, int t) {
  return {t, (A.ray.width + 7) / 8, 0, 0, A.out, A.ray.width, A.ray.rows};
}
__device__ __forceinline__ TileAt view_tile(const BatchArgs& B, int t, int view) {
  const BatchView& v = B.v[view];
  return {t - v.item0, v.tiles_x, v.tf, view, B.A.out + v.out, v.width, v.height};
}
__device__ __forceinline__ TileAt tile_at(const BatchArgs& B, int t) {
  int lo = 0, hi = B.n_views - 1;  // last view whose first tile is <= t
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (B.v[mid].item0 <= t) lo = mid;
    else hi = mid - 1;
  }
  return view_tile(B, t, lo);
}
// the tile of a chunk (its view is known)
__device__ __forceinline__ TileAt chunk_tile(const RenderArgs& A, int4 meta) { return tile_at(A, meta.x); }
__device__ __forceinline__ TileAt chunk_tile(const BatchArgs& B, int4 meta) {
  return view_tile(B, meta.x, meta.w);
}

__device__ __forceinline__ const RayArgs& tile_rays(const RenderArgs& A, const TileAt&) { return A.ray; }
__device__ __forceinline__ const RayArgs& tile_rays(const BatchArgs& B, const TileAt& p) {
  return B.A.ts.views[p.view];
}

// Transfer functions for a launch's tiles: one image's staged in shared memory with its prefix
// counts and threshold; a batch's read where they are (staging up to eight would take the L1
// cache from the bricks), with their prefix counts and thresholds staged.
template <typename Args>
struct StagedTf;
template <>
struct StagedTf<RenderArgs> {
  float4* s_tf;
  int* s_nz;
  float clear;
  static __host__ __device__ size_t bytes(const RenderArgs& A) {
    return (((size_t)A.tf_n * sizeof(float4) + (size_t)(A.tf_n + 1) * sizeof(int)) + 15) & ~(size_t)15;
  }
  __device__ __forceinline__ StagedTf(const RenderArgs& A, float4* smem, int tid) {
    __shared__ float s_clear;
    s_tf = smem;
    s_nz = reinterpret_cast<int*>(smem + A.tf_n);
    stage_tf(A, s_tf, s_nz, &s_clear, tid, 128);
    clear = s_clear;
  }
  __device__ __forceinline__ const float4* tf(const TileAt&) const { return s_tf; }
  __device__ __forceinline__ const int* nz(const TileAt&) const { return s_nz; }
  __device__ __forceinline__ float clear_below(const TileAt&) const { return clear; }
};
template <>
struct StagedTf<BatchArgs> {
  const float4* all;
  int* s_nz;
  const float* s_clear;
  int n;
  static __host__ __device__ size_t bytes(const BatchArgs& B) {
    return ((size_t)B.n_tf * (B.A.tf_n + 1) * sizeof(int) + 15) & ~(size_t)15;
  }
  __device__ __forceinline__ StagedTf(const BatchArgs& B, float4* smem, int tid) {
    __shared__ float below[8];
    all = B.A.tf;
    s_nz = reinterpret_cast<int*>(smem);
    s_clear = below;
    n = B.A.tf_n;
    for (int t = tid >> 5; t < B.n_tf; t += 4) {
      int* z = s_nz + t * (n + 1);
      tf_prefix_warp(all + t * n, n, z, tid & 31);
      const float m = tf_threshold_warp(B.A, z, tid & 31);
      if ((tid & 31) == 0) below[t] = m;
    }
    __syncthreads();
  }
  __device__ __forceinline__ const float4* tf(const TileAt& p) const { return all + p.tf * n; }
  __device__ __forceinline__ const int* nz(const TileAt& p) const { return s_nz + p.tf * (n + 1); }
  __device__ __forceinline__ float clear_below(const TileAt& p) const { return s_clear[p.tf]; }
};

// Schedule 3 in one kernel: persistent warps taking 8x4-pixel tiles from the global queue (as
// march_kernel does for the per-ray loop), each marching its tile with deferred shading.
template <int ST, int SHADE, typename Args = RenderArgs>
__global__ void __launch_bounds__(128, AMR_MIN_BLOCKS_DEFERRED)
    deferred_kernel(const __grid_constant__ Args P) {
  const RenderArgs& A = render_args(P);
  const int all_tiles = count_tiles(P);
  const RestTiles rest(A, all_tiles);
  const int n_tiles = rest.count();
  if (n_tiles == 0) return;
  extern __shared__ float4 smem[];
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  DeferArea& Q = reinterpret_cast<DeferArea*>(reinterpret_cast<char*>(smem) +
                                              StagedTf<Args>::bytes(P))[tid >> 5];
  const StagedTf<Args> staged(P, smem, tid);
  const int lane = tid & 31;
  unsigned nsamp = 0;
  unsigned long long status = 0;
  // each pass takes one tile, and the queue hands out every tile once
  for (;;) {
    int t = 0;
    if (lane == 0) {
      const unsigned long long q = atomicAdd(A.counters + kQueueCounter, 1ull);
      t = q < (unsigned long long)n_tiles ? (int)q : n_tiles;
    }
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= n_tiles) break;
    t = rest.tile(A, t);
    const TileAt p = tile_at(P, t);
    const RayArgs& R = tile_rays(P, p);
    int i, jr;
    p.pixel(lane, i, jr);
    const int j = R.row0 + jr;
    const bool active = i < p.width && jr < p.rows && j < R.height;
    const float4 c = march_deferred<ST, SHADE>(A, R, i, j, active, staged.tf(p), staged.nz(p),
                                              staged.clear_below(p), Q, nsamp, status);
    if (active) p.out[p.at(i, jr)] = c;
  }
  const unsigned total = __reduce_add_sync(0xffffffffu, nsamp);
  if (lane == 0 && total) atomicAdd(A.counters, (unsigned long long)total);
  if (status) atomicOr(A.counters + 1, status);
}

}  // namespace amr
