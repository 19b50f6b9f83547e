// Frame march with compacted evaluation, and shading in a kernel of its own.
//
// In the single-kernel schedules the march and the shading share one register budget (128 to
// 168 registers, 12 to 16 warps per SM) and every phase waits on chains of dependent loads:
// on the 5-level hierarchy at 1024^2 a warp spent 10,000 cycles per segment fetch and 12,000
// per 32 shaded samples, and candidates were evaluated five lanes at a time.  Here
//   split_march_kernel marches a warp's 8x4 tile in step:
//     fetch    - lanes whose segment ended find their next non-empty segment;
//     test     - lanes with samples left test their next few (stencil maxima, or the values
//                themselves) and queue those that may be opaque in shared memory;
//     evaluate - once 32 are queued, each lane evaluates one of them (value, transfer
//                function, opacity) and every lane adds its own opacities in sample order, so
//                early ray termination is decided here;
//   and the opaque samples become tasks in device memory (unshaded: they are composited at
//   once and there is no second kernel);
//   split_shade_kernel takes a tile's tasks 32 at a time: gradient and Phong, one per lane;
//   the neighbour values of gradients that leave their leaf are shared out over the lanes;
//   then every lane adds its own pixel's colours in sample order.
// A pixel sees the same opacities and colours, added in the same order, as in the per-ray
// loop, so the image is bit-identical to it.  A ray that ended early may have queued samples
// beyond its end: they are dropped, and not counted.  (With secondary rays each light ray's
// transmittance is a product taken 32 samples per round, so those images agree to rounding.)
//
// Measured (5-level hierarchy, 1.3e8 cells, Phong with every brick, one kernel against this when
// it came in, ms): 640 x 479 3.49 / 1.99, 1024^2 9.3 / 5.3 (march 5.2, shading 0.64 + 0.95, sums
// 0.25 alone under the profiler), 2048^2 23.5 / 17.4; 8 levels, BF16, 1500 x 1100 17.0 / 10.1;
// secondary rays 393 x 371 21.2 / 5.7 (a tile's light rays no longer wait for one another).  The
// march is bound by the latency of dependent loads (fetches a third of it) at 16 warps per SM;
// shaded, 5 and 6 blocks spill and lose (unshaded 5 win: fewer registers are live).
//
// The tasks live in a workspace of bounded size, so a launch of large or dense images goes in
// rounds: the march hands out tiles until the rest of the workspace is what the tiles under way
// will take, the other kernels empty it, and the next round goes on.  A tile that finds it full
// is given up, whole, until a later round.  Every task passes through device memory, so dense
// images are faster in the one-kernel marches: plan_tasks says where, the march counts tasks and
// segments as it goes, and what it leaves - with dense tiles, and what the last round leaves -
// goes to one of those, which need no workspace.
#pragma once
#include "march_deferred.cuh"

namespace amr {

constexpr int kCandRing = 64;  // at most 31 candidates wait before a step adds up to 32

// A warp's queue of candidates, one array per field.  (The values are not used with
// stencil-maximum bricks; without their array there, unshaded frames take 3 to 6 % longer.)
template <bool SHADED>
struct CandArea {
  float beta[3][kCandRing];   // brick coordinates
  float v[kCandRing];         // value (without stencil-maximum bricks)
  float step[kCandRing];      // world length of a sample step
  int leaf[kCandRing];
  int k_lane[kCandRing];      // sample number (bits 0..22) and its ray's lane (23..27)
  int rec[kCandRing];         // segment record
  unsigned taken[kCandRing];  // samples the ray has taken up to this one
  unsigned own[32];           // per lane: which of the 32 candidates at hand are its own
  float w[32];                // opacity, then compositing weight; kNoWeight: not opaque
};
template <>
struct CandArea<false> {
  float beta[3][kCandRing];
  float v[kCandRing];
  float step[kCandRing];
  int leaf[kCandRing];
  int k_lane[kCandRing];
  unsigned taken[kCandRing];
  unsigned own[32];
  float w[32];
  float3 col[32];
};
constexpr float kNoWeight = -2.0f;
constexpr unsigned kCrowded = 512;
constexpr float kDenseSlack = 4096.0f;  // segments (in 32s) before the density counts

// The bits of a warp's `count` tasks (lane q holds the owner of task q) that belong to the
// calling lane.
__device__ __forceinline__ unsigned own_tasks(unsigned* own, int lane, unsigned lt_mask, int owner,
                                              int count) {
  own[lane] = 0;
  __syncwarp();
  const unsigned same = __match_any_sync(0xffffffffu, lane < count ? owner : -1);
  if (lane < count && (same & lt_mask) == 0) own[owner] = same;
  __syncwarp();
  return own[lane];
}

// samples whose stencil maxima (with stencil-maximum bricks) or values (without) a lane
// takes together
#ifndef AMR_SPLIT_GROUP
#define AMR_SPLIT_GROUP 8
#endif
#ifndef AMR_SPLIT_VALUES
#define AMR_SPLIT_VALUES 4
#endif
// Samples a lane takes between fetches: shaded, the caller's samples_per_iter, which the host
// has checked to lie in [1, 64]; unshaded (schedule 0, where that field has no meaning and any
// value) a constant.  At least one group either way, so that every pass makes progress.
constexpr int kPlainStep = 16;
static_assert(kPlainStep >= AMR_SPLIT_GROUP, "a pass takes samples");

// A warp's part of the workspace while it marches: its block of segment records.
struct SegBlock {
  int base = 0, used = kSegBlock;
};

// The march of pixel (i, j) of view R by one lane of a warp whose 32 lanes all call this
// together (lanes without a pixel pass active = false).  Shaded: px receives the headlight
// direction and the opacity, tile the first chunk and the number of the warp's tasks, and segs
// the segments its rays fetched; unshaded: px receives the pixel.  Returns kTileDone, or why the tile was given up.
enum { kTileDone = 0, kTileNoRoom = 1, kTileDense = 2 };
template <int ST, int SHADE>
__device__ __forceinline__ int march_tile(const RenderArgs& A, const RayArgs& R, int i, int j,
                                           bool active, const float4* s_tf, const int* s_nz,
                                           float clear_below, CandArea<(SHADE & 3) != 0>& Q,
                                           RayF& rf, SegBlock& blk, int tile_id, int view, float4& px,
                                           int2& tile, int& segs, unsigned& nsamp,
                                           unsigned long long& status) {
  constexpr bool MX = (SHADE & kShadeMaxBit) != 0;  // the stencil-maximum test
  constexpr bool SHADED = (SHADE & 3) != 0;
  const unsigned FULL = 0xffffffffu;
  constexpr int RM = kCandRing - 1;
  const int lane = (int)(threadIdx.x + blockDim.x * threadIdx.y) & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  bool live = false;
  px = make_float4(0.f, 0.f, 0.f, 0.f);
  {
    RayX rx;
    if (active && make_ray(R, i, j, rx)) {
      make_frame(R, rx, rf);
      live = true;
    }
  }
  if (SHADED && live) {
    const float inv_dn = 1.0f / rf.dn;
    px.x = -rf.Dd[0] * (float)R.hf[0] * inv_dn;
    px.y = -rf.Dd[1] * (float)R.hf[1] * inv_dn;
    px.z = -rf.Dd[2] * (float)R.hf[2] * inv_dn;
  }
  int pid0 = kPidIn, seg = 0, prev = -1;
  float tau0 = 0.f, e0 = 0.f;
  uint32_t start = 0;
  SegSetup g;
  MaxWalk<ST> walk;
  g.s.n = 0;
  int k = 0, rec = -1;
  float Acc = 0.f;
  unsigned taken = 0;       // samples of this ray
  bool over = false;        // early ray termination
  // bounds the ray has met; kept only if it did not end, by a sample evaluated later, before
  // it met them: the first two stop the ray, the third counts for samples after raised_at
  constexpr int kMetSegments = 1, kMetTree = 2, kMetSamples = 4;
  int met = 0;
  unsigned raised_at = 0;
  int nc = 0, hc = 0;       // warp-uniform: candidates queued, and the first one's slot
  int tasks = 0, chunk = 0; // warp-uniform: tasks written, and the chunk being filled
  int first = -1;
  bool full = false;        // warp-uniform: the tile is given up

  // evaluate the first `count` candidates, add each lane's own opacities in order, and write
  // (unshaded: composite) the opaque ones
  auto evaluate = [&](int count) {
    __syncwarp();
    const int q = (hc + lane) & RM;
    int owner = lane;
    float v = 0.f;
    Q.w[lane] = kNoWeight;
    if (lane < count) {
      owner = Q.k_lane[q] >> kTaskSampleBits;
      if constexpr (MX) {
        const BrickRef b = leaf_brick(A.patches, A.leaves[Q.leaf[q]]);
        v = trilinear<ST>(A, b, Q.beta[0][q], Q.beta[1][q], Q.beta[2][q]);
      } else {
        v = Q.v[q];
      }
      if constexpr (SHADED) {
        const float a = tf_alpha(s_tf, A.tf_n, v, A.vmin, A.inv_range);
        if (a > 0.0f) Q.w[lane] = -expm1f(-A.kappa * a * Q.step[q]);
      } else {
        const float4 c = tf_lookup(s_tf, A.tf_n, v, A.vmin, A.inv_range);
        if (c.w > 0.0f) Q.w[lane] = -expm1f(-A.kappa * c.w * Q.step[q]);
        Q.col[lane] = make_float3(c.x, c.y, c.z);
      }
    }
    unsigned m = own_tasks(Q.own, lane, lt_mask, owner, count);
    if constexpr (SHADED) {
      for (; m != 0; m &= m - 1) {
        const int e = __ffs(m) - 1;
        const float alpha = Q.w[e];
        if (alpha == kNoWeight) continue;
        if (over) {  // beyond the ray's end
          Q.w[e] = kNoWeight;
          continue;
        }
        const float w = (1.0f - Acc) * alpha;
        Q.w[e] = w;
        Acc += w;
        if (Acc >= A.ert_thresh) {  // early ray termination: later samples were not taken
          over = true;
          live = false;
          taken = Q.taken[(hc + e) & RM];
          met = taken > raised_at ? met & kMetSamples : 0;
        }
      }
    } else {
      for (; m != 0 && !over; m &= m - 1) {
        const int e = __ffs(m) - 1;
        const float alpha = Q.w[e];
        if (alpha == kNoWeight) continue;
        const float w = (1.0f - Acc) * alpha;
        const float3 c = Q.col[e];
        px.x = fmaf(w, c.x, px.x);
        px.y = fmaf(w, c.y, px.y);
        px.z = fmaf(w, c.z, px.z);
        Acc += w;
        if (Acc >= A.ert_thresh) {
          over = true;
          live = false;
          taken = Q.taken[(hc + e) & RM];
          met = taken > raised_at ? met & kMetSamples : 0;
        }
      }
    }
    __syncwarp();
    if constexpr (SHADED) {
      const float w = Q.w[lane];
      const unsigned om = __ballot_sync(FULL, w != kNoWeight);
      const int n = __popc(om);
      if (n != 0) {
        const int at = tasks & (kTaskChunk - 1);
        const int room = at == 0 ? 0 : kTaskChunk - at;
        int fresh = chunk;
        if (n > room) {
          if (lane == 0) {
            const unsigned c = tasks / kTaskChunk < A.ts.tile_chunks
                                   ? atomicAdd(A.ts.heads + kHeadChunk, 1u) : ~0u;
            fresh = c < (unsigned)A.ts.chunks ? (int)c : -1;
            if (fresh >= 0) {
              A.ts.meta[fresh] = make_int4(tile_id, 0, -1, view);
              if (tasks != 0) {  // the chunk is full
                A.ts.meta[chunk].y = kTaskChunk;
                A.ts.meta[chunk].z = fresh;
              }
            }
          }
          fresh = __shfl_sync(FULL, fresh, 0);
          if (fresh < 0) {
            full = true;
            live = false;
            fresh = chunk;
          } else if (first < 0) {
            first = fresh;
          }
        }
        if (!full && w != kNoWeight) {
          const int o = __popc(om & lt_mask);
          const size_t slot = o < room ? (size_t)chunk * kTaskChunk + at + o
                                       : (size_t)fresh * kTaskChunk + (o - room);
          A.ts.tasks[slot] = make_float4(__int_as_float(Q.rec[q]), __int_as_float(Q.k_lane[q]), v, w);
        }
        chunk = fresh;
        if (!full) tasks += n;
      }
      __syncwarp();
    }
    nc -= count;
    hc += count;
  };

  // Every pass either fetches segments for at least one lane or takes samples, and each
  // ray has finitely many of both, so the loop ends with every lane's ray finished.
  for (;;) {
    const bool flush = !__any_sync(FULL, live);  // every ray has ended: only the queue is left
    if ((flush && nc == 0) || full) break;
    // lanes whose segment ended fetch their next non-empty one (waiting for 8, 16 or 24 of
    // them was no faster)
    if (live && k >= g.s.n) {
      for (;;) {
        if (pid0 == kPidOut) {
          live = false;
          break;
        }
        if (seg >= A.max_segments) {
          met |= kMetSegments;
          live = false;
          break;
        }
        ++seg;
        int pid1 = kPidOut;
        float tau1 = rf.tau_out, e1 = exit_bound(rf);
        const int lmin = lod_min_level(R, A.lv, rf, i, j, pid0, tau0, e0);
        const int lid = next_leaf(A.nodes, A.leaves, A.face_node, A.node_box, R, i, j, rf,
                                  start, prev, pid0, tau0, e0, pid1, tau1, e1, lmin);
        if (lid < 0) {
          met |= kMetTree;
          live = false;
          break;
        }
        prev = lid;
        const DLeaf lf = A.leaves[lid];
        const DLevel& lv = A.lv[lf.level];
        int n = segment_count(R, i, j, rf, pid0, tau0, e0, pid1, tau1, e1, lv);
        if (n > kMaxSamplesPerSegment) {
          if (!(met & kMetSamples)) raised_at = taken;
          met |= kMetSamples;
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
        rec = -1;
        pid0 = pid1;  // where the next segment starts
        tau0 = tau1;
        e0 = e1;
        break;
      }
    }
    // A lane takes its next G samples at a time: a mask of those that may be opaque (by
    // their stencil maxima, or by their values), queued in order.  Most masks are empty.
    constexpr int G = MX ? AMR_SPLIT_GROUP : AMR_SPLIT_VALUES;
    const int steps = SHADED ? A.samples_per_iter : kPlainStep;
    for (int step = 0; step < steps; step += G) {
      const int kb = k;
      const int cnt = live ? min(min(G, steps - step), g.s.n - k) : 0;
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
      }
      if constexpr (SHADED) {
        // the record of a segment, written with its first candidate
        const unsigned need = __ballot_sync(FULL, mask != 0 && rec < 0);
        if (need != 0) {
          const int n = __popc(need);
          if (blk.used + n > kSegBlock) {
            unsigned b = 0;
            if (lane == 0) b = atomicAdd(A.ts.heads + kHeadSegBlock, 1u);
            b = __shfl_sync(FULL, b, 0);
            if (b >= (unsigned)A.ts.seg_blocks) {
              full = true;
              break;
            }
            blk.base = (int)b * kSegBlock;
            blk.used = 0;
          }
          if (mask != 0 && rec < 0) {
            rec = blk.base + blk.used + __popc(need & lt_mask);
            float4* s = A.ts.segs + 3 * (size_t)rec;
            s[0] = make_float4(g.b0[0], g.b0[1], g.b0[2], g.db[0]);
            s[1] = make_float4(g.db[1], g.db[2], g.s.margin, __int_as_float(g.s.leaf));
            s[2] = make_float4(__int_as_float(g.s.pid0), __int_as_float(g.s.pid1),
                               __int_as_float(g.s.n), 0.0f);
          }
          blk.used += n;
        }
      }
      for (;;) {
        const unsigned cm = __ballot_sync(FULL, mask != 0);
        if (mask != 0) {
          const int e = __ffs(mask) - 1;
          mask &= mask - 1;
          const int kk = kb + e;
          const int q = (hc + nc + __popc(cm & lt_mask)) & RM;
#pragma unroll
          for (int a = 0; a < 3; ++a) Q.beta[a][q] = fmaf((float)kk, g.db[a], g.b0[a]);
          if constexpr (!MX) {
            float v = val[0];
#pragma unroll
            for (int z = 1; z < G; ++z) v = e == z ? val[z] : v;
            Q.v[q] = v;
          }
          Q.step[q] = g.delta;
          Q.leaf[q] = leaf_of(g.s.leaf);
          Q.k_lane[q] = kk | (lane << kTaskSampleBits);
          if constexpr (SHADED) Q.rec[q] = rec;
          Q.taken[q] = taken + (unsigned)e + 1u;
        }
        nc += __popc(cm);
        if (nc >= 32 || (flush && nc != 0)) {
          evaluate(min(nc, 32));
          if (!live) mask = 0;  // ended: its later samples were not taken
        }
        if (full || (cm == 0 && nc < 32)) break;
      }
      if (live) taken += (unsigned)cnt;
      if (flush || full) break;
    }
  }
  if constexpr (SHADED) {
    tile = make_int2(first, tasks);
    segs = __reduce_add_sync(FULL, seg);
  }
  if (full) return tasks / kTaskChunk >= A.ts.tile_chunks ? kTileDense : kTileNoRoom;
  if (SHADED && lane == 0 && tasks != 0) {
    const int last = tasks & (kTaskChunk - 1);
    A.ts.meta[chunk].y = last == 0 ? kTaskChunk : last;
  }
  nsamp += taken;
  if (met & (kMetSegments | kMetSamples)) status |= kStatusCapacity;
  if (met & kMetTree) status |= kStatusDevice;
  px.w = Acc;
  return kTileDone;
}

// resident blocks the register budgets allow for.  The ray frame (22 words, read once per
// segment) lies in shared memory; measured, ms, frame in registers / shared, shaded with 4
// blocks: atlas 512^2 1.87 / 1.78, 640 x 479 2.44 / 2.39, 1024^2 7.00 / 6.81, 32-view batch 25.2 /
// 24.3 (5 blocks 2.03, 2.59, 7.16, 26.0); unshaded f16 1917 x 1083 4.39 in registers with 4
// blocks, shared with 4 / 5 / 6 / 7 blocks 4.54 / 4.28 / 4.65 / 5.09.
#ifndef AMR_SPLIT_MARCH_BLOCKS
#define AMR_SPLIT_MARCH_BLOCKS 4
#endif
#ifndef AMR_SPLIT_PLAIN_BLOCKS
#define AMR_SPLIT_PLAIN_BLOCKS 5
#endif
#ifndef AMR_SPLIT_SHADE_BLOCKS
#define AMR_SPLIT_SHADE_BLOCKS 6
#endif
#ifndef AMR_SPLIT_OUTER_BLOCKS
#define AMR_SPLIT_OUTER_BLOCKS 8
#endif

// Persistent warps taking 8x4-pixel tiles from a queue, as march_kernel does.
template <int ST, int SHADE, typename Args = RenderArgs>
__global__ void __launch_bounds__(128, (SHADE & 3) != 0 ? AMR_SPLIT_MARCH_BLOCKS : AMR_SPLIT_PLAIN_BLOCKS)
    split_march_kernel(const __grid_constant__ Args P) {
  constexpr bool SHADED = (SHADE & 3) != 0;
  const RenderArgs& A = render_args(P);
  const int n_tiles = count_tiles(P);
  unsigned ready = 0;  // tiles that earlier rounds gave up
  float warps = 0.0f;  // that will have a tile at once
  if constexpr (SHADED) {
    ready = __ldcg(A.ts.heads + kHeadReady);
    const unsigned again = ready - min(__ldcg(A.ts.heads + kHeadRest), ready);
    const unsigned todo = (unsigned)n_tiles - min(__ldcg(A.ts.heads + kHeadTile), (unsigned)n_tiles) + again;
    if (todo == 0) return;
    // so many tiles found no room that half as many go at once
    if (again >= kCrowded && (blockIdx.x & 1)) return;
    warps = (float)min(gridDim.x * (again >= kCrowded ? 2u : 4u), todo);
  }
  extern __shared__ float4 smem[];
  const int tid = threadIdx.x + blockDim.x * threadIdx.y;
  using Area = CandArea<SHADED>;
  Area& Q = reinterpret_cast<Area*>(reinterpret_cast<char*>(smem) +
                                    StagedTf<Args>::bytes(P))[tid >> 5];
  const StagedTf<Args> staged(P, smem, tid);
  if constexpr (SHADED && std::is_same<Args, RenderArgs>::value)
    if (staged.clear <= A.dense_below) return;  // every tile is dense (below)
  const int lane = tid & 31;
  unsigned nsamp = 0;
  unsigned long long status = 0;
  SegBlock blk;
  __shared__ RayFSlot s_rf[128];
  RayF& rf = s_rf[tid].f;
  // each pass takes one tile, and the queue hands out every tile once
  for (;;) {
    int t = n_tiles;
    if (lane == 0) {
      if constexpr (SHADED) {
        // Room is kept for the tiles that are under way: a quarter of the pool, or what as many
        // tiles as there are warps take on average (with a quarter alone, dense tiles were given
        // up by the hundred and marched again).  An image with more tasks per segment than
        // pays is left to the one-kernel march from there on.
        const unsigned* H = A.ts.heads;
        const float taken = (float)max(__ldcg(H + kHeadTile), 1u), tasks = (float)__ldcg(H + kHeadTasks);
        const float chunks = tasks * (32.0f / kTaskChunk) / taken;  // of a tile, but for its last
        const float room = fmaxf(0.25f * (float)A.ts.chunks, warps * fminf(chunks + 0.5f, 2.0f * chunks));
        if ((float)__ldcg(H + kHeadChunk) + room < (float)A.ts.chunks &&
            __ldcg(H + kHeadSegBlock) < (unsigned)(A.ts.seg_blocks - A.ts.seg_blocks / 4) &&
            tasks <= A.ts.dense_ratio * ((float)__ldcg(H + kHeadSegs) + kDenseSlack)) {
          t = (int)min(atomicAdd(A.ts.heads + kHeadTile, 1u), (unsigned)n_tiles);
          if (t == n_tiles && ready != 0) {
            // (a warp that takes one too many puts it back)
            const unsigned r = atomicAdd(A.ts.heads + kHeadRest, 1u);
            if (r < ready) t = __ldcg(A.ts.left + r);
            else atomicSub(A.ts.heads + kHeadRest, 1u);
          }
        }
      } else {
        t = (int)min(atomicAdd(A.counters + kQueueCounter, 1ull), (unsigned long long)n_tiles);
      }
    }
    t = __shfl_sync(0xffffffffu, t, 0);
    if (t >= n_tiles) break;
    const TileAt p = tile_at(P, t);
    const RayArgs& R = tile_rays(P, p);
    int i, jr;
    p.pixel(lane, i, jr);
    const int j = R.row0 + jr;
    const bool active = i < p.width && jr < p.rows && j < R.height;
    float4 px;
    int2 tile = make_int2(-1, 0);
    int segs = 0;
    // nearly everything opaque: one kernel is faster (640 x 479, 480 opaque samples a pixel:
    // 16.1 ms alone, 24.7 after a workspace full of tasks), so the tile is left to it
    int how = kTileDense;
    if (!SHADED || staged.clear_below(p) > A.dense_below)
      how = march_tile<ST, SHADE>(A, R, i, j, active, staged.tf(p), staged.nz(p),
                                  staged.clear_below(p), Q, rf, blk, t, p.view, px, tile, segs, nsamp,
                                  status);
    if constexpr (SHADED) {
      if (lane == 0 && segs != 0) {
        atomicAdd(A.ts.heads + kHeadTasks, (unsigned)(tile.y + 31) >> 5);
        atomicAdd(A.ts.heads + kHeadSegs, (unsigned)(segs + 31) >> 5);
      }
    }
    if (how == kTileDone) {
      if (SHADED && tile.y == 0) px = make_float4(0.f, 0.f, 0.f, px.w);  // nothing to shade
      if (active) p.out[p.at(i, jr)] = px;
      if (SHADED && lane == 0 && tile.y != 0) A.ts.tile[t] = tile;
    } else if (lane == 0) {
      if (how == kTileDense) A.ts.dense[atomicAdd(A.ts.heads + kHeadDense, 1u)] = t;
      else A.ts.left[atomicAdd(A.ts.heads + kHeadLeft, 1u)] = t;
    }
  }
  const unsigned total = __reduce_add_sync(0xffffffffu, nsamp);
  if (lane == 0 && total) atomicAdd(A.counters, (unsigned long long)total);
  if (status) atomicOr(A.counters + 1, status);
}

// The segment and brick position of a task.
__device__ __forceinline__ SegState task_segment(const RenderArgs& A, int rec, int k, int px, int py,
                                                 float* beta) {
  const float4* r = A.ts.segs + 3 * (size_t)rec;
  const float4 r0 = __ldcg(r), r1 = __ldcg(r + 1), r2 = __ldcg(r + 2);
  SegState s;
  s.leaf = __float_as_int(r1.w);
  const DLeaf lf = A.leaves[leaf_of(s.leaf)];
  s.brick = leaf_brick(A.patches, lf);
  s.level = lf.level;
  leaf_bounds(lf, A.lv[lf.level], s.brick, lod_of(s.leaf), s.leaf_lo, s.bl, s.bh);
  s.margin = r1.z;
  s.pid0 = __float_as_int(r2.x);
  s.pid1 = __float_as_int(r2.y);
  s.n = __float_as_int(r2.z);
  s.px = px;
  s.py = py;
  beta[0] = fmaf((float)k, r0.w, r0.x);
  beta[1] = fmaf((float)k, r1.x, r0.y);
  beta[2] = fmaf((float)k, r1.y, r0.z);
  return s;
}

// Colour of a task of value v whose gradient is gr; L the headlight direction, T the
// transmittance to the light.
template <int SHADE>
__device__ __forceinline__ float3 task_colour(const RenderArgs& A, const float4* s_tf, float v,
                                              const DLevel& lv, const float* gr, float4 L, float T) {
  const float4 c = tf_lookup(s_tf, A.tf_n, v, A.vmin, A.inv_range);
  float cr = c.x, cg = c.y, cb = c.z;
  phong(A, lv, gr, L.x, L.y, L.z, cr, cg, cb);
  if constexpr ((SHADE & kShadeShadow) != 0) {
    const float I = fmaf(1.0f - A.light_ambient, T, A.light_ambient);
    cr *= I;
    cg *= I;
    cb *= I;
  }
  return make_float3(cr, cg, cb);
}

// Shade every task whose gradient stays in its leaf, one per lane, and list the others.
template <int ST, int SHADE, typename Args = RenderArgs>
__global__ void __launch_bounds__(128, AMR_SPLIT_SHADE_BLOCKS)
    split_shade_kernel(const __grid_constant__ Args P) {
  extern __shared__ float4 smem[];
  const RenderArgs& A = render_args(P);
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, lane = tid & 31;
  const int units = (int)min(__ldcg(A.ts.heads + kHeadChunk), (unsigned)A.ts.chunks) * (kTaskChunk / 32);
  if ((int)blockIdx.x * 4 >= units) return;
  const StagedTf<Args> staged(P, smem, tid);
  for (int u = blockIdx.x * 4 + (tid >> 5); u < units; u += gridDim.x * 4) {
    const int4 meta = __ldcg(A.ts.meta + u / (kTaskChunk / 32));
    const int count = min(32, meta.y - (u % (kTaskChunk / 32)) * 32);
    if (count <= 0) continue;
    const TileAt p = chunk_tile(P, meta);
    const RayArgs& R = tile_rays(P, p);
    const float4* tf = staged.tf(p);
    const int slot = u * 32 + lane;
    bool inner = true;
    float4 t;
    int level = 0;
    float x[3] = {0.f, 0.f, 0.f}, gr[3] = {0.f, 0.f, 0.f};
    float4 L;
    if (lane < count) {
      t = __ldcg(A.ts.tasks + slot);
      const int kl = __float_as_int(t.y);
      int i, jr;
      p.pixel(kl >> kTaskSampleBits, i, jr);
      L = __ldcg(p.out + p.at(i, jr));
      float beta[3];
      const SegState s = task_segment(A, __float_as_int(t.x), kl & ((1 << kTaskSampleBits) - 1),
                                      i, R.row0 + jr, beta);
      level = s.level;
      inner = gradient_inner(s, beta);
      if (inner) gradient_brick<ST, (SHADE & 3) == 2>(A, s.brick, beta, A.lv[level], gr);
      if constexpr ((SHADE & kShadeShadow) != 0) {
        const float sc = (float)A.lv[level].sc;
#pragma unroll
        for (int a = 0; a < 3; ++a) x[a] = (beta[a] - 0.5f + (float)s.brick.lo[a]) * sc;
      }
    }
    float T = 1.0f;
    if constexpr ((SHADE & kShadeShadow) != 0) {
      // the samples' light rays, one after the other, each by the whole warp
      for (int e = 0; e < count; ++e) {
        const float Te = warp_shadow_transmittance<ST>(A, R, tf, __shfl_sync(FULL, x[0], e),
                                                       __shfl_sync(FULL, x[1], e),
                                                       __shfl_sync(FULL, x[2], e));
        if (lane == e) T = Te;
      }
    }
    if (lane < count) {
      float3 c = make_float3(T, 0.f, 0.f);  // an outer task's transmittance waits here
      if (inner) c = task_colour<SHADE>(A, tf, t.z, A.lv[level], gr, L, T);
      A.ts.col[slot] = make_float4(c.x, c.y, c.z, t.w);
    }
    const unsigned outer = __ballot_sync(FULL, !inner);
    if (outer != 0) {
      unsigned at = 0;
      if (lane == 0) at = atomicAdd(A.ts.heads + kHeadOuter, (unsigned)__popc(outer));
      at = __shfl_sync(FULL, at, 0);
      if (!inner) A.ts.outer[at + __popc(outer & ((1u << lane) - 1u))] = slot;
    }
  }
}

// Shade the listed tasks: six lanes take one's six neighbours, five tasks per warp.
template <int ST, int SHADE, typename Args = RenderArgs>
__global__ void __launch_bounds__(128, AMR_SPLIT_OUTER_BLOCKS)
    split_outer_kernel(const __grid_constant__ Args P) {
  extern __shared__ float4 smem[];
  const RenderArgs& A = render_args(P);
  const unsigned FULL = 0xffffffffu;
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, lane = tid & 31;
  const int n = (int)__ldcg(A.ts.heads + kHeadOuter);
  if ((int)blockIdx.x * 20 >= n) return;
  const StagedTf<Args> staged(P, smem, tid);
  const int e = lane / 6, q = lane % 6, ax = q >> 1;
  const float sg = (q & 1) ? -1.0f : 1.0f;
  for (int b = (blockIdx.x * 4 + (tid >> 5)) * 5; b < n; b += gridDim.x * 20) {
    const bool on = e < 5 && b + e < n;
    int slot = 0, level = 0, i = 0, jr = 0;
    float4 t = make_float4(0.f, 0.f, 0.f, 0.f);
    float v = 0.f;
    TileAt p = {};
    if (on) {
      slot = __ldcg(A.ts.outer + b + e);
      t = __ldcg(A.ts.tasks + slot);
      const int kl = __float_as_int(t.y), k = kl & ((1 << kTaskSampleBits) - 1);
      p = chunk_tile(P, __ldcg(A.ts.meta + slot / kTaskChunk));
      const RayArgs& R = tile_rays(P, p);
      p.pixel(kl >> kTaskSampleBits, i, jr);
      float bn[3];
      const SegState s = task_segment(A, __float_as_int(t.x), k, i, R.row0 + jr, bn);
      level = s.level;
      bn[0] += ax == 0 ? sg : 0.0f;
      bn[1] += ax == 1 ? sg : 0.0f;
      bn[2] += ax == 2 ? sg : 0.0f;
      v = neighbour_at<ST, 1>(A, R, s, A.lv[level], bn, k, ax, sg);
    }
    float w[6];
#pragma unroll
    for (int z = 0; z < 6; ++z) w[z] = __shfl_down_sync(FULL, v, z);
    if (on && q == 0) {
      const DLevel& lv = A.lv[level];
      const float gr[3] = {(w[0] - w[1]) * lv.ginv[0], (w[2] - w[3]) * lv.ginv[1],
                           (w[4] - w[5]) * lv.ginv[2]};
      const float4 L = __ldcg(p.out + p.at(i, jr));
      const float T = (SHADE & kShadeShadow) != 0 ? __ldcg(&A.ts.col[slot].x) : 1.0f;
      const float3 c = task_colour<SHADE>(A, staged.tf(p), t.z, lv, gr, L, T);
      A.ts.col[slot] = make_float4(c.x, c.y, c.z, t.w);
    }
  }
}

// Add up each tile's colours: every lane those of its pixel, in sample order.
struct SumArea {
  float4 col[32];
  unsigned own[32];
};
template <typename Args>
__global__ void __launch_bounds__(128) split_sum_kernel(const __grid_constant__ Args P) {
  __shared__ SumArea area[4];
  const RenderArgs& A = render_args(P);
  if (blockIdx.x == 0 && threadIdx.x + threadIdx.y == 0)
    A.ts.heads[kHeadReady] = __ldcg(A.ts.heads + kHeadLeft);
  if (__ldcg(A.ts.heads + kHeadChunk) == 0) return;  // an empty round
  const int tid = threadIdx.x + blockDim.x * threadIdx.y, lane = tid & 31;
  const unsigned lt_mask = (1u << lane) - 1u;
  SumArea& Q = area[tid >> 5];
  const int n_tiles = count_tiles(P);
  for (int t = blockIdx.x * 4 + (tid >> 5); t < n_tiles; t += gridDim.x * 4) {
    const int2 tile = __ldcg(A.ts.tile + t);
    if (tile.y < 0) continue;  // none, or of another round
    float C0 = 0.f, C1 = 0.f, C2 = 0.f;
    int chunk = tile.x;
    for (int b = 0; b < tile.y; b += 32) {
      if (b != 0 && (b & (kTaskChunk - 1)) == 0) chunk = __ldcg(&A.ts.meta[chunk].z);
      const int count = min(32, tile.y - b);
      int owner = lane;
      if (lane < count) {
        const size_t slot = (size_t)chunk * kTaskChunk + (b & (kTaskChunk - 1)) + lane;
        owner = __float_as_int(__ldcg(&A.ts.tasks[slot].y)) >> kTaskSampleBits;
        Q.col[lane] = __ldcg(A.ts.col + slot);
      }
      for (unsigned m = own_tasks(Q.own, lane, lt_mask, owner, count); m != 0; m &= m - 1) {
        const float4 c = Q.col[__ffs(m) - 1];
        C0 = fmaf(c.w, c.x, C0);
        C1 = fmaf(c.w, c.y, C1);
        C2 = fmaf(c.w, c.z, C2);
      }
      __syncwarp();
    }
    const TileAt p = tile_at(P, t);
    int i, jr;
    p.pixel(lane, i, jr);
    if (i < p.width && jr < p.rows && tile_rays(P, p).row0 + jr < tile_rays(P, p).height) {
      float4* o = p.out + p.at(i, jr);
      *o = make_float4(C0, C1, C2, __ldcg(&o->w));
    }
    if (lane == 0) A.ts.tile[t].y = -1;
  }
}

// The rays of a batch's views.
static __global__ void __launch_bounds__(kMaxBatchViews) batch_views_kernel(const __grid_constant__ BatchArgs B) {
  const int v = threadIdx.x;
  if (v >= B.n_views) return;
  RayArgs r = B.A.ray;
  const BatchView& b = B.v[v];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    r.eye[a] = b.eye[a];
    r.fwd[a] = b.fwd[a];
    r.right[a] = b.right[a];
    r.up[a] = b.up[a];
  }
  r.tan_half_fov_y = b.tan_half_fov_y;
  r.width = b.width;
  r.height = b.height;
  r.row0 = 0;
  r.rows = b.height;
  r.lod_scale = b.lod_scale;
  r.lod_scale_f = b.lod_scale_f;
  B.A.ts.views[v] = r;
}

}  // namespace amr
