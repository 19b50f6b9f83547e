// Upload of the tree, leaves, patch table and bricks to the device, in one of the four
// brick storage strategies (Sec. 4.1 packed pool, Sec. 4.2 handle table, rebuilt for CUDA).
#include <algorithm>
#include <cstring>
#include <deque>
#include <new>

#include "ctx.h"
#include "storage16.h"

namespace amr {

namespace {

#define CK(call)                                                                      \
  do {                                                                                \
    cudaError_t e_ = (call);                                                          \
    if (e_ != cudaSuccess)                                                            \
      return fail(c, e_ == cudaErrorMemoryAllocation ? AMR_ERR_OOM : AMR_ERR_CUDA,    \
                  std::string(#call) + ": " + cudaGetErrorString(e_));                \
  } while (0)

// breadth-first re-layout: children of a node are adjacent, the top levels contiguous;
// lod receives each slot's pruned-leaf entry (id << 5 | level) or -1, box each slot's box
// (lo, hi as two int4, finest cells) starting from the root box with the highest label
// level of a type-(a) node above the slot in lo.w, leaf_anc that level per leaf
std::vector<DNode> layout_nodes(const Tree& t, const int64_t* root, std::vector<int32_t>& lod,
                                std::vector<int32_t>& slot_of, std::vector<int4>& box,
                                std::vector<int32_t>& leaf_anc) {
  const size_t n = t.axis.size();
  std::vector<DNode> out(n);
  lod.assign(n, -1);
  slot_of.assign(n, 0);
  box.assign(2 * std::max<size_t>(n, 1), make_int4(0, 0, 0, 0));
  leaf_anc.assign(t.leaf_patch.size(), -1);
  struct Item {
    int pre, slot;
    int32_t b[6];
    int32_t anc;  // highest label level of a type-(a) node above this one, -1: none
  };
  std::deque<Item> q;
  Item r{0, 0, {}, -1};
  for (int k = 0; k < 6; ++k) r.b[k] = (int32_t)root[k];
  q.push_back(r);
  int next = 1;
  while (!q.empty()) {
    const Item it = q.front();
    q.pop_front();
    const int pre = it.pre, slot = it.slot;
    slot_of[pre] = slot;
    box[2 * (size_t)slot] = make_int4(it.b[0], it.b[1], it.b[2], it.anc);
    box[2 * (size_t)slot + 1] = make_int4(it.b[3], it.b[4], it.b[5], 0);
    const int32_t lq = t.node_lod.empty() ? -1 : t.node_lod[pre];
    const int32_t lvl = lq >= 0 ? t.lod_level[(size_t)lq - t.leaf_patch.size()] : -1;
    if (lq >= 0) lod[slot] = (lq << 5) | lvl;
    DNode d;
    if (t.axis[pre] < 0) {
      d.meta = ((uint32_t)kLeafAxis << 30) | ((uint32_t)t.leaf[pre] & kIndexMask);
      d.split = 0;
      leaf_anc[(size_t)t.leaf[pre]] = it.anc;
    } else {
      int first = next;
      next += 2;
      const int ax = t.axis[pre];
      d.meta = ((uint32_t)ax << 30) | ((uint32_t)first & kIndexMask);
      d.split = t.split[pre];
      const int32_t anc = std::max(it.anc, lvl);
      Item lc{t.left[pre], first, {}, anc}, rc{t.right[pre], first + 1, {}, anc};
      std::memcpy(lc.b, it.b, sizeof lc.b);
      std::memcpy(rc.b, it.b, sizeof rc.b);
      lc.b[3 + ax] = t.split[pre];
      rc.b[ax] = t.split[pre];
      q.push_back(lc);
      q.push_back(rc);
    }
    out[slot] = d;
  }
  return out;
}

// Macro grid over the root for point location: cells of G finest cells per axis (G = the
// finest cells of one level-0 cell, doubled until the grid has at most 2^21 cells), each
// holding the slot of the deepest node whose box contains the whole cell.  A point lies
// in its cell, so a descent from that node reaches the same leaf as one from the root.
std::vector<uint32_t> macro_grid(const std::vector<DNode>& nodes, const int64_t* root, int64_t R,
                                 int32_t* cell, int32_t* dims) {
  int64_t G = std::max<int64_t>(R, 1), ext[3], n[3];
  for (int a = 0; a < 3; ++a) ext[a] = root[3 + a] - root[a];
  for (;;) {
    for (int a = 0; a < 3; ++a) n[a] = (ext[a] + G - 1) / G;
    if (n[0] * n[1] * n[2] <= ((int64_t)1 << 21)) break;
    G *= 2;
  }
  *cell = (int32_t)G;
  for (int a = 0; a < 3; ++a) dims[a] = (int32_t)n[a];
  std::vector<uint32_t> out((size_t)(n[0] * n[1] * n[2]), 0u);
#pragma omp parallel for schedule(static)
  for (long long gi = 0; gi < (long long)out.size(); ++gi) {
    const int64_t g[3] = {gi % n[0], (gi / n[0]) % n[1], gi / (n[0] * n[1])};
    int64_t lo[3], hi[3];
    for (int a = 0; a < 3; ++a) {
      lo[a] = root[a] + g[a] * G;
      hi[a] = std::min(root[a] + (g[a] + 1) * G, root[3 + a]);
    }
    uint32_t i = 0;
    for (int depth = 0; depth < kMaxDepth; ++depth) {
      const DNode& nd = nodes[i];
      const uint32_t ax = nd.meta >> 30;
      if (ax == (uint32_t)kLeafAxis) break;
      const uint32_t c0 = nd.meta & kIndexMask;
      if (hi[ax] <= nd.split) i = c0;
      else if (lo[ax] >= nd.split) i = c0 + 1;
      else break;
    }
    out[(size_t)gi] = i;
  }
  return out;
}

// Bricks of element type T (float values, or float4 value + central differences) in the
// layout of the context's storage strategy; fills base (or gbase) of every patch record.
template <typename T>
amr_status upload_bricks(amr_ctx* c, const std::vector<std::vector<T>>& bricks,
                         std::vector<DPatch>& pt, bool gradient, cudaStream_t stream) {
  DeviceState& d = c->dev;
  const size_t P = c->patches.size();
  const int storage = c->storage;
  void*& pool = gradient ? d.gpool : d.pool;
  size_t& pool_bytes = gradient ? d.gpool_bytes : d.pool_bytes;
  auto set_base = [&](size_t p, long long v) { (gradient ? pt[p].gbase : pt[p].base) = v; };
  const cudaChannelFormatDesc ch = cudaCreateChannelDesc<T>();
  cudaTextureDesc td;
  std::memset(&td, 0, sizeof td);
  td.addressMode[0] = td.addressMode[1] = td.addressMode[2] = cudaAddressModeClamp;
  td.filterMode = cudaFilterModePoint;
  td.readMode = cudaReadModeElementType;
  td.normalizedCoords = 0;
  if (storage == AMR_STORE_PTR || storage == AMR_STORE_TEXOBJ) {
    // the kernels address a per-patch brick with 32-bit element offsets
    for (size_t p = 0; p < P; ++p)
      if (bricks[p].size() >= ((size_t)1 << 31))
        return fail(c, AMR_ERR_CAPACITY, "a brick holds 2^31 cells or more");
  }
  if (storage == AMR_STORE_PTR) {
    // one pool, each brick 128-byte aligned; the table holds the device addresses
    std::vector<size_t> off(P);
    size_t elems = 0;
    const size_t align = 128 / sizeof(T);
    for (size_t p = 0; p < P; ++p) {
      off[p] = elems;
      elems += (bricks[p].size() + align - 1) / align * align;
    }
    pool_bytes = elems * sizeof(T);
    CK(cudaMalloc(&pool, pool_bytes));
    for (size_t p = 0; p < P; ++p) {
      T* dst = (T*)pool + off[p];
      CK(cudaMemcpyAsync(dst, bricks[p].data(), bricks[p].size() * sizeof(T),
                         cudaMemcpyHostToDevice, stream));
      set_base(p, (long long)(uintptr_t)dst);
      pt[p].sy = pt[p].dim[0];
      pt[p].sz = pt[p].dim[0] * pt[p].dim[1];
    }
  } else if (storage == AMR_STORE_TEXOBJ) {
    std::vector<void*>& arrays = gradient ? d.garrays : d.arrays;
    std::vector<cudaTextureObject_t>& tex = gradient ? d.gtexobjs : d.texobjs;
    arrays.assign(P, nullptr);
    tex.assign(P, 0);
    pool_bytes = 0;
    for (size_t p = 0; p < P; ++p) {
      cudaExtent ext = make_cudaExtent(pt[p].dim[0], pt[p].dim[1], pt[p].dim[2]);
      cudaArray_t arr = nullptr;
      CK(cudaMalloc3DArray(&arr, &ch, ext));
      arrays[p] = arr;
      cudaMemcpy3DParms cp;
      std::memset(&cp, 0, sizeof cp);
      cp.srcPtr = make_cudaPitchedPtr((void*)bricks[p].data(), pt[p].dim[0] * sizeof(T),
                                      pt[p].dim[0], pt[p].dim[1]);
      cp.dstArray = arr;
      cp.extent = ext;
      cp.kind = cudaMemcpyHostToDevice;
      CK(cudaMemcpy3DAsync(&cp, stream));
      cudaResourceDesc rd;
      std::memset(&rd, 0, sizeof rd);
      rd.resType = cudaResourceTypeArray;
      rd.res.array.array = arr;
      cudaTextureObject_t t = 0;
      CK(cudaCreateTextureObject(&t, &rd, &td, nullptr));
      tex[p] = t;
      set_base(p, (long long)t);
      pool_bytes += bricks[p].size() * sizeof(T);
    }
    CK(cudaStreamSynchronize(stream));
  } else {
    // packed atlas (NFDH), linear memory or one 3D array
    const int64_t AX = c->packing.dims[0], AY = c->packing.dims[1], AZ = c->packing.dims[2];
    const size_t total = (size_t)(AX * AY * AZ);
    std::vector<T> img(total);
    std::memset((void*)img.data(), 0, total * sizeof(T));
    for (size_t p = 0; p < P; ++p) {
      const int64_t* o = &c->packing.org[3 * p];
      const int64_t d0 = pt[p].dim[0], d1 = pt[p].dim[1], d2 = pt[p].dim[2];
      for (int64_t k = 0; k < d2; ++k)
        for (int64_t j = 0; j < d1; ++j)
          std::memcpy((void*)&img[(size_t)(o[0] + AX * ((o[1] + j) + AY * (o[2] + k)))],
                      &bricks[p][(size_t)(d0 * (j + d1 * k))], sizeof(T) * (size_t)d0);
      for (int a = 0; a < 3; ++a) pt[p].org[a] = (int32_t)o[a];
      set_base(p, (long long)(o[0] + AX * (o[1] + AY * o[2])));
      pt[p].sy = (int32_t)AX;
      pt[p].sz = (int32_t)(AX * AY);
    }
    pool_bytes = total * sizeof(T);
    if (storage == AMR_STORE_ATLAS_LINEAR) {
      CK(cudaMalloc(&pool, pool_bytes));
      CK(cudaMemcpyAsync(pool, img.data(), pool_bytes, cudaMemcpyHostToDevice, stream));
      CK(cudaStreamSynchronize(stream));
    } else {
      cudaDeviceProp prop;
      CK(cudaGetDeviceProperties(&prop, d.device));
      if (AX > prop.maxTexture3D[0] || AY > prop.maxTexture3D[1] || AZ > prop.maxTexture3D[2])
        return fail(c, AMR_ERR_CAPACITY, "atlas exceeds the 3D texture extent limit");
      cudaExtent ext = make_cudaExtent(AX, AY, AZ);
      cudaArray_t arr = nullptr;
      CK(cudaMalloc3DArray(&arr, &ch, ext));
      (gradient ? d.gatlas_array : d.atlas_array) = arr;
      cudaMemcpy3DParms cp;
      std::memset(&cp, 0, sizeof cp);
      cp.srcPtr = make_cudaPitchedPtr(img.data(), AX * sizeof(T), AX, AY);
      cp.dstArray = arr;
      cp.extent = ext;
      cp.kind = cudaMemcpyHostToDevice;
      CK(cudaMemcpy3DAsync(&cp, stream));
      cudaResourceDesc rd;
      std::memset(&rd, 0, sizeof rd);
      rd.resType = cudaResourceTypeArray;
      rd.res.array.array = arr;
      CK(cudaCreateTextureObject(gradient ? &d.gatlas_tex : &d.atlas_tex, &rd, &td, nullptr));
      CK(cudaStreamSynchronize(stream));
    }
  }
  return AMR_OK;
}

// Stencil-maximum bricks of the pointer storage: a second pool with the value pool's
// offsets (the same brick sizes and alignment), so a brick's maximum brick lies at a fixed
// byte distance (mpool - pool) from it.
template <typename T>
amr_status upload_max_pool(amr_ctx* c, const std::vector<std::vector<T>>& mb, cudaStream_t stream) {
  DeviceState& d = c->dev;
  const size_t P = mb.size();
  const size_t align = 128 / sizeof(T);
  std::vector<size_t> off(P);
  size_t elems = 0;
  for (size_t p = 0; p < P; ++p) {
    off[p] = elems;
    elems += (mb[p].size() + align - 1) / align * align;
  }
  if (elems * sizeof(T) != d.pool_bytes)
    return fail(c, AMR_ERR_STATE, "stencil-maximum pool does not match the brick pool");
  CK(cudaMalloc(&d.mpool, elems * sizeof(T)));
  for (size_t p = 0; p < P; ++p)
    CK(cudaMemcpyAsync((T*)d.mpool + off[p], mb[p].data(), mb[p].size() * sizeof(T),
                       cudaMemcpyHostToDevice, stream));
  return AMR_OK;
}

}  // namespace

// Workspace of the split march: a pool (36 bytes a task, and a segment record of 48 bytes for
// every third) and records of its tiles.  The pool has kTasksPerPixel tasks for every pixel - the
// 5-level hierarchy with a ramp transfer function takes 23, and 8 segment records -, up to
// kMaxTasks, but kTileChunks chunks (320 tasks a pixel) for every tile under way, so that dense
// tiles need not be given up: 1.7 GB for most images, 3.5 GB at most.  (With 40 tasks a pixel
// alone, at 640 x 479 tiles were given up and the frame took 5.4 instead of 2.7 ms.)
static constexpr int64_t kTasksPerPixel = 40, kTileChunks = 80;
static constexpr int64_t kMaxTasks = (int64_t)1 << 26;
static constexpr int64_t kWarps = 152 * 16;  // of the march, at once

// Rounds for so many tasks a pixel; the one-kernel march takes what they leave.
static int64_t task_rounds(int64_t tiles, int64_t chunks, int64_t per_pixel) {
  const int64_t usable = (chunks - chunks / 4) * kTaskChunk;
  return std::min<int64_t>(64, (tiles * 32 * per_pixel + usable - 1) / usable);
}

int TaskPlan::rounds(long long tiles_of_band) const {
  return (int)std::min<int64_t>(task_rounds(tiles_of_band, ts.chunks, per_pixel),
                                left / std::max(1LL, tiles_of_band));
}

// A larger buffer in place of b; the old one is freed (the last call's work has ended then), or
// kept for the captured calls that hold its address.  False, and b as it was, when out of memory.
static bool replace_buffer(DeviceState& d, TaskBuffer& b, size_t bytes) {
  try {
    d.task_retired.reserve(d.task_retired.size() + 1);
  } catch (const std::bad_alloc&) {
    return false;
  }
  // (relaxed: another thread's capture must not be disturbed, nor refuse this)
  cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
  cudaThreadExchangeStreamCaptureMode(&mode);
  void* p = nullptr;
  const bool ok = cudaMalloc(&p, bytes) == cudaSuccess;
  if (!ok) {
    cudaGetLastError();
  } else {
    if (b.captured) {
      d.task_retired.push_back(b.p);
    } else if (b.p) {
      cudaEventSynchronize(d.work_event);
      cudaFree(b.p);
    }
    b.p = p;
    b.captured = false;
  }
  cudaThreadExchangeStreamCaptureMode(&mode);
  return ok;
}

// Offsets of consecutive arrays, each on a 256-byte boundary; returns the bytes of all.
template <int N>
static size_t lay_out(const size_t (&bytes)[N], size_t (&off)[N]) {
  size_t at = 0;
  for (int k = 0; k < N; ++k) {
    off[k] = at;
    at += (bytes[k] + 255) & ~(size_t)255;
  }
  return at;
}

static void grow_pool(DeviceState& d, int64_t tiles) {
  const int64_t under_way = std::min(tiles, kWarps) * kTileChunks * kTaskChunk * 4 / 3;
  const int64_t most = kMaxTasks / kTaskChunk;
  const int64_t need =
      std::min(std::max(tiles * 32 * kTasksPerPixel, under_way) / kTaskChunk, most);
  if (need <= d.tasks.chunks || need >= d.task_refused) return;
  int64_t chunks = std::max(need, std::min<int64_t>(2 * (int64_t)d.tasks.chunks, most));
  if (fault_injected("small_pool")) chunks = std::min<int64_t>(chunks, 256);
  const size_t slots = (size_t)chunks * kTaskChunk;
  const int64_t blocks = (int64_t)slots / 3 / kSegBlock + 2 * kWarps;
  const size_t sizes[7] = {slots * sizeof(float4), slots * sizeof(float4), slots * sizeof(int32_t),
                           (size_t)chunks * sizeof(int4),
                           (size_t)blocks * kSegBlock * 3 * sizeof(float4),
                           kHeads * sizeof(unsigned), kMaxBatchViews * sizeof(RayArgs)};
  size_t off[7];
  if (!replace_buffer(d, d.task_pool, lay_out(sizes, off))) {
    d.task_refused = need;
    return;
  }
  char* p = (char*)d.task_pool.p;
  d.tasks.tasks = (float4*)(p + off[0]);
  d.tasks.col = (float4*)(p + off[1]);
  d.tasks.outer = (int32_t*)(p + off[2]);
  d.tasks.meta = (int4*)(p + off[3]);
  d.tasks.segs = (float4*)(p + off[4]);
  d.tasks.heads = (unsigned*)(p + off[5]);
  d.tasks.views = (RayArgs*)(p + off[6]);
  d.tasks.chunks = (int32_t)chunks;
  d.tasks.seg_blocks = (int32_t)blocks;
}

// (the list of tiles given up is as long as the rounds of the pool at hand need it; a larger
// pool needs fewer)
static void grow_tiles(DeviceState& d, int64_t need) {
  if (need <= d.task_tile_cap || need >= d.task_tiles_refused) return;
  int64_t tiles = std::max(need, std::min(2 * d.task_tile_cap, kTaskTiles));
  if (fault_injected("few_tiles")) tiles = std::min<int64_t>(tiles, 240);
  const int64_t left = tiles * task_rounds(tiles, d.tasks.chunks, 128);
  const size_t sizes[3] = {(size_t)tiles * sizeof(int2), (size_t)left * sizeof(int32_t),
                           (size_t)tiles * sizeof(int32_t)};
  size_t off[3];
  if (!replace_buffer(d, d.task_tiles, lay_out(sizes, off))) {
    d.task_tiles_refused = need;
    return;
  }
  char* p = (char*)d.task_tiles.p;
  d.tasks.tile = (int2*)(p + off[0]);
  d.tasks.left = (int32_t*)(p + off[1]);
  d.tasks.dense = (int32_t*)(p + off[2]);
  d.task_tile_cap = tiles;
  d.task_left_cap = left;
}

// Where the split march pays.  It saves segment fetches their latency and pays for every task's
// way through memory, so what decides is the tasks per segment (counted as tiles are done), how
// dear a fetch is (the leaves), and how well rays of large images stay together in the one-kernel
// marches; small images wait for their longest rays.  Measured at 300^2 to 2048^2 on hierarchies of
// 77 to 32,198 leaves with transfer functions that make 2 to 100 % of the cells opaque (ms, split
// / one kernel, tasks per segment): 1,175 leaves 1024^2 3.19 / 3.41 (2.3), 5.11 / 4.82 (4.9);
// 3,998 leaves 1024^2 5.59 / 5.81 (3.5), 8.26 / 7.26 (5.6), 640 x 479 2.92 / 3.34 (7.6), 2048^2 9.56
// / 9.94 (1.0), 11.8 / 11.3 (1.5); 30,164 leaves 1024^2 14.7 / 16.0 (4.1), 21.3 / 20.5 (6.6), 2048^2
// 28.8 / 30.8 (1.7), 38.7 / 37.2 (2.8); 32,198 leaves of 1,150 cells, where every fourth gradient
// leaves its leaf, 1500 x 1100 8.1 / 11.3 (2.0), 2048^2 33.8 / 36.0 (3.3); 77 leaves 64^2 0.23 /
// 0.33, 256^2 0.308 / 0.303, 1024^2 1.26 / 1.02, batches of 64 views of 64^2 0.59 / 0.70, of 4 of
// 900^2 3.71 / 2.52.
constexpr int64_t kFewLeaves = 1000, kManyLeaves = 10000;  // of the hierarchy
constexpr double kSmallLeaf = 2000.0;                      // cells
constexpr int64_t kFewTiles = 1024;      // images that gain on any hierarchy,
constexpr int64_t kFewViewTiles = 4096;  // and batches, with fewer tiles per view than this
constexpr int64_t kWaveTiles = 600000 / 32;  // images of a few tiles per warp: no time to stop

TaskPlan plan_tasks(amr_ctx* c, long long call_tiles, TaskUse use, void* stream, int views) {
  TaskPlan plan;
  DeviceState& d = c->dev;
  const int64_t leaves = (int64_t)c->tree.leaf_patch.size();
  const bool many = leaves >= kManyLeaves;
  if (call_tiles <= 0) return plan;
  if (use != TaskUse::shadow && leaves < kFewLeaves &&
      call_tiles > (use == TaskUse::batch ? views * kFewViewTiles : kFewTiles))
    return plan;
  if (use == TaskUse::image && !many && call_tiles * 32 >= kLargePixels) return plan;
  const int64_t tiles = std::min<int64_t>(call_tiles, kTaskTiles);
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing((cudaStream_t)stream, &cap) != cudaSuccess) cudaGetLastError();
  if (cap == cudaStreamCaptureStatusNone) {
    grow_pool(d, tiles);
    if (d.tasks.chunks > 0) grow_tiles(d, tiles);
  } else {
    d.task_pool.captured = d.task_tiles.captured = true;
  }
  plan.ts = d.tasks;
  plan.tiles = d.task_tile_cap;
  plan.left = d.task_left_cap;
  const bool small_leaves = many && d.leaf_cells < kSmallLeaf;
  plan.ts.dense_ratio = use == TaskUse::shadow ? INFINITY
                        : use == TaskUse::image && tiles * 32 >= kLargePixels
                            ? (small_leaves ? 4.0f : 2.5f)
                        : small_leaves || tiles < kWaveTiles ? 12.0f
                                                             : (many ? 6.0f : 4.3f);
  // Rounds for the densest images that are not stopped (a round that finds nothing to do costs
  // four launches, about 10 us).
  plan.per_pixel = use == TaskUse::image && (!many || tiles * 32 >= kLargePixels) ? 64 : 128;
  // Not begun at all: transfer functions that make four fifths of the cells opaque, or half of
  // them where the pool cannot hold the image whatever it shows.
  const bool holds = (int64_t)d.tasks.chunks * kTaskChunk >= tiles * 32 * 250;
  plan.dense_below = small_leaves || holds || use != TaskUse::image ? d.fifth_below : d.half_below;
  plan.ts.tile_chunks = (int32_t)std::max<int64_t>(
      1, 3 * (int64_t)d.tasks.chunks / std::min(std::max<int64_t>(1, std::min(tiles, d.task_tile_cap)), kWarps));
  return plan;
}

void release_device(amr_ctx* c) {
  DeviceState& d = c->dev;
  if (d.device >= 0) cudaSetDevice(d.device);
  if (d.atlas_tex) cudaDestroyTextureObject(d.atlas_tex);
  if (d.gatlas_tex) cudaDestroyTextureObject(d.gatlas_tex);
  for (auto t : d.texobjs)
    if (t) cudaDestroyTextureObject(t);
  for (auto t : d.gtexobjs)
    if (t) cudaDestroyTextureObject(t);
  for (void* a : d.arrays)
    if (a) cudaFreeArray((cudaArray_t)a);
  for (void* a : d.garrays)
    if (a) cudaFreeArray((cudaArray_t)a);
  if (d.atlas_array) cudaFreeArray((cudaArray_t)d.atlas_array);
  if (d.gatlas_array) cudaFreeArray((cudaArray_t)d.gatlas_array);
  cudaFree(d.gpool);
  cudaFree(d.mpool);
  cudaFree(d.nodes);
  cudaFree(d.lod);
  cudaFree(d.face_node);
  cudaFree(d.face_list);
  cudaFree(d.node_box);
  cudaFree(d.macro);
  cudaFree(d.leaves);
  cudaFree(d.patches);
  cudaFree(d.pool);
  cudaFree(d.counters);
  cudaFree(d.tf_scratch);
  cudaFree(d.proposal);
  cudaFree(d.img_scratch);
  cudaFree(d.log_counts);
  cudaFree(d.log_offsets);
  cudaFree(d.task_pool.p);
  cudaFree(d.task_tiles.p);
  for (void* p : d.task_retired) cudaFree(p);
  if (d.work_event) cudaEventDestroy(d.work_event);
  d = DeviceState();
  c->device_built = false;
}

// The leaves beyond face f (2 axis + side) of leaf m, all in the subtree of pre-order node
// `pre`, as a list at the end of `lists` (RayArgs::face_list): its word there, or -1 when there
// are too many, their rectangles do not fit the bytes, or the face is one of the root's.
static int32_t face_list(const Tree& t, const int64_t* root, size_t m, int f, int32_t pre,
                          int32_t slot, std::vector<int4>& lists) {
  const int32_t* box = &t.leaf_box[6 * m];
  const int a = f >> 1, b = a == 0 ? 1 : 0, c = a == 2 ? 1 : 2;
  const int64_t plane = (f & 1) ? box[3 + a] : box[a];
  if (plane == ((f & 1) ? root[3 + a] : root[a])) return -1;
  const int64_t cell = (f & 1) ? plane : plane - 1;  // the finest cells beyond the face
  struct Rect { int32_t u0, u1, v0, v1, id; };
  Rect r[kFaceListMax];
  int n = 0;
  std::vector<int32_t> stack(1, pre);
  while (!stack.empty()) {
    const int32_t i = stack.back();
    stack.pop_back();
    const int ax = t.axis[i];
    if (ax < 0) {
      const int32_t id = t.leaf[i];
      const int32_t* q = &t.leaf_box[6 * (size_t)id];
      if (n == kFaceListMax) return -1;
      r[n++] = {std::max(q[b], box[b]) - box[b], std::min(q[3 + b], box[3 + b]) - box[b],
                   std::max(q[c], box[c]) - box[c], std::min(q[3 + c], box[3 + c]) - box[c], id};
      continue;
    }
    const int64_t sp = t.split[i], lo = ax == a ? cell : box[ax], hi = ax == a ? cell + 1 : box[3 + ax];
    if (lo < sp) stack.push_back(t.left[i]);
    if (hi > sp) stack.push_back(t.right[i]);
  }
  int32_t bits = 0;  // the rectangles' unit: the largest power of two in all their corners
  for (int k = 0; k < n; ++k) bits |= r[k].u0 | r[k].u1 | r[k].v0 | r[k].v1;
  if (bits == 0) return -1;
  const int shift = __builtin_ctz((unsigned)bits);
  for (int k = 0; k < n; ++k)
    if ((r[k].u1 >> shift) > 255 || (r[k].v1 >> shift) > 255) return -1;
  const size_t word = lists.size();
  lists.push_back(int4{box[b], box[c], slot, n + 32 * shift});
  for (int k = 0; k < n; k += 2) {
    int4 w = {0, 0, 0, 0};
    for (int e = 0; e < 2 && k + e < n; ++e) {
      const Rect& q = r[k + e];
      const uint32_t p = (uint32_t)(q.u0 >> shift) | (uint32_t)(q.u1 >> shift) << 8 |
                         (uint32_t)(q.v0 >> shift) << 16 | (uint32_t)(q.v1 >> shift) << 24;
      (e == 0 ? w.x : w.z) = (int)p;
      (e == 0 ? w.y : w.w) = q.id;
    }
    lists.push_back(w);
  }
  return (int32_t)word;
}

// The values a fifth and half of the bricks' cells lie below, from at most about 2^16 of them.
static void low_quantiles(amr_ctx* c) {
  size_t cells = 0, at = 0;
  for (const auto& b : c->bricks) cells += b.size();
  const size_t stride = std::max<size_t>(1, cells >> 16);
  std::vector<float> v;
  for (const auto& b : c->bricks) {
    for (; at < b.size(); at += stride)
      if (!std::isnan(b[at])) v.push_back(b[at]);
    at -= b.size();
  }
  c->dev.fifth_below = c->dev.half_below = -INFINITY;
  if (v.empty()) return;
  const auto half = v.begin() + v.size() / 2, fifth = v.begin() + v.size() / 5;
  std::nth_element(v.begin(), half, v.end());
  c->dev.half_below = *half;
  if (fifth != half) std::nth_element(v.begin(), fifth, half);
  c->dev.fifth_below = *fifth;
}

amr_status upload(amr_ctx* c, void* stream_v) {
  cudaStream_t stream = (cudaStream_t)stream_v;
  if (c->device_built) release_device(c);
  DeviceState& d = c->dev;
  low_quantiles(c);
  double cells = 0.0;
  for (const Patch& q : c->patches) cells += (double)(q.n[0] * q.n[1] * q.n[2]);
  d.leaf_cells = cells / std::max<size_t>(1, c->tree.leaf_patch.size());
  CK(cudaGetDevice(&d.device));
  if (!d.work_event) CK(cudaEventCreateWithFlags(&d.work_event, cudaEventDisableTiming));
  const Tree& t = c->tree;
  const size_t P = c->patches.size();
  const size_t M = t.leaf_patch.size();
  if (t.axis.size() >= (size_t)kIndexMask || M >= (size_t)kIndexMask)
    return fail(c, AMR_ERR_CAPACITY, "tree too large for 30-bit node indices");
  std::vector<int32_t> lodv, slot_of;
  std::vector<int4> boxes;
  std::vector<int32_t> leaf_anc;
  std::vector<DNode> nodes = layout_nodes(t, c->root, lodv, slot_of, boxes, leaf_anc);
  if (fault_injected("corrupt_node") && nodes.size() > 1 &&
      (nodes[0].meta >> 30) != (uint32_t)kLeafAxis)
    nodes[0].meta &= ~kIndexMask;  // the root's children become slots 0 (itself) and 1
  std::vector<int32_t> face_slots(std::max<size_t>(1, 18 * M), 0);
  for (size_t k = 0; k < t.face_node.size(); ++k) {
    const int32_t pre = t.face_node[k];
    face_slots[k] = t.axis[pre] < 0 ? (int32_t)(kFaceLeaf | (uint32_t)t.leaf[pre]) : slot_of[pre];
  }
  // the ropes: the nodes holding the cells beyond the faces alone, again
  for (size_t m = 0; m < M; ++m)
    std::copy_n(&face_slots[12 * m + 6], 6, &face_slots[12 * M + 6 * m]);
  // leaf lists for the ropes whose node is an inner one: per leaf, then one after the other
  std::vector<std::vector<int4>> leaf_lists(M);
  std::vector<int32_t> list_word(6 * M, -1);
  bool no_memory = false;  // (an exception may not leave the parallel loop)
#pragma omp parallel for schedule(dynamic, 256)
  for (long long m = 0; m < (long long)M; ++m) {
    try {
      for (int f = 0; f < 6; ++f) {
        const int32_t pre = t.face_node[12 * (size_t)m + 6 + f];
        if (t.axis[pre] >= 0)
          list_word[6 * (size_t)m + f] =
              face_list(t, c->root, (size_t)m, f, pre, slot_of[pre], leaf_lists[(size_t)m]);
      }
    } catch (const std::bad_alloc&) {
#pragma omp atomic write
      no_memory = true;
    }
  }
  if (no_memory) throw std::bad_alloc();
  std::vector<int4> face_lists;
  for (size_t m = 0; m < M; ++m) {
    const size_t base = face_lists.size();
    if (base + leaf_lists[m].size() >= (size_t)kFaceList) break;
    face_lists.insert(face_lists.end(), leaf_lists[m].begin(), leaf_lists[m].end());
    for (int f = 0; f < 6; ++f)
      if (list_word[6 * m + f] >= 0)
        face_slots[12 * M + 6 * m + f] = (int32_t)(kFaceList | (uint32_t)(base + list_word[6 * m + f]));
  }
  face_lists.resize(face_lists.size() + kFaceListMax / 2, int4{0, 0, 0, 0});
  const size_t ML = t.lod_patch.size();
  if (M + ML >= ((size_t)1 << 26)) return fail(c, AMR_ERR_CAPACITY, "too many leaves");
  std::vector<DLeaf> leaves(M + ML);
  for (size_t m = 0; m < M + ML; ++m) {
    DLeaf& l = leaves[m];
    std::memset(&l, 0, sizeof l);
    const bool lod = m >= M;
    const int32_t* box = lod ? &t.lod_box[6 * (m - M)] : &t.leaf_box[6 * m];
    for (int k = 0; k < 6; ++k) (k < 3 ? l.lo[k] : l.hi[k - 3]) = box[k];
    l.patch = lod ? t.lod_patch[m - M] : t.leaf_patch[m];
    l.level = lod ? t.lod_level[m - M] : t.leaf_level[m];
    l.faces = (lod || t.leaf_faces.empty()) ? 0 : t.leaf_faces[m];
    l.lod_anc = lod ? -1 : leaf_anc[m];
    // the range of the cells as stored; rounding is monotone, so the rounded extremes
    // bound every rounded cell and empty-space skipping stays exact
    l.vmin = storage_round(c->dtype, c->leaf_vmin[m]);
    l.vmax = storage_round(c->dtype, c->leaf_vmax[m]);
  }
  std::vector<DPatch> pt(P);
  for (size_t p = 0; p < P; ++p) {
    std::memset(&pt[p], 0, sizeof(DPatch));
    for (int a = 0; a < 3; ++a) {
      // brick index = cell - lo + 1 in every kernel: a halo of H cells shifts lo by H - 1
      pt[p].lo[a] = (int32_t)(c->patches[p].box[a] - (c->halo - 1));
      pt[p].dim[a] = (int32_t)(c->patches[p].n[a] + 2 * c->halo);
    }
  }
  if (fault_injected("oom")) return fail(c, AMR_ERR_OOM, "injected device allocation failure");
  CK(cudaMalloc(&d.nodes, nodes.size() * sizeof(DNode)));
  CK(cudaMalloc(&d.lod, lodv.size() * sizeof(int32_t)));
  CK(cudaMalloc(&d.face_node, face_slots.size() * sizeof(int32_t)));
  CK(cudaMalloc(&d.face_list, face_lists.size() * sizeof(int4)));
  CK(cudaMalloc(&d.node_box, boxes.size() * sizeof(int4)));
  CK(cudaMalloc(&d.leaves, std::max<size_t>(1, M + ML) * sizeof(DLeaf)));
  CK(cudaMalloc(&d.patches, P * sizeof(DPatch)));
  CK(cudaMalloc(&d.counters, kNumCounters * sizeof(unsigned long long)));
  const std::vector<uint32_t> macro = macro_grid(nodes, c->root, c->R, &d.macro_cell, d.macro_dims);
  CK(cudaMalloc(&d.macro, macro.size() * sizeof(uint32_t)));
  CK(cudaMemcpyAsync(d.macro, macro.data(), macro.size() * sizeof(uint32_t),
                     cudaMemcpyHostToDevice, stream));
  CK(cudaMemsetAsync(d.counters, 0, kNumCounters * sizeof(unsigned long long), stream));

  amr_status st;
  if (c->dtype == AMR_F32) {
    st = upload_bricks<float>(c, c->bricks, pt, false, stream);
    if (st != AMR_OK) return st;
    if (c->want_max && c->storage == AMR_STORE_PTR) {
      st = upload_max_pool<float>(c, c->mbricks, stream);
      if (st != AMR_OK) return st;
    }
    if (c->want_gradient) {
      st = upload_bricks<float4>(c, c->gbricks, pt, true, stream);
      if (st != AMR_OK) return st;
    }
  } else {
    // 16-bit cells (and 4 x 16-bit value + central differences)
    {
      std::vector<std::vector<uint16_t>> b16(P);
#pragma omp parallel for schedule(dynamic, 4)
      for (long long pi = 0; pi < (long long)P; ++pi) {
        const size_t p = (size_t)pi;
        const std::vector<float>& b = c->bricks[p];
        b16[p].resize(b.size());
        for (size_t i = 0; i < b.size(); ++i) b16[p][i] = storage_bits(c->dtype, b[i]);
      }
      st = upload_bricks<uint16_t>(c, b16, pt, false, stream);
      if (st != AMR_OK) return st;
      if (c->want_max && c->storage == AMR_STORE_PTR) {
        // the maximum of the rounded cells is the rounded maximum (rounding is monotone)
#pragma omp parallel for schedule(dynamic, 4)
        for (long long pi = 0; pi < (long long)P; ++pi) {
          const size_t p = (size_t)pi;
          const std::vector<float>& m = c->mbricks[p];
          for (size_t i = 0; i < m.size(); ++i) b16[p][i] = storage_bits(c->dtype, m[i]);
        }
        st = upload_max_pool<uint16_t>(c, b16, stream);
        if (st != AMR_OK) return st;
      }
    }
    if (c->want_gradient) {
      std::vector<std::vector<ushort4>> g16(P);
#pragma omp parallel for schedule(dynamic, 4)
      for (long long pi = 0; pi < (long long)P; ++pi) {
        const size_t p = (size_t)pi;
        const std::vector<float4>& g = c->gbricks[p];
        g16[p].resize(g.size());
        for (size_t i = 0; i < g.size(); ++i)
          g16[p][i] = make_ushort4(storage_bits(c->dtype, g[i].x), storage_bits(c->dtype, g[i].y),
                                   storage_bits(c->dtype, g[i].z), storage_bits(c->dtype, g[i].w));
      }
      st = upload_bricks<ushort4>(c, g16, pt, true, stream);
      if (st != AMR_OK) return st;
    }
  }
  CK(cudaMemcpyAsync(d.nodes, nodes.data(), nodes.size() * sizeof(DNode), cudaMemcpyHostToDevice,
                     stream));
  CK(cudaMemcpyAsync(d.lod, lodv.data(), lodv.size() * sizeof(int32_t), cudaMemcpyHostToDevice,
                     stream));
  CK(cudaMemcpyAsync(d.face_list, face_lists.data(), face_lists.size() * sizeof(int4),
                     cudaMemcpyHostToDevice, stream));
  CK(cudaMemcpyAsync(d.face_node, face_slots.data(), face_slots.size() * sizeof(int32_t),
                     cudaMemcpyHostToDevice, stream));
  CK(cudaMemcpyAsync(d.node_box, boxes.data(), boxes.size() * sizeof(int4), cudaMemcpyHostToDevice,
                     stream));
  for (DLeaf& l : leaves) {  // brick addressing, now that the bricks are placed
    const DPatch& q = pt[(size_t)l.patch];
    l.base = q.base;
    l.gbase = q.gbase;
    l.sy = q.sy;
    l.sz = q.sz;
    for (int a = 0; a < 3; ++a) {
      l.blo[a] = q.lo[a];
      l.dim[a] = q.dim[a];
    }
  }
  if (M + ML)
    CK(cudaMemcpyAsync(d.leaves, leaves.data(), (M + ML) * sizeof(DLeaf), cudaMemcpyHostToDevice,
                       stream));
  CK(cudaMemcpyAsync(d.patches, pt.data(), P * sizeof(DPatch), cudaMemcpyHostToDevice, stream));
  CK(cudaStreamSynchronize(stream));
  CK(cudaEventRecord(d.work_event, stream));
  c->device_built = true;
  return AMR_OK;
}

}  // namespace amr
