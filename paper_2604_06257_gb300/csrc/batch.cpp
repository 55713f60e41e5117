// batch.cpp -- ragged batches of DAS instances (host side): a persistent launch over the lane
// mappings, and launches over the frame tiles of repacked instances.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>
#include <memory>
#include <new>
#include <stdexcept>
#include <vector>

#include "mach.h"
#include "mach_internal.h"

using namespace mach;

struct mach_batch_s {
  int n = 0;
  int iq_dtype = 0;
  std::vector<mach_plan> plans;          // tables of each instance
  std::vector<BatchInstance> host_insts;
  std::vector<mach_tile_shape> shapes;
  BatchInstance* d_insts = nullptr;
  int2* d_items = nullptr;
  int* d_counter = nullptr;
  int n_items = 0;
  int grid = 0;
  int per_sm = 0;
  size_t slot_bytes = 128;               // ring slot of the staged path (largest staged window)
  std::vector<void*> bounds;             // 2 per instance (null: not staged): tile boxes, transmit-delay ranges
  int64_t points = 0;
  bool bound = false;
  // repacked instances: what each needs before the shared launches, and the launches (one
  // per exact-frame shape and kMultiMax entries)
  struct Repacked {
    int inst, dtype, F, tiles;
    int64_t TC, V;
    int S, range[2];                     // samples per row, those that windows touch
    size_t at;                           // its bytes in the workspace below
    size_t pd_at;
  };
  struct Multi {
    Variant v;
    MultiArgs args;
    int2* d_items;
    int n_items;
  };
  std::vector<Repacked> repacked;
  std::vector<std::unique_ptr<Multi>> multi;
  char* ws = nullptr;
};

namespace {

void drop_repacked(mach_batch_s* b) {
  for (auto& m : b->multi) cudaFree(m->d_items);
  cudaFree(b->ws);
  b->multi.clear();
  b->repacked.clear();
  b->ws = nullptr;
}

void release(mach_batch_s* b) {
  if (!b) return;
  for (mach_plan p : b->plans) mach_plan_destroy(p);
  for (void* q : b->bounds) cudaFree(q);
  drop_repacked(b);
  cudaFree(b->d_insts);
  cudaFree(b->d_items);
  cudaFree(b->d_counter);
  delete b;
}

int voxels_per_block(const mach_tile_shape& s) {
  if (s.mode == kBatchChannels) return 32;
  if (s.mode == kBatchStaged) return 7 * 4 * (32 / s.frame_lanes);   // 7 consumer warps + a producer warp
  if (s.frame_lanes == 2) return 8 * 2 * 16;   // 8 warps x 16 lane pairs x 2 voxels
  return 8 * 4 * (32 / s.frame_lanes);         // 8 warps x (32 / FL) lane groups x 4 voxels
}

// Default lane mapping (measured on the 64-instance float16 batch): channel lanes for
// F <= 4; staged windows for F > 16 when F is not a multiple of 4 (rows off the 16-byte
// grid: the L1 path then reads one sample per frame from global memory, the staged path
// from shared memory); frame lanes through L1 otherwise, as few lanes per voxel as cover F.
mach_tile_shape default_shape(int F) {
  mach_tile_shape s{};
  if (F <= 4) {
    s.mode = kBatchChannels;
    s.frame_lanes = 0;
  } else if (F > 16 && F % 4 != 0) {
    s.mode = kBatchStaged;
    s.frame_lanes = F <= 32 ? 8 : 16;
  } else {
    s.mode = kBatchFrames;
    s.frame_lanes = F <= 8 ? 2 : F <= 16 ? 4 : (F <= 32 ? 8 : 16);
  }
  return s;
}

// The frame-lane mapping an instance falls back to when its staged windows do not fit.
mach_tile_shape frames_shape(int F) {
  mach_tile_shape s{};
  s.mode = kBatchFrames;
  s.frame_lanes = F <= 8 ? 2 : F <= 16 ? 4 : (F <= 32 ? 8 : 16);
  return s;
}

// Default voxel box of a staged block: shallow and wide (a window spans ~2 sample rows
// per voxel of depth but a fraction of a row per voxel of width).
void staged_tile(int n, int nx, int ny, int nz, bool list, int tile[3]) {
  if (list || (ny == 1 && nz == 1)) {
    tile[0] = n; tile[1] = 1; tile[2] = 1;
  } else if (ny == 1) {
    tile[0] = n / 4; tile[1] = 1; tile[2] = 4;
  } else {   // 112 = 4 x 4 x 7, 56 = 4 x 2 x 7
    tile[0] = 4; tile[1] = n / 28; tile[2] = 7;
  }
}

// Which instances are repacked (bytes of `repack`, one per plan).  Repacking an instance takes launches
// of its own, in which the others wait; the lane mappings share one persistent launch but do more
// work per term.  Microseconds of either, fitted to batches of 30 equal float16 and complex64
// instances (2D of 48^2 ... 128^2 px, 3D of 28^3 voxels, 1 and 3 transmits, F-numbers 1 ... 3, 5 to 64
// frames; lanes within a tenth, repacked runs within a sixth, half of the time):
//  * lanes: every (voxel, element) and (voxel, element, transmit) is looked at, terms inside the
//    aperture take the lanes' frame slots; staged windows skip most of the rest;
//  * repacked: the pass, a reduction when there are several frame tiles, points and terms.
// The launch of the lane mappings takes 25 us at least.  Both are estimates, so lanes have to be a
// third cheaper.  Against always repacking (3, 6, 12 and 30 equal instances): 0.7 to 7.8 times the
// speed, hardly ever below 1; against never repacking 0.54 ... 8, in 90 of 100 above 0.85.  In a mixed batch a
// persistent launch of a few small instances is all tail (ten float16 instances 3.58 ms, 3.77 with
// the four small ones on lanes).
void choose_repacked(const std::vector<mach_plan>& plans, const mach_das_desc* descs, std::vector<char>& repack) {
  constexpr double kLaunch = 9.0, kReduce = 4.0, kFloor = 25.0, kMargin = 1.3;
  std::vector<char> cheap(plans.size(), 0);   // lanes would be cheaper
  double lanes_sum = 0.0, repacked_sum = 0.0;
  for (size_t i = 0; i < plans.size(); ++i) {
    RepackNeeds q;
    if (!plan_repack(plans[i], &q)) continue;
    repack[i] = 1;
    const DasParams& p = *plan_params(plans[i]);
    const FrameSplit fs = split_frames(p.F);
    const double vc = static_cast<double>(p.V) * p.C, terms = q.points / fs.padded();
    const double repacked = kLaunch + (fs.tiles() > 1 ? kReduce : 0.0) + q.points / 1.04e6 + terms / 1.78e5;
    const mach_tile_shape sh = default_shape(descs[i].n_frames);
    const double lanes =
        sh.mode == kBatchStaged
            ? vc * p.T / 5.9e5 + terms * 2 * sh.frame_lanes / 6.0e5
            : vc / 2.5e5 + vc * p.T / (sh.frame_lanes <= 2 ? 4.0e5 : sh.frame_lanes <= 4 ? 2.1e5 : sh.frame_lanes <= 8 ? 1.6e5 : 1.0e5) +
                  terms * 4 * sh.frame_lanes / 1.15e6;
    if (repacked < kMargin * lanes) continue;
    cheap[i] = 1;
    lanes_sum += lanes;
    repacked_sum += repacked;
  }
  if (repack_forced() || repacked_sum < kMargin * (kFloor + lanes_sum)) return;
  for (size_t i = 0; i < plans.size(); ++i)
    if (cheap[i]) repack[i] = 0;
}

// The launches over the repacked instances' frame tiles: instances grouped by exact-frame
// shape, each group's (frame tile, voxel tile) items longest first; the workspace for all of
// them, which runs share in stream order as they do the work counter.  OOM, UNSUPPORTED: the
// instances can still take their lane mappings.
mach_status plan_repacked(mach_batch_s* b, cudaStream_t s) {
  struct Item { int entry, ftile; int64_t tile; double cost; };
  struct Group { std::vector<Item> items; mach_batch_s::Multi* m = nullptr; };
  std::vector<Group> groups;
  for (const auto& q : b->repacked) {
    RepackNeeds needs;
    const int np = plan_repack(b->plans[q.inst], &needs);
    const RepackPart* parts = needs.parts;
    for (int k = 0; k < np; ++k) {
      // 2D and 3D shapes of 32 frames are one kernel
      const Variant v = parts[k].v == V_SX32_F8V1W7_T8X7E ? V_SX32_F8V1W7T14E : parts[k].v;
      Group* g = nullptr;
      for (auto& c : groups)
        if (c.m->v == v && c.m->args.n < kMultiMax) g = &c;
      if (!g) {
        b->multi.emplace_back(new mach_batch_s::Multi{});
        groups.emplace_back();
        g = &groups.back();
        g->m = b->multi.back().get();
        g->m->v = v;
      }
      const int entry = g->m->args.n++;
      g->m->args.inst[entry] = q.inst;
      DasParams& p = g->m->args.p[entry];
      p = parts[k].base;
      p.iq = b->ws + q.at + parts[k].at;
      p.pd_part = reinterpret_cast<float*>(b->ws + q.at + q.pd_at);
      const int64_t tiles = static_cast<int64_t>(p.tiles_x) * p.tiles_y * p.tiles_z;
      const double cost = static_cast<double>(p.C) * p.T * p.tile_x * p.tile_y * p.tile_z;
      for (int64_t t = tiles - 1; t >= 0; --t)
        for (int f = 0; f < parts[k].tiles; ++f) g->items.push_back({entry, f, t, cost});
    }
  }
  for (auto& g : groups) {
    if (g.items.size() > static_cast<size_t>(INT32_MAX)) return MACH_ERR_UNSUPPORTED;
    std::stable_sort(g.items.begin(), g.items.end(), [](const Item& a, const Item& c) { return a.cost > c.cost; });
    std::vector<int2> h(g.items.size());
    for (size_t k = 0; k < h.size(); ++k)
      h[k] = make_int2(g.items[k].entry | g.items[k].ftile << 16, static_cast<int>(g.items[k].tile));
    g.m->n_items = static_cast<int>(h.size());
    int64_t bytes = 0;
    if (const mach_status st = dev_alloc(reinterpret_cast<void**>(&g.m->d_items), sizeof(int2) * h.size(), &bytes);
        st != MACH_OK)
      return st;
    if (cudaMemcpyAsync(g.m->d_items, h.data(), sizeof(int2) * h.size(), cudaMemcpyHostToDevice, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
      return MACH_ERR_CUDA;
  }
  return MACH_OK;
}

}  // namespace

extern "C" {

// Everything of a batch into b, which the caller releases if this fails.
static mach_status plan_batch(const mach_das_desc* descs, int32_t n, const mach_tile_shape* shapes, cudaStream_t s,
                              mach_batch_s* b) {
  const int dt = descs[0].iq_dtype;
  b->n = n;
  b->iq_dtype = dt;
  b->plans.assign(n, nullptr);
  b->host_insts.resize(n);
  b->shapes.resize(n);
  size_t free_mem = 0, total_mem = 0, ws_total = 0;
  if (cudaMemGetInfo(&free_mem, &total_mem) != cudaSuccess) {
    cudaGetLastError();
    return MACH_ERR_CUDA;
  }
  struct Item { int inst; int64_t tile; double cost; };
  std::vector<Item> items;
  std::vector<char> is_repacked(n, 0);
  std::vector<size_t> slots(n, 0);         // ring slots that staged instances need
  b->bounds.assign(2 * static_cast<size_t>(n), nullptr);
  for (int i = 0; i < n; ++i)
    if (const mach_status st = make_batch_plan(&descs[i], !shapes, s, &b->plans[i]); st != MACH_OK) return st;
  // default shapes only: the instances worth repacking join the launches over repacked tiles
  if (!shapes) choose_repacked(b->plans, descs, is_repacked);
  for (int i = 0; i < n; ++i) {
    if (!is_repacked[i]) continue;
    RepackNeeds q;
    plan_repack(b->plans[i], &q);
    if (ws_total + q.ws_bytes > total_mem / 16) {
      is_repacked[i] = 0;
      continue;
    }
    const DasParams& p = *plan_params(b->plans[i]);
    b->repacked.push_back({i, dt, p.F, q.parts[0].base.frame_tiles, static_cast<int64_t>(p.T) * p.C, p.V, p.S,
                           {q.range[0], q.range[1]}, ws_total, q.pd_at});
    ws_total += (q.ws_bytes + 255) / 256 * 256;
  }
  for (int i = 0; i < n; ++i) {
    mach_tile_shape sh = shapes ? shapes[i] : default_shape(descs[i].n_frames);
    const DasParams base = *plan_params(b->plans[i]);
    DasParams p = base;
    const bool list = descs[i].vox_pos != nullptr;
    auto set_tiles = [&](mach_tile_shape& t) -> bool {
      int tile[3] = {t.tile[0], t.tile[1], t.tile[2]};
      if (tile[0] == 0) {
        if (t.mode == kBatchStaged) staged_tile(voxels_per_block(t), p.nx, p.ny, p.nz, list, tile);
        else pick_tile_shape(voxels_per_block(t), p.nx, p.ny, p.nz, list, tile);
      }
      if (tile[0] * tile[1] * tile[2] != voxels_per_block(t)) return false;
      t.tile[0] = tile[0];
      t.tile[1] = tile[1];
      t.tile[2] = tile[2];
      p.tile_x = tile[0];
      p.tile_y = tile[1];
      p.tile_z = tile[2];
      p.tiles_x = (p.nx + tile[0] - 1) / tile[0];
      p.tiles_y = (p.ny + tile[1] - 1) / tile[1];
      p.tiles_z = (p.nz + tile[2] - 1) / tile[2];
      return true;
    };
    if (!set_tiles(sh)) {
      if (sh.mode != kBatchStaged || shapes) return MACH_ERR_UNSUPPORTED;
      sh = frames_shape(descs[i].n_frames);
      if (!set_tiles(sh)) return MACH_ERR_UNSUPPORTED;
    }
    p.frame_tiles = 1;
    p.wb_x = p.wb_y = p.wb_z = 0;
    p.ystride = p.F;
    p.iq = nullptr;
    p.y = nullptr;
    p.pd = nullptr;
    if (sh.mode == kBatchStaged) {
      // per-tile bounds for the batch tiling, and the largest window; instances whose
      // windows exceed the ring slot take the frame-lane path instead
      const int64_t tiles = static_cast<int64_t>(p.tiles_x) * p.tiles_y * p.tiles_z;
      void *tb = nullptr, *tr = nullptr, *st = nullptr;
      int64_t bytes = 0;
      mach_status ms = dev_alloc(&tb, sizeof(float4) * 2 * tiles, &bytes);
      if (ms == MACH_OK) ms = dev_alloc(&tr, sizeof(float2) * p.T * tiles, &bytes);
      if (ms == MACH_OK) ms = dev_alloc(&st, sizeof(BoundStats), &bytes);
      if (ms != MACH_OK) {
        cudaFree(tb);
        cudaFree(tr);
        cudaFree(st);
        return ms;
      }
      b->bounds[2 * i] = tb;
      b->bounds[2 * i + 1] = tr;
      p.tbox = static_cast<float4*>(tb);
      p.txr = static_cast<float2*>(tr);
      p.txr_stride = p.T;
      BoundStats stats{};
      if (launch_tile_bounds(p, static_cast<float4*>(tb), static_cast<float2*>(tr), static_cast<BoundStats*>(st), s) != cudaSuccess ||
          cudaMemcpyAsync(&stats, st, sizeof(stats), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
          cudaStreamSynchronize(s) != cudaSuccess) {
        cudaFree(st);
        return MACH_ERR_CUDA;
      }
      cudaFree(st);
      p.rows_cap = std::max(2, stats.rows);
      const size_t sample = (dt == MACH_IQ_F16X2 || dt == MACH_IQ_BF16X2) ? 4 : 8;
      const size_t need = (static_cast<size_t>(p.rows_cap) * p.F * sample + 32 + 127) / 128 * 128;
      if (need <= kBatchSlotCap) {
        slots[i] = need;
      } else if (shapes) {
        return MACH_ERR_UNSUPPORTED;
      } else {
        sh = frames_shape(descs[i].n_frames);
        sh.tile[0] = sh.tile[1] = sh.tile[2] = 0;
        if (!set_tiles(sh)) return MACH_ERR_UNSUPPORTED;
      }
    }
    b->host_insts[i].p = p;
    b->host_insts[i].mode = sh.mode;
    b->host_insts[i].frame_lanes = sh.frame_lanes;
    b->shapes[i] = sh;
    const int64_t tiles = static_cast<int64_t>(p.tiles_x) * p.tiles_y * p.tiles_z;
    // estimated cost of one tile: voxels x elements x transmits x frame slots it occupies
    const double frames_slots = sh.mode == kBatchChannels ? 4.0 : (sh.mode == kBatchStaged ? 2.0 * sh.frame_lanes
                                                                                          : 4.0 * sh.frame_lanes);
    const double cost = static_cast<double>(voxels_per_block(sh)) * p.C * p.T * frames_slots;
    // an instance's deepest tiles (widest apertures) first, its shallow ones last
    for (int64_t t = tiles - 1; t >= 0; --t) items.push_back({i, t, cost});
    b->points += static_cast<int64_t>(p.V) * p.C * p.T * p.F;
  }
  int64_t bytes = 0;
  if (!b->repacked.empty()) {
    mach_status st = dev_alloc(reinterpret_cast<void**>(&b->ws), ws_total, &bytes);
    if (st == MACH_OK) st = plan_repacked(b, s);
    if (st == MACH_ERR_CUDA) return st;
    if (st == MACH_OK) {
      items.erase(std::remove_if(items.begin(), items.end(), [&](const Item& t) { return is_repacked[t.inst]; }),
                  items.end());
      for (int i = 0; i < n; ++i) {   // what the lane mappings of repacked instances would have needed
        if (!is_repacked[i]) continue;
        slots[i] = 0;
        b->host_insts[i].p.tbox = nullptr;
        b->host_insts[i].p.txr = nullptr;
        for (int k = 0; k < 2; ++k) {
          cudaFree(b->bounds[2 * i + k]);
          b->bounds[2 * i + k] = nullptr;
        }
      }
    } else {   // no memory for the workspace or its lists: every instance on its lane mapping
      drop_repacked(b);
    }
  }
  for (const size_t q : slots) b->slot_bytes = std::max(b->slot_bytes, q);
  if (items.size() > static_cast<size_t>(INT32_MAX)) return MACH_ERR_UNSUPPORTED;
  std::stable_sort(items.begin(), items.end(), [](const Item& a, const Item& c) { return a.cost > c.cost; });
  std::vector<int2> hitems(items.size());
  for (size_t k = 0; k < items.size(); ++k) hitems[k] = make_int2(items[k].inst, static_cast<int>(items[k].tile));
  b->n_items = static_cast<int>(items.size());
  mach_status ms = dev_alloc(reinterpret_cast<void**>(&b->d_insts), sizeof(BatchInstance) * n, &bytes);
  if (ms == MACH_OK) ms = dev_alloc(reinterpret_cast<void**>(&b->d_items), sizeof(int2) * hitems.size(), &bytes);
  if (ms == MACH_OK) ms = dev_alloc(reinterpret_cast<void**>(&b->d_counter), 2 * sizeof(int), &bytes);
  if (ms != MACH_OK) return ms;
  for (auto& m : b->multi) m->args.insts = b->d_insts;
  if ((!hitems.empty() && cudaMemcpyAsync(b->d_items, hitems.data(), sizeof(int2) * hitems.size(),
                                          cudaMemcpyHostToDevice, s) != cudaSuccess) ||
      cudaMemsetAsync(b->d_counter, 0, 2 * sizeof(int), s) != cudaSuccess ||
      cudaMemcpyAsync(b->d_insts, b->host_insts.data(), sizeof(BatchInstance) * n, cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return MACH_ERR_CUDA;
  int dev = 0, sms = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  b->per_sm = batch_blocks_per_sm(dt, b->slot_bytes);
  b->grid = std::max(1, std::min(b->n_items, sms * b->per_sm));
  return MACH_OK;
}

mach_status mach_batch_plan(const mach_das_desc* descs, int32_t n, const mach_tile_shape* shapes, void* stream,
                            mach_batch* out) {
  if (!out) return MACH_ERR_INVALID_ARG;
  *out = nullptr;
  if (!descs || n < 1) return MACH_ERR_INVALID_ARG;
  const int dt = descs[0].iq_dtype;
  for (int i = 0; i < n; ++i) {
    mach_status st = host_validate(&descs[i]);
    if (st != MACH_OK) return st;
    if (descs[i].term_table) return MACH_ERR_UNSUPPORTED;
    if (descs[i].iq_dtype != dt) return MACH_ERR_INVALID_ARG;
    if (descs[i].n_frames > 64) return MACH_ERR_UNSUPPORTED;
    if (shapes) {
      const mach_tile_shape& s = shapes[i];
      if (s.mode == kBatchChannels) {
        if (descs[i].n_frames > 4) return MACH_ERR_INVALID_ARG;
      } else if (s.mode == kBatchStaged) {
        if (s.frame_lanes != 8 && s.frame_lanes != 16) return MACH_ERR_INVALID_ARG;
        if (4 * s.frame_lanes < descs[i].n_frames) return MACH_ERR_INVALID_ARG;
      } else if (s.mode == kBatchFrames) {
        if (s.frame_lanes != 2 && s.frame_lanes != 4 && s.frame_lanes != 8 && s.frame_lanes != 16)
          return MACH_ERR_INVALID_ARG;
        if (4 * s.frame_lanes < descs[i].n_frames) return MACH_ERR_INVALID_ARG;
      } else {
        return MACH_ERR_INVALID_ARG;
      }
      const bool zero = s.tile[0] == 0 && s.tile[1] == 0 && s.tile[2] == 0;
      if (!zero && (s.tile[0] < 1 || s.tile[1] < 1 || s.tile[2] < 1 ||
                    s.tile[0] * s.tile[1] * s.tile[2] != voxels_per_block(s)))
        return MACH_ERR_INVALID_ARG;
    }
  }
  if (dt == MACH_IQ_C64_SPLIT) return MACH_ERR_UNSUPPORTED;
  mach_batch_s* b = new (std::nothrow) mach_batch_s();
  if (!b) return MACH_ERR_OOM;
  mach_status st;
  try {
    st = plan_batch(descs, n, shapes, static_cast<cudaStream_t>(stream), b);
  } catch (const std::bad_alloc&) {   // the host lists grow with the tiles of every instance
    st = MACH_ERR_OOM;
  } catch (const std::length_error&) {
    st = MACH_ERR_OOM;
  }
  if (st != MACH_OK) {
    release(b);
    return st;
  }
  *out = b;
  return MACH_OK;
}

mach_status mach_batch_bind(mach_batch b, const void* const* iq_devs, void* const* y_devs, float* const* pd_devs,
                            void* stream) {
  if (!b || !iq_devs) return MACH_ERR_INVALID_ARG;
  for (int i = 0; i < b->n; ++i) {
    void* y = y_devs ? y_devs[i] : nullptr;
    float* pd = pd_devs ? pd_devs[i] : nullptr;
    if (!iq_devs[i] || (!y && !pd)) return MACH_ERR_INVALID_ARG;
    if ((reinterpret_cast<uintptr_t>(iq_devs[i]) & 15u) || (reinterpret_cast<uintptr_t>(y) & 15u) ||
        (reinterpret_cast<uintptr_t>(pd) & 3u))
      return MACH_ERR_INVALID_ARG;
  }
  for (int i = 0; i < b->n; ++i) {
    b->host_insts[i].p.iq = iq_devs[i];
    b->host_insts[i].p.y = static_cast<float2*>(y_devs ? y_devs[i] : nullptr);
    b->host_insts[i].p.pd = pd_devs ? pd_devs[i] : nullptr;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  if (cudaMemcpyAsync(b->d_insts, b->host_insts.data(), sizeof(BatchInstance) * b->n, cudaMemcpyHostToDevice, s) !=
          cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return MACH_ERR_CUDA;
  b->bound = true;
  return MACH_OK;
}

mach_status mach_batch_run(mach_batch b, void* stream) {
  if (!b || !b->bound) return MACH_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  // the repacked tiles first: their launches hold the longest blocks
  for (const auto& q : b->repacked) {
    if (e != cudaSuccess) break;
    e = launch_iq_repack(nullptr, &b->d_insts[q.inst].p.iq, q.dtype, reinterpret_cast<float*>(b->ws + q.at), q.TC, q.S,
                         q.range[0], q.range[1], q.F, s);
  }
  for (const auto& m : b->multi) {
    if (e != cudaSuccess) break;
    e = launch_das_multi(m->args, m->v, m->d_items, m->n_items, s);
  }
  for (const auto& q : b->repacked) {
    if (e != cudaSuccess) break;
    if (q.tiles > 1)
      e = launch_pd_reduce(reinterpret_cast<const float*>(b->ws + q.at + q.pd_at), nullptr, &b->d_insts[q.inst].p.pd, q.V,
                           q.tiles, s);
  }
  if (e == cudaSuccess && b->n_items)
    e = launch_batch(b->iq_dtype, b->d_insts, b->d_items, b->n_items, b->d_counter, b->grid, b->slot_bytes, s);
  return e == cudaSuccess ? MACH_OK : MACH_ERR_CUDA;
}

mach_status mach_batch_get_info(mach_batch b, mach_batch_info* info, mach_tile_shape* shapes_or_null) {
  if (!b || !info) return MACH_ERR_INVALID_ARG;
  info->instances = b->n;
  info->items = b->n_items;
  for (const auto& m : b->multi) info->items += m->n_items;
  info->blocks = b->grid;
  info->blocks_per_sm = b->per_sm;
  info->points = b->points;
  if (shapes_or_null) std::memcpy(shapes_or_null, b->shapes.data(), sizeof(mach_tile_shape) * b->n);
  return MACH_OK;
}

mach_status mach_batch_destroy(mach_batch b) {
  release(b);
  return MACH_OK;
}

}  // extern "C"
