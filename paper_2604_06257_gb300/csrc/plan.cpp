// plan.cpp -- the C ABI: argument validation, plan construction (Sec. 4.3 precompute),
// kernel-variant selection and the run entry points.
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstdio>
#include <cstring>
#include <map>
#include <mutex>
#include <new>
#include <set>
#include <vector>

#include "mach.h"
#include "mach_internal.h"

using namespace mach;

struct mach_plan_s {
  mach_das_desc d{};          // copy; pointer fields cleared
  int device = 0;
  Variant variant = V_COUNT;
  DasParams base{};           // everything but iq / y / pd
  float4* d_vox = nullptr;
  float4* d_elem = nullptr;
  float* d_tx = nullptr;
  float* d_pd_part = nullptr;
  float4* d_tbox = nullptr;     // staged variants: per-tile bounding boxes
  float2* d_txr = nullptr;      // staged variants: per-tile transmit-delay ranges
  int* d_err = nullptr;         // device error word
  int rows_cap = 0;
  int64_t copy_pairs = 0;
  int64_t device_bytes = 0;
  bool table = false;           // terms read from the plan-time term table
  int64_t* d_tile_pairs = nullptr;
  int4* d_pair_desc = nullptr;
  float4* d_term_rec = nullptr;
  int64_t table_bytes = 0;
  // repacked route (see repack_plan): the exact-frame launches over repacked frame tiles, and
  // the device's pool that each run takes its workspace from
  RepackPart parts[2];
  int n_parts = 0;
  size_t ws_bytes = 0;          // workspace of one run: repacked IQ, partial Power Doppler sums
  size_t pd_at = 0;
  int range[2] = {0, 0};        // samples that the parts' windows touch
  double points = 0.0;          // what the parts beamform: voxels x windows x padded frames
  cudaMemPool_t pool = nullptr;
};

namespace {

// The pools that repacked runs take their workspaces from, one per device for all plans: stream
// order keeps concurrent runs' blocks apart, and what lies idle between runs is one
// workspace, of the largest plan there is, however many plans there are.  The last plan of a
// device gives its pool back.
struct DevicePool {
  cudaMemPool_t pool = nullptr;
  std::multiset<size_t> plans;   // workspace bytes of each plan
};
std::mutex g_pools_lock;
std::map<int, DevicePool>& pools() {
  static auto* p = new std::map<int, DevicePool>;   // never destroyed: plans may outlive statics
  return *p;
}

void keep_largest(DevicePool& d) {
  uint64_t keep = (*d.plans.rbegin() >> 25 << 25) + (64u << 20);   // the pool maps memory in blocks
  if (cudaMemPoolSetAttribute(d.pool, cudaMemPoolAttrReleaseThreshold, &keep) != cudaSuccess) cudaGetLastError();
}

cudaMemPool_t take_pool(int device, size_t bytes) {
  std::lock_guard<std::mutex> hold(g_pools_lock);
  DevicePool& d = pools()[device];
  if (!d.pool) {
    cudaMemPoolProps props{};
    props.allocType = cudaMemAllocationTypePinned;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = device;
    if (cudaMemPoolCreate(&d.pool, &props) != cudaSuccess) {
      cudaGetLastError();
      d.pool = nullptr;
      return nullptr;
    }
  }
  d.plans.insert(bytes);
  keep_largest(d);
  return d.pool;
}

void return_pool(int device, size_t bytes) {
  std::lock_guard<std::mutex> hold(g_pools_lock);
  DevicePool& d = pools()[device];
  d.plans.erase(d.plans.find(bytes));
  if (d.plans.empty()) {
    cudaMemPoolDestroy(d.pool);
    d.pool = nullptr;
    return;
  }
  keep_largest(d);
  if (*d.plans.rbegin() < bytes && cudaMemPoolTrimTo(d.pool, *d.plans.rbegin()) != cudaSuccess) cudaGetLastError();
}

std::atomic<int> g_fail_alloc_countdown{0};   // test hook: > 0 -> the n-th allocation fails
int g_force_variant = -1;         // test hook: variant index, or -1 for automatic choice
bool g_force_repack = false;      // test hook: repack whenever the kernels can
uint32_t g_wait_limit = 0;        // test hook: polls per bounded wait (0 = default)
int g_stall = 0;                  // test hook: staged producer never issues its copies

float float_of(int bits) {
  float f;
  std::memcpy(&f, &bits, sizeof(f));
  return f;
}

bool finite3(const float* p, int64_t n) {
  for (int64_t i = 0; i < 3 * n; ++i)
    if (!std::isfinite(p[i])) return false;
  return true;
}

mach_status validate(const mach_das_desc* d) {
  if (!d) return MACH_ERR_INVALID_ARG;
  if (d->ndim != 2 && d->ndim != 3) return MACH_ERR_INVALID_ARG;
  if (d->n_elem < 1 || !d->elem_pos) return MACH_ERR_INVALID_ARG;
  if (d->n_tx < 1 || (!d->tx_angles && !d->tx_table_dev)) return MACH_ERR_INVALID_ARG;
  if (!(d->fs > 0.0) || !std::isfinite(d->fs) || !(d->c > 0.0) || !std::isfinite(d->c))
    return MACH_ERR_INVALID_ARG;
  if (!(d->fc >= 0.0) || !std::isfinite(d->fc) || !std::isfinite(d->t0)) return MACH_ERR_INVALID_ARG;
  if (!(d->f_number >= 0.0) || !std::isfinite(d->f_number)) return MACH_ERR_INVALID_ARG;
  if (d->apod < MACH_APOD_NONE || d->apod > MACH_APOD_GAUSS) return MACH_ERR_INVALID_ARG;
  if (d->iq_dtype < MACH_IQ_C64 || d->iq_dtype > MACH_IQ_C64_SPLIT) return MACH_ERR_INVALID_ARG;
  if (d->term_table != 0 && d->term_table != 1) return MACH_ERR_INVALID_ARG;
  if (d->iq_dtype == MACH_IQ_C64_SPLIT && (d->n_frames % 4 != 0 || d->n_frames <= 4)) return MACH_ERR_UNSUPPORTED;
  if (d->n_samples < 2 || d->n_samples > (1 << 24)) return MACH_ERR_INVALID_ARG;
  if (d->n_frames < 1) return MACH_ERR_INVALID_ARG;
  // per-(t, c) slab offsets are computed in 64 bits, but one slab must stay indexable
  if (static_cast<int64_t>(d->n_samples) * d->n_frames > (int64_t{1} << 31) - 1) return MACH_ERR_UNSUPPORTED;
  if (!finite3(d->elem_pos, d->n_elem)) return MACH_ERR_INVALID_ARG;
  int64_t V;
  if (d->vox_pos) {
    if (d->n_vox < 1) return MACH_ERR_INVALID_ARG;
    V = d->n_vox;
    if (!finite3(d->vox_pos, V)) return MACH_ERR_INVALID_ARG;
  } else {
    for (int k = 0; k < 3; ++k) {
      if (d->grid_dims[k] < 1) return MACH_ERR_INVALID_ARG;
      if (!std::isfinite(d->grid_origin[k]) || !std::isfinite(d->grid_step[k])) return MACH_ERR_INVALID_ARG;
    }
    V = static_cast<int64_t>(d->grid_dims[0]) * d->grid_dims[1] * d->grid_dims[2];
    if (d->n_vox != 0 && d->n_vox != V) return MACH_ERR_INVALID_ARG;
  }
  if (V > (int64_t{1} << 40)) return MACH_ERR_UNSUPPORTED;
  if (d->tx_angles)
    for (int t = 0; t < 2 * d->n_tx; ++t)
      if (!std::isfinite(d->tx_angles[t])) return MACH_ERR_INVALID_ARG;
  if (d->ndim == 2) {   // a 2D acquisition lives in the plane y = 0
    for (int c = 0; c < d->n_elem; ++c)
      if (d->elem_pos[3 * c + 1] != 0.0f) return MACH_ERR_INVALID_ARG;
    if (d->tx_angles && !d->tx_table_dev)
      for (int t = 0; t < d->n_tx; ++t)
        if (d->tx_angles[2 * t + 1] != 0.0) return MACH_ERR_INVALID_ARG;
    if (d->vox_pos) {
      for (int64_t v = 0; v < V; ++v)
        if (d->vox_pos[3 * v + 1] != 0.0f) return MACH_ERR_INVALID_ARG;
    } else if (d->grid_dims[1] != 1 || d->grid_origin[1] != 0.0) {
      return MACH_ERR_INVALID_ARG;
    }
  }
  return MACH_OK;
}

Variant pick_variant(int iq_dtype, int F) {
  // staged 4-voxel-group kernels for 16 < F <= 64 (fastest measured shapes); L1-path
  // kernels for short, long (frame-tiled) or odd ensembles
  if (iq_dtype == MACH_IQ_C64) {
    if (F <= 4) return V_CH_C64;
    if (F % 2 == 0) {
      if (F <= 16) return V_F16_C64;
      if (F <= 32) return V_ST32_C64_V4W7;
      if (F <= 64) return V_ST64_C64_V4;
      return V_F64_C64;
    }
    return V_S32_C64;
  }
  if (iq_dtype == MACH_IQ_C64_SPLIT) {   // F % 4 == 0 and F > 4 (checked by validate)
    if (F == 8) return V_SX8_F4V1W7;
    if (F == 16) return V_SX16_F4V2W7;
    if (F == 32) return V_SX32_F8V1W7T14E;
    if (F == 64) return V_SX64_C64P;
    if (F <= 16) return V_F32_C64P;
    if (F <= 32) return V_ST32_C64P_V4W7;
    if (F <= 64) return V_ST64_C64P_V4;
    return V_F64_C64P;
  }
  if (iq_dtype == MACH_IQ_BF16X2) {
    if (F <= 4) return V_CH_B16;
    if (F % 4 == 0) {
      if (F <= 16) return V_F32_B16;
      if (F <= 32) return V_ST32_B16_V4;
      if (F <= 64) return V_ST64_B16_V4;
      return V_F64_B16;
    }
    return V_S32_B16;
  }
  if (F <= 4) return V_CH_H16;
  if (F % 4 == 0) {
    if (F <= 16) return V_F32_H16;
    if (F <= 32) return V_ST32_H16_V4;
    if (F <= 64) return V_ST64_H16_V4;
    return V_F64_H16;
  }
  return V_S32_H16;
}

// The non-staged variant with the same frame tile (used when the ring would not fit).
Variant unstaged(Variant v) {
  switch (v) {
    case V_ST32_C64: case V_ST32_C64_V4: case V_ST32_C64_V4W4: case V_ST32_C64_V4R56: case V_ST32_C64_V4W7:
      return V_F32_C64;
    case V_ST64_C64: case V_ST64_C64_V4: return V_F64_C64;
    case V_ST32_H16: case V_ST32_H16_V4: return V_F32_H16;
    case V_ST64_H16: case V_ST64_H16_V4: return V_F64_H16;
    case V_ST32_B16: case V_ST32_B16_V4: return V_F32_B16;
    case V_ST32_C64P_V4: case V_ST32_C64P_V4W7: case V_SX32_C64P: case V_SX32_F4V2W7: case V_SX32_F8V1W7:
    case V_SX32_F4V2W15: case V_SX32_F8V1W15: case V_SX32_F8V1W15T24: case V_SX32_F8V1W15T40:
    case V_SX32_F8V1W15T24S: case V_SX32_F8V1W7T14: case V_SX32_F8V1W7T14E: case V_SX32_F4V2W7T14:
    case V_SX32_F8V1W15T30R12: case V_SX32_F8V1W15T30R12E: case V_SX32_C64P_T8X14: case V_SX32_F8V1W7_T8X7E:
      return V_F32_C64P;
    case V_ST64_C64P_V4: case V_SX64_C64P: case V_SX64_F8V2: case V_SX64_C64PS: case V_SX64_C64PE:
    case V_SX64_C64P_T16: case V_SX64_C64P_T16E: case V_SX64_C64P_T8X8:
      return V_F64_C64P;
    case V_SX16_F4V2W7: case V_SX16_F4V1W7: case V_SX8_F4V1W7: case V_SX16_F4V2W7_T8X14: case V_SX8_F4V1W7_T8X14:
    case V_SX16_F8V1W7: case V_SX16_F8V1W4: case V_SX8_F8V1W4:
      return V_F32_C64P;
    case V_ST64_B16_V4: return V_F64_B16;
    default: return v;
  }
}

bool variant_accepts(Variant v, int iq_dtype, int F) {
  const VariantShape& s = variant_shape(v);
  if (s.iq_type != iq_dtype) return false;
  if (s.channel_lanes) return F <= s.frame_tile;
  const int vec = s.frames_per_lane == 1 ? 1 : (s.iq_type == MACH_IQ_C64 ? 2 : 4);
  if (F % vec != 0) return false;
  if (s.staged && F > s.frame_tile) return false;
  if (s.exact_frames && F != s.frame_tile) return false;
  return true;
}

// The variant to try when a staged variant's ring does not fit in shared memory: one with
// fewer ring slots (the variant itself when there is none).
Variant staged_fallback(Variant v) {
  switch (v) {
    case V_ST64_C64_V4: return V_ST64_C64;
    case V_ST64_H16_V4: return V_ST64_H16;
    case V_SX32_F8V1W15: case V_SX32_F4V2W15: case V_SX32_F8V1W7: case V_SX32_F4V2W7: case V_SX32_F8V1W15T24:
    case V_SX32_F8V1W15T40: case V_SX32_F8V1W15T24S: case V_SX32_F8V1W7T14: case V_SX32_F8V1W7T14E:
    case V_SX32_F4V2W7T14: case V_SX32_F8V1W15T30R12: case V_SX32_F8V1W15T30R12E: case V_SX32_F8V1W7_T8X7E:
      return V_SX32_C64P;
    default: return v;
  }
}

// The generic staged variant an exact-frame variant specialises (term tables are built
// for the generic kernels' record layout).
Variant generic_staged(Variant v) {
  switch (v) {
    case V_SX32_C64P: case V_SX32_F4V2W7: case V_SX32_F8V1W7: case V_SX32_F4V2W15: case V_SX32_F8V1W15:
    case V_SX32_F8V1W15T24: case V_SX32_F8V1W15T40: case V_SX32_F8V1W15T24S: case V_SX32_F8V1W7T14:
    case V_SX32_F8V1W7T14E: case V_SX32_F4V2W7T14: case V_SX32_F8V1W15T30R12: case V_SX32_F8V1W15T30R12E:
    case V_SX32_C64P_T8X14: case V_SX32_F8V1W7_T8X7E:
      return V_ST32_C64P_V4W7;
    case V_SX64_C64P: case V_SX64_F8V2: case V_SX64_C64PS: case V_SX64_C64PE: case V_SX64_C64P_T16:
    case V_SX64_C64P_T16E: case V_SX64_C64P_T8X8:
      return V_ST64_C64P_V4;
    case V_SX16_F4V2W7: case V_SX16_F4V1W7: case V_SX8_F4V1W7: case V_SX16_F4V2W7_T8X14: case V_SX8_F4V1W7_T8X14:
    case V_SX16_F8V1W7:
      return V_F32_C64P;
    default: return v;
  }
}

// Voxel tile of one block: compact boxes so that the voxels sharing a block (and the
// L1 cache) read overlapping sample windows of each element.
void pick_tile(int n, int nx, int ny, int nz, bool list, int tile[3]) {
  // the box always holds exactly n voxel slots
  if (list || (ny == 1 && nz == 1)) {
    tile[0] = n; tile[1] = 1; tile[2] = 1;
    return;
  }
  if (ny == 1) {   // 2D x-z grid: the squarest power-of-two width that divides n
    int tx = 1;
    while (tx * tx < n) tx *= 2;
    while (n % tx) tx /= 2;
    tile[0] = tx; tile[1] = 1; tile[2] = n / tx;
    return;
  }
  // 3D: up to 8 along x and 4 along y (powers of two dividing n), the rest along z
  int tx = 8;
  while (n % tx) tx /= 2;
  int ty = 4;
  while ((n / tx) % ty) ty /= 2;
  tile[0] = tx; tile[1] = ty; tile[2] = n / (tx * ty);
}

uint32_t fixed_cycles(double cycles) {   // round(2^32 frac(cycles))
  double f = cycles - std::floor(cycles);
  double r = std::nearbyint(f * 4294967296.0);
  if (r >= 4294967296.0) r -= 4294967296.0;
  return static_cast<uint32_t>(r);
}

void release(mach_plan_s* p) {
  if (!p) return;
  cudaFree(p->d_vox);
  cudaFree(p->d_elem);
  cudaFree(p->d_tx);
  cudaFree(p->d_pd_part);
  cudaFree(p->d_tbox);
  cudaFree(p->d_txr);
  cudaFree(p->d_err);
  cudaFree(p->d_tile_pairs);
  cudaFree(p->d_pair_desc);
  cudaFree(p->d_term_rec);
  for (auto& q : p->parts) {
    cudaFree(q.d_tbox);
    cudaFree(q.d_txr);
  }
  if (p->pool) return_pool(p->device, p->ws_bytes);
  delete p;
}

}  // namespace

extern "C" {

const char* mach_status_string(mach_status s) {
  switch (s) {
    case MACH_OK: return "ok";
    case MACH_ERR_INVALID_ARG: return "invalid argument";
    case MACH_ERR_CUDA: return "CUDA error";
    case MACH_ERR_OOM: return "out of device memory";
    case MACH_ERR_UNSUPPORTED: return "unsupported configuration";
    case MACH_ERR_TIMEOUT: return "device wait timed out";
  }
  return "unknown status";
}

const char* mach_version(void) { return "mach-gb300 0.1.0 sm_103a"; }

void mach_debug_fail_alloc_after(int32_t n) { g_fail_alloc_countdown = n > 0 ? n : 0; }

int32_t mach_debug_allocs_to_failure(void) { return g_fail_alloc_countdown.load(); }

// Tile geometry of a variant: voxel box per block and the number of blocks.
static mach_status configure_tiles(DasParams& b, Variant var, bool list, int64_t V, int F) {
  const VariantShape& shp = variant_shape(var);
  const int per_cta = shp.voxels_per_warp * shp.warps;
  int tile[3];
  pick_tile(per_cta, b.nx, b.ny, b.nz, list, tile);
  if (shp.tile2d_x && !list && b.ny == 1 && b.nz > 1 && per_cta % shp.tile2d_x == 0) {
    tile[0] = shp.tile2d_x;
    tile[1] = 1;
    tile[2] = per_cta / shp.tile2d_x;
  }
  if (shp.tile3d_x && !list && b.ny > 1 && per_cta % (shp.tile3d_x * shp.tile3d_y) == 0) {
    tile[0] = shp.tile3d_x;
    tile[1] = shp.tile3d_y;
    tile[2] = per_cta / (shp.tile3d_x * shp.tile3d_y);
  }
  if (tile[0] * tile[1] * tile[2] != per_cta) return MACH_ERR_UNSUPPORTED;   // slots must map 1:1
  b.tile_x = tile[0];
  b.tile_y = tile[1];
  b.tile_z = tile[2];
  b.tiles_x = (b.nx + tile[0] - 1) / tile[0];
  b.tiles_y = (b.ny + tile[1] - 1) / tile[1];
  b.tiles_z = (b.nz + tile[2] - 1) / tile[2];
  b.frame_tiles = (F + shp.frame_tile - 1) / shp.frame_tile;
  (void)V;
  // staged kernels: each warp owns a compact block of the tile, so that its voxels tend to
  // agree on which (element, transmit) pairs they use (the warp skips pairs none of them use)
  b.wb_x = b.wb_y = b.wb_z = 0;
  if (shp.staged && !list && !(b.ny == 1 && b.nz == 1)) {
    // candidate blocks, most compact first; the first one that divides the tile is used
    static const int c2d32[][3] = {{8, 1, 4}, {16, 1, 2}, {4, 1, 8}};
    static const int c2d16[][3] = {{4, 1, 4}, {8, 1, 2}, {16, 1, 1}};
    static const int c2d8[][3] = {{4, 1, 2}, {8, 1, 1}, {2, 1, 4}};
    static const int c3d32[][3] = {{4, 4, 2}, {8, 4, 1}};
    static const int c3d16[][3] = {{4, 4, 1}, {8, 2, 1}};
    static const int c3d8[][3] = {{4, 2, 1}, {8, 1, 1}};
    const int wv = shp.voxels_per_warp;
    const int(*cand)[3] = nullptr;
    int nc = 0;
    if (b.ny == 1) {
      if (wv == 32) { cand = c2d32; nc = 3; } else if (wv == 16) { cand = c2d16; nc = 3; } else if (wv == 8) { cand = c2d8; nc = 3; }
    } else {
      if (wv == 32) { cand = c3d32; nc = 2; } else if (wv == 16) { cand = c3d16; nc = 2; } else if (wv == 8) { cand = c3d8; nc = 2; }
    }
    for (int k = 0; k < nc; ++k) {
      if (tile[0] % cand[k][0] == 0 && tile[1] % cand[k][1] == 0 && tile[2] % cand[k][2] == 0) {
        b.wb_x = cand[k][0];
        b.wb_y = cand[k][1];
        b.wb_z = cand[k][2];
        break;
      }
    }
  }
  if (b.frame_tiles > 65535) return MACH_ERR_UNSUPPORTED;   // grid y limit
  if (static_cast<int64_t>(b.tiles_x) * b.tiles_y * b.tiles_z > INT32_MAX) return MACH_ERR_UNSUPPORTED;
  return MACH_OK;
}

// Plan-time term table (table mode): every usable (tile, element, transmit) pair's
// window and the records of all voxel slots of the block, in the order a run consumes
// them.  The windows come first; their counts, scanned on the host, give each pair its
// index, and one block per (tile, element) then writes the records.
static mach_status build_term_table(mach_plan_s* p, DasParams& b, cudaStream_t s) {
  const int64_t tiles = static_cast<int64_t>(b.tiles_x) * b.tiles_y * b.tiles_z;
  const int64_t n = tiles * b.C;
  if (n > INT32_MAX) return MACH_ERR_UNSUPPORTED;   // one record block per (tile, element)
  const VariantShape& sh = variant_shape(p->variant);
  const int64_t nrec = static_cast<int64_t>(sh.warps) * sh.voxels_per_warp;
  int2* d_win = nullptr;
  int* d_count = nullptr;
  int64_t* d_first = nullptr;
  int64_t scratch = 0;
  auto done = [&](mach_status e) {
    cudaFree(d_win);
    cudaFree(d_count);
    cudaFree(d_first);
    return e;
  };
  mach_status st;
  if ((st = dev_alloc(reinterpret_cast<void**>(&d_win), sizeof(int2) * n * b.T, &scratch)) != MACH_OK) return done(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&d_count), sizeof(int) * n, &scratch)) != MACH_OK) return done(st);
  if (launch_pair_windows(b, d_win, d_count, s) != cudaSuccess) return done(MACH_ERR_CUDA);
  std::vector<int> count(static_cast<size_t>(n));
  if (cudaMemcpyAsync(count.data(), d_count, sizeof(int) * n, cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return done(MACH_ERR_CUDA);
  std::vector<int64_t> first(static_cast<size_t>(n) + 1, 0);
  for (int64_t i = 0; i < n; ++i) first[i + 1] = first[i] + count[i];
  const int64_t pairs = first[n];
  std::vector<int64_t> tile_first(static_cast<size_t>(tiles) + 1);
  for (int64_t t = 0; t < tiles; ++t) tile_first[t] = first[t * b.C];
  tile_first[tiles] = pairs;
  const size_t bytes = sizeof(int64_t) * (tiles + 1) + sizeof(int4) * pairs + sizeof(float4) * pairs * nrec;
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    return done(MACH_ERR_CUDA);
  }
  if (bytes + sizeof(int64_t) * (n + 1) > free_b) return done(MACH_ERR_OOM);
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_tile_pairs), sizeof(int64_t) * (tiles + 1), &p->device_bytes)) != MACH_OK)
    return done(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_pair_desc), sizeof(int4) * pairs, &p->device_bytes)) != MACH_OK)
    return done(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_term_rec), sizeof(float4) * pairs * nrec, &p->device_bytes)) != MACH_OK)
    return done(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&d_first), sizeof(int64_t) * (n + 1), &scratch)) != MACH_OK)
    return done(st);
  if (cudaMemcpyAsync(d_first, first.data(), sizeof(int64_t) * (n + 1), cudaMemcpyHostToDevice, s) != cudaSuccess ||
      cudaMemcpyAsync(p->d_tile_pairs, tile_first.data(), sizeof(int64_t) * (tiles + 1), cudaMemcpyHostToDevice, s) !=
          cudaSuccess)
    return done(MACH_ERR_CUDA);
  if (launch_term_records(b, p->variant, d_win, d_first, p->d_pair_desc, p->d_term_rec, s) != cudaSuccess)
    return done(MACH_ERR_CUDA);
  if (cudaStreamSynchronize(s) != cudaSuccess) return done(MACH_ERR_CUDA);
  b.tile_pairs = p->d_tile_pairs;
  b.pair_desc = p->d_pair_desc;
  b.term_rec = p->d_term_rec;
  p->table_bytes = static_cast<int64_t>(bytes);
  p->table = true;
  return done(MACH_OK);
}

// Repacked route: ensembles that no exact-frame kernel reads directly are rewritten into
// split complex64 rows of whole frame tiles on every run (k_iq_repack) and beamformed by the
// exact-frame kernels.
// What it buys (251 x 251 px, 128 elements, 2048 samples, V / S = 31, cold L2; direct kernel
// -> repacking and exact-frame kernels, us): complex64 5 frames 304 -> 71, 8: 214 -> 71,
// 16: 214 -> 86, 25: 314 -> 122, 32: 154 -> 116, 40: 273 -> 192, 64: 378 -> 234,
// 200: 1193 -> 731; float16 25: 322 -> 124, 32: 162 -> 125, 64: 257 -> 235.  (All but
// complex64 at 32 frames with every sample rewritten; only those that windows touch are now,
// which took 25 frames from 123 to 111 between other work.)  The odd counts gain most: the
// direct kernels read them one frame at a time.
// The repacking costs a few launches and one pass over the IQ, the gain grows with the voxels
// that read each sample: hence the bounds on V / S, and repack_pays.  A workspace above a
// sixteenth of the device's memory, a capturing stream, or a failed workspace allocation takes
// the direct kernel.

// Whether repacking pays over the direct kernel, from what the repacked launches would do: points
// (voxels x windows x padded frames) and their share of the whole grid's, and the direct
// kernel's tiles.  Measured as the direct kernel's time over the repacked run's, cold L2: 2D
// grids of 48^2 ... 384^2 px with 64 ... 192 elements, 3D of 20^3 ... 64^3 voxels with 256 and
// 576, 1 ... 9 transmits, F-numbers 1 ... 6 and no aperture, all storage types.
//  * L1 kernels (5 to 16 frames, odd and long ensembles): 1.05 ... 5.5 wherever V >= 6 S.
//  * Staged kernels of 32 frames, which read split or interleaved rows as they are: 0.59 ... 1.8 below
//    1e7 points, four fifths of them slower; from there on 0.64 ... 1.4 at shares of 1/9 and below,
//    seven tenths of them slower; else 0.81 ... 2.15, nine tenths of them faster, half above 1.23.  (The
//    slower ones are mostly 2D grids at shares of 0.12 to 0.2, among others of 1.1 to 1.5.)
//  * Staged kernels of 64 frames (33 to 64): a tile holds 8 x 4 or 16 x 4 voxels for all frames, and
//    two frame tiles double the term evaluations: 0.40 ... 1.5, slower in more than half of the
//    grids.  From three waves of two blocks per SM and a share of 0.4 on, where the direct
//    kernel's tail is short and its terms many: 0.98 ... 1.5, half of them above 1.13; at shares of
//    0.33 to 0.36 from 0.94 on.  (A 64-frame ring of two pairs,
//    taken for long windows: 0.87 ... 2.4, from 2e7 points on 0.97 ... 2.4.)
// A batch's instances have other kernels to compare with: batch.cpp decides.
static bool repack_pays(Variant direct, double points, double share, int64_t tiles) {
  switch (direct) {
    case V_ST32_C64_V4W7: case V_ST32_C64P_V4W7: case V_ST32_H16_V4: case V_ST32_B16_V4:
      return points >= 1e7 && share >= 0.1125;
    case V_ST64_C64: return points >= 2e7;
    case V_ST64_C64_V4: case V_ST64_C64P_V4: case V_ST64_H16_V4: case V_ST64_B16_V4: case V_ST64_H16:
      return tiles >= 3 * 2 * 152 && share >= 0.4;
    default: return true;
  }
}

// What a plan is for: runs of its own, a batch's repacked launches, a batch's lane mappings.
enum PlanFor { kForRuns, kForBatch, kForLanes };

static mach_status repack_plan(mach_plan_s* p, const DasParams& b, bool list, cudaStream_t s,
                               size_t total_mem, PlanFor use) {
  const VariantShape& direct = variant_shape(p->variant);
  if (direct.exact_frames || direct.channel_lanes) return MACH_OK;
  const int64_t N = static_cast<int64_t>(b.T) * b.C * b.S;
  if (b.V < static_cast<int64_t>(direct.staged ? 16 : 6) * b.S || N > (int64_t{1} << 36)) return MACH_OK;
  const FrameSplit fs = split_frames(b.F);
  const size_t iq_bytes = static_cast<size_t>(N) * 8 * fs.padded();
  const size_t pd_bytes = fs.tiles() > 1 ? sizeof(float) * static_cast<size_t>(b.V) * fs.tiles() : 0;
  if (iq_bytes + pd_bytes > total_mem / 16 || b.S > kWindowsHold) return MACH_OK;
  if (fs.full > 65535) return MACH_OK;   // grid y limit
  const bool grid3d = !list && b.ny > 1;
  struct Want { Variant v; int tiles; } want[2];
  int n = 0;
  if (fs.full) want[n++] = {grid3d ? V_SX32_F8V1W7_T8X7E : V_SX32_F8V1W7T14E, fs.full};
  // Tails, time of the exact-frame kernel alone (256 x 256 px, 128 elements, 1 transmit |
  // 201 x 233 px, 192 elements, 3 transmits | 64^3 voxels, 1024 elements, 3 transmits):
  //   16 frames: 8 per lane, 7 warps 81 | 144 | 3840 us, 4 warps 83 | 130 | 3621 us;
  //              4 per lane, 7 warps 91 | 124 | 5345 us
  //    8 frames: 4 per lane, 7 warps 64 | 115 | 2947 us; 8 per lane, 4 warps 91 | 138 | 2672 us
  if (fs.tail == 8) want[n++] = {grid3d ? V_SX8_F8V1W4 : V_SX8_F4V1W7, 1};
  if (fs.tail == 16) want[n++] = {grid3d ? V_SX16_F8V1W4 : b.T == 1 ? V_SX16_F8V1W7 : V_SX16_F4V1W7, 1};
  BoundStats* d_stats = nullptr;
  int64_t scratch = 0, bytes = 0;
  // every way out but the last one leaves the plan on its direct kernel
  auto done = [&](mach_status e) {
    cudaFree(d_stats);
    if (p->n_parts == 0)
      for (auto& q : p->parts) {
        cudaFree(q.d_tbox);
        cudaFree(q.d_txr);
        q.d_tbox = nullptr;
        q.d_txr = nullptr;
      }
    return e;
  };
  if (dev_alloc(reinterpret_cast<void**>(&d_stats), 2 * sizeof(BoundStats), &scratch) != MACH_OK) return done(MACH_OK);
  for (int k = 0; k < n; ++k) {
    RepackPart& q = p->parts[k];
    const VariantShape& sh = variant_shape(want[k].v);
    DasParams t = b;
    if (configure_tiles(t, want[k].v, list, b.V, sh.frame_tile) != MACH_OK) return done(MACH_OK);
    const int64_t tiles = static_cast<int64_t>(t.tiles_x) * t.tiles_y * t.tiles_z;
    if (dev_alloc(reinterpret_cast<void**>(&q.d_tbox), sizeof(float4) * 2 * tiles, &bytes) != MACH_OK ||
        dev_alloc(reinterpret_cast<void**>(&q.d_txr), sizeof(float2) * b.T * tiles, &bytes) != MACH_OK)
      return done(MACH_OK);
    t.F = sh.frame_tile;
    t.frame_tiles = fs.tiles();
    t.tbox = q.d_tbox;
    t.txr = q.d_txr;
    t.f_first = k == 0 ? 0 : 32 * fs.full;
    t.f_total = b.F;
    t.f_tile = k == 0 ? 0 : fs.full;
    t.iq_tile_bytes = static_cast<size_t>(N) * 8 * sh.frame_tile;
    q.v = want[k].v;
    q.tiles = want[k].tiles;
    q.base = t;
    q.at = k == 0 ? 0 : static_cast<size_t>(N) * 8 * 32 * fs.full;
    if (launch_tile_bounds(t, q.d_tbox, q.d_txr, d_stats + k, s) != cudaSuccess) return done(MACH_ERR_CUDA);
  }
  BoundStats stats[2] = {};
  if (cudaMemcpyAsync(stats, d_stats, n * sizeof(BoundStats), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
      cudaStreamSynchronize(s) != cudaSuccess)
    return done(MACH_ERR_CUDA);
  double points = 0.0;
  int lo = b.S, hi = 0;
  for (int k = 0; k < n; ++k) {
    DasParams& t = p->parts[k].base;
    t.rows_cap = std::max(2, stats[k].rows);
    if (!windows_hold(b.S, float_of(stats[k].reach_bits))) return done(MACH_OK);   // its kernels have no other way
    if (repacked_smem_bytes(want[k].v, t.rows_cap, b.T) > kStagedSmemCap) return done(MACH_OK);
    lo = std::min(lo, b.S - stats[k].from_end);
    hi = std::max(hi, stats[k].last);
    points += static_cast<double>(stats[k].pairs) * (t.tile_x * t.tile_y * t.tile_z) * t.F * want[k].tiles;
  }
  p->range[0] = lo;
  p->range[1] = hi;
  const double all = static_cast<double>(b.V) * b.C * b.T * fs.padded();
  if (!g_force_repack && use != kForBatch &&
      !repack_pays(p->variant, points, points / all, static_cast<int64_t>(b.tiles_x) * b.tiles_y * b.tiles_z))
    return done(MACH_OK);
  p->points = points;
  p->pd_at = iq_bytes;
  p->ws_bytes = iq_bytes + pd_bytes;
  if (use == kForBatch) {
    p->device_bytes += bytes;
    p->n_parts = n;
    return done(MACH_OK);
  }
  // each run takes its workspace in stream order, so that calls on several streams never share one
  p->pool = take_pool(p->device, p->ws_bytes);
  if (!p->pool) return done(MACH_OK);
  void* first = nullptr;   // mapped now rather than in the first run
  if (alloc_denied() || cudaMallocFromPoolAsync(&first, p->ws_bytes, p->pool, s) != cudaSuccess ||
      cudaFreeAsync(first, s) != cudaSuccess) {
    cudaGetLastError();
    return_pool(p->device, p->ws_bytes);
    p->pool = nullptr;
    return done(MACH_OK);
  }
  p->device_bytes += bytes + static_cast<int64_t>(p->ws_bytes);   // kept by the pool, once for all plans
  p->n_parts = n;
  return done(MACH_OK);
}

static mach_status make_plan(const mach_das_desc* d, void* stream, PlanFor use, mach_plan* out) {
  if (!out) return MACH_ERR_INVALID_ARG;
  *out = nullptr;
  mach_status st = validate(d);
  if (st != MACH_OK) return st;
  cudaStream_t s = static_cast<cudaStream_t>(stream);

  const int C = d->n_elem, T = d->n_tx, S = d->n_samples, F = d->n_frames;
  const bool list = d->vox_pos != nullptr;
  const int64_t V = list ? d->n_vox
                         : static_cast<int64_t>(d->grid_dims[0]) * d->grid_dims[1] * d->grid_dims[2];
  if (list && V > INT32_MAX) return MACH_ERR_UNSUPPORTED;
  Variant var = pick_variant(d->iq_dtype, F);
  // 3D grids with 32 frames: one-plane 8 x 7 x 1 tiles.  A step in depth moves the two-way
  // delay about twice as far as the step itself, a lateral step far less, so a tile one
  // plane deep needs the shortest sample windows; with 256-byte rows that shrinks the ring
  // (15 instead of 36 rows a slot) and more blocks stay resident (94 x 94 x 178 voxels,
  // 1024 elements: 2.82 T points/s, against 2.31 for 8 x 2 x 7 tiles at 4 frames per lane
  // and 2.10 for 8 x 1 x 7 tiles at 8)
  if (var == V_SX32_F8V1W7T14E && !list && d->grid_dims[1] > 1) var = V_SX32_F8V1W7_T8X7E;
  // 2D grids with 64 frames: shallow 16 x 4 tiles keep the windows short enough for the
  // 8-slot ring of 512-byte rows (the squarest 8 x 8 tiles do not fit; the L1 path then
  // ran 256 x 256 px at 1.47 against 2.11 T points/s)
  if (var == V_SX64_C64P && !list && d->grid_dims[1] == 1) var = V_SX64_C64P_T16;
  if (d->term_table) var = generic_staged(var);
  const bool forced = g_force_variant >= 0;
  if (forced) {
    if (g_force_variant >= V_COUNT || !variant_accepts(static_cast<Variant>(g_force_variant), d->iq_dtype, F))
      return MACH_ERR_UNSUPPORTED;
    var = static_cast<Variant>(g_force_variant);
  }

  DasParams b{};
  if (list) {
    b.nx = static_cast<int>(V);
    b.ny = b.nz = 1;
  } else {
    b.nx = d->grid_dims[0];
    b.ny = d->grid_dims[1];
    b.nz = d->grid_dims[2];
  }
  if ((st = configure_tiles(b, var, list, V, F)) != MACH_OK) return st;
  const int64_t tiles0 = static_cast<int64_t>(b.tiles_x) * b.tiles_y * b.tiles_z;

  // host-side size check before touching the device
  const size_t need = static_cast<size_t>(V) * (sizeof(float4) + sizeof(float) * T) + sizeof(float4) * C +
                      (b.frame_tiles > 1 ? sizeof(float) * V * b.frame_tiles : 0) +
                      (list ? sizeof(float) * 3 * V : 0) + sizeof(double) * 3 * T +
                      (variant_shape(var).staged ? static_cast<size_t>(tiles0) * (2 * sizeof(float4) + T * sizeof(float2)) : 0);
  size_t free_b = 0, total_b = 0;
  if (cudaMemGetInfo(&free_b, &total_b) != cudaSuccess) {
    cudaGetLastError();
    return MACH_ERR_CUDA;
  }
  if (need > free_b) return MACH_ERR_OOM;

  const double k = d->fs / d->c;
  const double t0fs = d->t0 * d->fs;
  std::vector<float4> elem(C);
  for (int c = 0; c < C; ++c)
    elem[c] = make_float4(static_cast<float>(static_cast<double>(d->elem_pos[3 * c]) * k),
                          static_cast<float>(static_cast<double>(d->elem_pos[3 * c + 1]) * k),
                          static_cast<float>(static_cast<double>(d->elem_pos[3 * c + 2]) * k), 0.0f);
  std::vector<double> u;
  if (!d->tx_table_dev) {
    u.resize(3 * static_cast<size_t>(T));
    for (int t = 0; t < T; ++t) {
      const double az = d->tx_angles[2 * t], el = d->tx_angles[2 * t + 1];
      u[3 * t] = std::sin(az) * std::cos(el);
      u[3 * t + 1] = std::sin(el);
      u[3 * t + 2] = std::cos(az) * std::cos(el);
    }
  }

  mach_plan_s* p = new (std::nothrow) mach_plan_s();
  if (!p) return MACH_ERR_OOM;
  p->d = *d;
  p->d.elem_pos = nullptr;
  p->d.vox_pos = nullptr;
  p->d.tx_angles = nullptr;
  p->d.tx_table_dev = nullptr;
  p->d.n_vox = V;
  p->variant = var;
  cudaGetDevice(&p->device);

  float* d_raw = nullptr;
  double* d_u = nullptr;
  BoundStats* d_stats = nullptr;
  int64_t scratch_bytes = 0;
  auto fail = [&](mach_status e) {
    cudaFree(d_raw);
    cudaFree(d_u);
    cudaFree(d_stats);
    release(p);
    return e;
  };
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_vox), sizeof(float4) * V, &p->device_bytes)) != MACH_OK) return fail(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_elem), sizeof(float4) * C, &p->device_bytes)) != MACH_OK) return fail(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_tx), sizeof(float) * T * V, &p->device_bytes)) != MACH_OK) return fail(st);
  if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_err), sizeof(int), &p->device_bytes)) != MACH_OK) return fail(st);
  if (list && (st = dev_alloc(reinterpret_cast<void**>(&d_raw), sizeof(float) * 3 * V, &scratch_bytes)) != MACH_OK)
    return fail(st);
  if (!u.empty() && (st = dev_alloc(reinterpret_cast<void**>(&d_u), sizeof(double) * u.size(), &scratch_bytes)) != MACH_OK)
    return fail(st);

  if (cudaMemsetAsync(p->d_err, 0, sizeof(int), s) != cudaSuccess) return fail(MACH_ERR_CUDA);
  if (cudaMemcpyAsync(p->d_elem, elem.data(), sizeof(float4) * C, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return fail(MACH_ERR_CUDA);
  if (list && cudaMemcpyAsync(d_raw, d->vox_pos, sizeof(float) * 3 * V, cudaMemcpyHostToDevice, s) != cudaSuccess)
    return fail(MACH_ERR_CUDA);
  if (d_u && cudaMemcpyAsync(d_u, u.data(), sizeof(double) * u.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
    return fail(MACH_ERR_CUDA);

  TableParams tp{};
  tp.raw_vox = d_raw;
  tp.u = d_u;
  tp.tx_seconds = d->tx_table_dev;
  tp.k = k;
  tp.t0fs = t0fs;
  tp.fs = d->fs;
  for (int a = 0; a < 3; ++a) {
    tp.origin[a] = list ? 0.0 : d->grid_origin[a];
    tp.step[a] = list ? 0.0 : d->grid_step[a];
  }
  tp.nx = list ? 1 : d->grid_dims[0];
  tp.ny = list ? 1 : d->grid_dims[1];
  tp.nz = list ? 1 : d->grid_dims[2];
  tp.V = V;
  tp.T = T;
  tp.vox_out = p->d_vox;
  tp.tx_out = p->d_tx;
  if (launch_tables(tp, s) != cudaSuccess) return fail(MACH_ERR_CUDA);

  b.vox = p->d_vox;
  b.elem = p->d_elem;
  b.tx = p->d_tx;
  b.pd_part = p->d_pd_part;
  b.V = V;
  b.C = C;
  b.T = T;
  b.S = S;
  b.F = F;
  b.ystride = F;
  b.txr_stride = T;
  b.apod = d->apod;
  b.two_f = static_cast<float>(2.0 * d->f_number);
  b.f_num = static_cast<float>(d->f_number);
  b.four_f2 = static_cast<float>(4.0 * d->f_number * d->f_number);
  b.f_num2 = static_cast<float>(d->f_number * d->f_number);
  b.s_max = static_cast<float>(S - 1);
  b.r_f = static_cast<float>(d->fc / d->fs);
  b.phase_R = fixed_cycles(d->fc / d->fs);
  b.phase_Phi = fixed_cycles(d->fc * d->t0);
  b.err = p->d_err;
  b.wait_limit = g_wait_limit ? g_wait_limit : kDefaultWaitLimit;
  b.debug_stall = g_stall;

  if (variant_shape(var).staged) {
    // per-tile bounds, ring size, and the number of windows one run copies.  When the
    // chosen variant's ring does not fit, variants with fewer ring slots are tried in turn
    // (their tiles differ, so each gets its own bounds), and last the L1-path variant.
    const bool tab = d->term_table != 0;
    Variant chain[4];
    int nchain = 0;
    chain[nchain++] = var;
    if (!forced)
      for (Variant f = staged_fallback(var); f != chain[nchain - 1] && nchain < 4; f = staged_fallback(f))
        chain[nchain++] = f;
    int64_t tiles_max = tiles0;
    for (int k = 1; k < nchain; ++k) {
      DasParams tmp = b;
      if ((st = configure_tiles(tmp, chain[k], list, V, F)) != MACH_OK) return fail(st);
      tiles_max = std::max<int64_t>(tiles_max, static_cast<int64_t>(tmp.tiles_x) * tmp.tiles_y * tmp.tiles_z);
    }
    if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_tbox), sizeof(float4) * 2 * tiles_max, &p->device_bytes)) != MACH_OK)
      return fail(st);
    if ((st = dev_alloc(reinterpret_cast<void**>(&p->d_txr), sizeof(float2) * T * tiles_max, &p->device_bytes)) != MACH_OK)
      return fail(st);
    if ((st = dev_alloc(reinterpret_cast<void**>(&d_stats), sizeof(BoundStats), &scratch_bytes)) != MACH_OK)
      return fail(st);
    b.tbox = p->d_tbox;
    b.txr = p->d_txr;
    bool fits = false;
    for (int k = 0; k < nchain && !fits; ++k) {
      if (k > 0) {
        var = chain[k];
        p->variant = var;
        if ((st = configure_tiles(b, var, list, V, F)) != MACH_OK) return fail(st);
      }
      if (launch_tile_bounds(b, p->d_tbox, p->d_txr, d_stats, s) != cudaSuccess) return fail(MACH_ERR_CUDA);
      BoundStats stats{};
      if (cudaMemcpyAsync(&stats, d_stats, sizeof(stats), cudaMemcpyDeviceToHost, s) != cudaSuccess)
        return fail(MACH_ERR_CUDA);
      if (cudaStreamSynchronize(s) != cudaSuccess) return fail(MACH_ERR_CUDA);
      p->rows_cap = std::max(2, stats.rows);
      p->copy_pairs = static_cast<int64_t>(stats.pairs);
      b.rows_cap = p->rows_cap;
      b.inside = windows_hold(S, float_of(stats.reach_bits));
      fits = staged_smem_bytes(var, p->rows_cap, F, T, tab) <= kStagedSmemCap;
    }
    if (!fits) {
      if (forced || tab) return fail(MACH_ERR_UNSUPPORTED);
      // the tiles' windows are too long for any ring: use the L1-cached variant
      cudaFree(p->d_tbox);
      cudaFree(p->d_txr);
      p->d_tbox = nullptr;
      p->d_txr = nullptr;
      b.tbox = nullptr;
      b.txr = nullptr;
      p->device_bytes -= static_cast<int64_t>(sizeof(float4) * 2 * tiles_max + sizeof(float2) * T * tiles_max);
      var = unstaged(var);
      p->variant = var;
      p->rows_cap = 0;
      p->copy_pairs = 0;
      if ((st = configure_tiles(b, var, list, V, F)) != MACH_OK) return fail(st);
    }
  }
  // partial Power Doppler sums when the frames span several frame tiles (known once the
  // variant is final)
  if (b.frame_tiles > 1 &&
      (st = dev_alloc(reinterpret_cast<void**>(&p->d_pd_part), sizeof(float) * b.frame_tiles * V, &p->device_bytes)) != MACH_OK)
    return fail(st);
  b.pd_part = p->d_pd_part;
  if (d->term_table) {
    // every term evaluated once here; runs read them instead of computing them
    if (!variant_shape(var).staged || !table_supported(var)) return fail(MACH_ERR_UNSUPPORTED);
    if ((st = build_term_table(p, b, s)) != MACH_OK) return fail(st);
  }
  if (use != kForLanes && !forced && !d->term_table && (st = repack_plan(p, b, list, s, total_b, use)) != MACH_OK)
    return fail(st);
  if (cudaStreamSynchronize(s) != cudaSuccess) return fail(MACH_ERR_CUDA);
  cudaFree(d_raw);
  cudaFree(d_u);
  cudaFree(d_stats);
  d_raw = nullptr;
  d_u = nullptr;
  d_stats = nullptr;
  p->base = b;
  *out = p;
  return MACH_OK;
}

mach_status mach_das_plan(const mach_das_desc* d, void* stream, mach_plan* out) {
  try {
    return make_plan(d, stream, kForRuns, out);
  } catch (const std::bad_alloc&) {   // of the host copies of the elements and transmits
    return MACH_ERR_OOM;
  }
}

mach_status mach_plan_destroy(mach_plan p) {
  if (!p) return MACH_OK;
  release(p);
  return MACH_OK;
}

// One run over the repacked ensemble; false (nothing launched) when the stream is being
// captured, where a run makes no allocation, or when there is no memory for the workspace.
static bool run_repacked(mach_plan p, const void* iq, float* pd, void* y, cudaStream_t s, cudaError_t* err) {
  cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(s, &cap) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  if (cap != cudaStreamCaptureStatusNone) return false;
  char* ws = nullptr;
  if (alloc_denied() || cudaMallocFromPoolAsync(reinterpret_cast<void**>(&ws), p->ws_bytes, p->pool, s) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  const DasParams& b = p->base;
  cudaError_t e = launch_iq_repack(iq, nullptr, p->d.iq_dtype, reinterpret_cast<float*>(ws),
                                   static_cast<int64_t>(b.T) * b.C, b.S, p->range[0], p->range[1], b.F, s);
  float* part = reinterpret_cast<float*>(ws + p->pd_at);
  for (int k = 0; k < p->n_parts && e == cudaSuccess; ++k) {
    DasParams q = p->parts[k].base;
    q.iq = ws + p->parts[k].at;
    q.y = static_cast<float2*>(y);
    q.pd = pd;
    q.pd_part = part;
    e = launch_das_parts(q, p->parts[k].v, p->parts[k].tiles, s);
  }
  const int tiles = p->parts[0].base.frame_tiles;
  if (e == cudaSuccess && pd && tiles > 1) e = launch_pd_reduce(part, pd, nullptr, b.V, tiles, s);
  const cudaError_t f = cudaFreeAsync(ws, s);
  *err = e != cudaSuccess ? e : f;
  return true;
}

static mach_status run(mach_plan p, const void* iq, float* pd, void* y, void* stream) {
  if (!p || !iq || (!pd && !y)) return MACH_ERR_INVALID_ARG;
  // vector loads and bulk copies need 16-byte aligned IQ; outputs are float2 / float4
  if ((reinterpret_cast<uintptr_t>(iq) & 15u) || (reinterpret_cast<uintptr_t>(y) & 15u) ||
      (reinterpret_cast<uintptr_t>(pd) & 3u))
    return MACH_ERR_INVALID_ARG;
  cudaError_t re = cudaSuccess;
  if (p->pool && run_repacked(p, iq, pd, y, static_cast<cudaStream_t>(stream), &re))
    return re == cudaSuccess ? MACH_OK : MACH_ERR_CUDA;
  DasParams q = p->base;
  q.iq = iq;
  q.y = static_cast<float2*>(y);
  q.pd = pd;
  const cudaError_t e = p->table ? launch_das_table(q, p->variant, static_cast<cudaStream_t>(stream))
                                 : launch_das(q, p->variant, static_cast<cudaStream_t>(stream));
  return e == cudaSuccess ? MACH_OK : MACH_ERR_CUDA;
}

mach_status mach_das_run(mach_plan p, const void* iq_dev, void* y_dev, void* stream) {
  if (!y_dev) return MACH_ERR_INVALID_ARG;
  return run(p, iq_dev, nullptr, y_dev, stream);
}

mach_status mach_das_run_per_tx(mach_plan p, const void* iq_dev, void* y_dev, void* stream) {
  if (!p || !iq_dev || !y_dev) return MACH_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(iq_dev) & 15u) || (reinterpret_cast<uintptr_t>(y_dev) & 15u))
    return MACH_ERR_INVALID_ARG;
  const DasParams& b = p->base;
  const int T = b.T, F = b.F;
  // bytes of one transmit's IQ block [C][S][F] (split rows hold the same values)
  const size_t sample_bytes = (p->d.iq_dtype == MACH_IQ_F16X2 || p->d.iq_dtype == MACH_IQ_BF16X2) ? 4 : 8;
  const size_t tx_bytes = sample_bytes * static_cast<size_t>(b.C) * b.S * F;
  // vector stores need each transmit's slice of a row on the same alignment as the row
  const int vec = F % 4 == 0 ? 4 : (F % 2 == 0 ? 2 : 1);
  if ((static_cast<int64_t>(T) * F) % vec) return MACH_ERR_UNSUPPORTED;
  for (int t = 0; t < T; ++t) {
    DasParams q = b;
    q.T = 1;
    q.tx = b.tx + static_cast<size_t>(t) * b.V;
    q.txr = b.txr ? b.txr + t : nullptr;
    q.iq = static_cast<const char*>(iq_dev) + t * tx_bytes;
    q.y = static_cast<float2*>(y_dev) + static_cast<size_t>(t) * F;
    q.ystride = static_cast<int64_t>(T) * F;
    q.pd = nullptr;
    const cudaError_t e = launch_das(q, p->variant, static_cast<cudaStream_t>(stream));
    if (e != cudaSuccess) return MACH_ERR_CUDA;
  }
  return MACH_OK;
}

mach_status mach_power_doppler(mach_plan p, const void* iq_dev, float* pd_dev, void* y_dev_or_null,
                               void* stream) {
  if (!pd_dev) return MACH_ERR_INVALID_ARG;
  return run(p, iq_dev, pd_dev, y_dev_or_null, stream);
}

mach_status mach_plan_get_info(mach_plan p, mach_plan_info* info) {
  if (!p || !info) return MACH_ERR_INVALID_ARG;
  std::memset(info, 0, sizeof(*info));
  const VariantShape& s = variant_shape(p->variant);
  std::strncpy(info->variant, s.name, sizeof(info->variant) - 1);
  if (p->pool) {   // the frame tiles that runs repack the ensemble into
    const size_t n = std::strlen(info->variant);
    std::snprintf(info->variant + n, sizeof(info->variant) - n, p->n_parts == 2 ? "+x%d+x%d" : "+x%d",
                  p->parts[0].base.F, p->parts[1].base.F);
  }
  info->frames_per_lane = s.frames_per_lane;
  info->lanes_per_voxel = s.lanes_per_voxel;
  info->voxels_per_cta = s.voxels_per_warp * s.warps;
  info->threads_per_cta = s.warps * 32;
  info->tile[0] = p->base.tile_x;
  info->tile[1] = p->base.tile_y;
  info->tile[2] = p->base.tile_z;
  info->frame_tiles = p->base.frame_tiles;
  info->ctas = static_cast<int64_t>(p->base.tiles_x) * p->base.tiles_y * p->base.tiles_z * p->base.frame_tiles;
  info->smem_bytes = static_cast<int64_t>(das_smem_bytes(p->variant));
  info->device_bytes = p->device_bytes;
  info->ring_rows = p->rows_cap;
  info->ring_slots = variant_shape(p->variant).ring_slots;
  info->copy_pairs = p->copy_pairs;
  info->term_table_bytes = p->table_bytes;
  if (variant_shape(p->variant).staged) {
    info->smem_bytes = static_cast<int64_t>(staged_smem_bytes(p->variant, p->rows_cap, p->base.F, p->base.T, p->table));
    info->threads_per_cta = (s.warps + 1) * 32;
  }
  return MACH_OK;
}

mach_status mach_plan_device_status(mach_plan p, void* stream) {
  if (!p) return MACH_ERR_INVALID_ARG;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  int err = 0;
  if (cudaMemcpyAsync(&err, p->d_err, sizeof(int), cudaMemcpyDeviceToHost, s) != cudaSuccess) return MACH_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return MACH_ERR_CUDA;
  if (err == 0) return MACH_OK;
  if (cudaMemsetAsync(p->d_err, 0, sizeof(int), s) != cudaSuccess) return MACH_ERR_CUDA;
  if (cudaStreamSynchronize(s) != cudaSuccess) return MACH_ERR_CUDA;
  return MACH_ERR_TIMEOUT;
}

mach_status mach_debug_force_variant(const char* name) {
  if (!name || !*name) {
    g_force_variant = -1;
    return MACH_OK;
  }
  for (int v = 0; v < V_COUNT; ++v)
    if (std::strcmp(variant_shape(static_cast<Variant>(v)).name, name) == 0) {
      g_force_variant = v;
      return MACH_OK;
    }
  return MACH_ERR_INVALID_ARG;
}

void mach_debug_force_repack(int32_t on) { g_force_repack = on != 0; }

void mach_debug_set_wait_limit(uint32_t polls) { g_wait_limit = polls; }

void mach_debug_stall_producer(int32_t on) { g_stall = on ? 1 : 0; }

mach_status mach_plan_tx_table(mach_plan p, float* out_dev, void* stream) {
  if (!p || !out_dev) return MACH_ERR_INVALID_ARG;
  const size_t bytes = sizeof(float) * static_cast<size_t>(p->base.T) * p->base.V;
  return cudaMemcpyAsync(out_dev, p->d_tx, bytes, cudaMemcpyDeviceToDevice, static_cast<cudaStream_t>(stream)) ==
                 cudaSuccess
             ? MACH_OK
             : MACH_ERR_CUDA;
}

mach_status mach_das_terms(mach_plan p, const int64_t* vox_idx_dev, int64_t n, int32_t* i0_dev, float* w_dev,
                           float* cw_dev, void* stream) {
  if (!p || n < 0 || (n > 0 && !vox_idx_dev)) return MACH_ERR_INVALID_ARG;
  return launch_terms(p->base, vox_idx_dev, n, i0_dev, w_dev, cw_dev, static_cast<cudaStream_t>(stream)) ==
                 cudaSuccess
             ? MACH_OK
             : MACH_ERR_CUDA;
}

}  // extern "C"

namespace mach {
bool alloc_denied() {
  return g_fail_alloc_countdown.load() > 0 && g_fail_alloc_countdown.fetch_sub(1) == 1;
}

mach_status dev_alloc(void** p, size_t bytes, int64_t* total) {
  *p = nullptr;
  if (alloc_denied()) return MACH_ERR_OOM;
  if (bytes == 0) bytes = 16;
  const cudaError_t e = cudaMalloc(p, bytes);
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return MACH_ERR_OOM;
  }
  if (e != cudaSuccess) return MACH_ERR_CUDA;
  *total += static_cast<int64_t>(bytes);
  return MACH_OK;
}

// Host steps shared with the allocation-free entry point (noalloc.cu): the same
// validation, choice among the non-staged kernels, voxel tiling and phase constants
// that a plan uses.
mach_status make_batch_plan(const mach_das_desc* d, bool repack, void* stream, mach_plan* out) {
  return make_plan(d, stream, repack ? kForBatch : kForLanes, out);
}
int plan_repack(mach_plan p, RepackNeeds* needs) {
  *needs = {p->parts, p->ws_bytes, p->pd_at, {p->range[0], p->range[1]}, p->points};
  return p->n_parts;
}
bool repack_forced() { return g_force_repack; }
mach_status host_validate(const mach_das_desc* d) { return validate(d); }
Variant host_unstaged_variant(int iq_dtype, int F) { return unstaged(pick_variant(iq_dtype, F)); }
mach_status host_configure_tiles(DasParams& b, Variant v, bool list, int64_t V, int F) {
  return configure_tiles(b, v, list, V, F);
}
uint32_t host_fixed_cycles(double cycles) { return fixed_cycles(cycles); }
}  // namespace mach

namespace mach {
const DasParams* plan_params(mach_plan p) { return p ? &p->base : nullptr; }
int plan_iq_dtype(mach_plan p) { return p ? p->d.iq_dtype : -1; }
void pick_tile_shape(int n, int nx, int ny, int nz, bool list, int tile[3]) { pick_tile(n, nx, ny, nz, list, tile); }
}  // namespace mach
