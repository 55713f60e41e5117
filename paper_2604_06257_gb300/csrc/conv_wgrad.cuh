// conv_wgrad.cuh -- weight gradient of the 3x3x3 "same" convolution,
//   dW[t][ci][co] += sum_v X[v + off(t)][ci] dY[v][co],
// on warp-level tensor cores (mma.sync m16n8k16, bfloat16 in, float32 accumulate) with the
// operands staged by TMA.  Part of k_conv_tc.cu, whose tensor-map encoder, waits and error
// word it uses.
//
// A block owns 16 input x 16 output channels, all 27 taps, and a run of 8 x 16 x 2 voxel
// tiles.  Per tile one warp's lane 0 loads the input halo brick (10 x 18 x 4 voxels, zero
// outside the volume) and the output-gradient tile (zero outside) as 8-channel groups of
// 16-byte voxel rows into a ring of four stages.  Twelve MMA warps share the work as
// 3 tap planes (dz) x 4 quarters of the tile's y rows, so that each scheduler holds three
// of them, and a warp keeps the 9 taps of its plane in registers (72 accumulators).  The
// products' K = 16 voxels are two x rows of 8: an ldmatrix half fragment is one x row at one
// dx, and serves the three dy that see it, so a plane of four rows takes 9 + 2 ldmatrix.x4
// for 36 MMAs (one fragment per tap would take 18 + 2).  At the end the quarters meet in
// shared memory and leave by one float32 atomic per weight and block.
//
// tcgen05 is not used: its M is at least 64, and in this brick layout (channel group outermost) the
// taps' voxel offsets and the channel groups are no arithmetic progression that one operand
// descriptor could walk.  (With the channel group between y and x they would be.)
// It runs at 440-490 TFLOP/s on every large layer (750 multiply-adds a cycle and SM): the
// warp-level MMA rate, not memory (16 -> 16 moves 1.1 GB in 495 us).  Batch 8, earlier kernel
// (whose copies' address arithmetic took more issue slots than its products) -> this one: 16 -> 16 at 128^3
// 1189 -> 495 us, 48 -> 16 4281 -> 1418, 32 -> 32 at 64^3 473 -> 260, 192 -> 64 at 32^3
// 897 -> 393, 128 -> 128 at 16^3 138 -> 88.  Layers of few tiles and many channel blocks lost: 64 -> 128
// at 1 x 9 x 11 x 13 voxels 12 -> 18 us, several waves of blocks of one tile each; one wave takes 10
// us, but its longer chains cost accuracy (see launch_conv_wgrad).
#pragma once

constexpr int kWgTZ = 2;                                        // z planes per tile
constexpr int kWgStages = 4;
constexpr int kWgMma = 12;                                      // MMA warps
constexpr uint32_t kWgAPitch = kHX * kHY * (kWgTZ + 2) * 16;    // one 8-channel group of the halo brick
constexpr uint32_t kWgGPitch = kTX * kTY * kWgTZ * 16;          // one 8-channel group of the gradient tile
constexpr uint32_t kWgStage = 2 * kWgAPitch + 2 * kWgGPitch;
constexpr uint32_t kWgSmem = kWgStages * kWgStage + 2 * kWgStages * 8;
static_assert(kWgAPitch % 128 == 0 && kWgGPitch % 128 == 0, "TMA destinations are 128-byte aligned");
static_assert(9 * 72 * 32 * 4 <= kWgStages * kWgStage, "the quarters' sums fit the stages");

struct WgradParams {
  float* dw;
  int Ci, Co;
  int tiles_x, tiles_y, tiles_z;
  int64_t tiles, per_block;
  uint32_t wait_limit;
  int debug_stall;
};

__device__ __forceinline__ void ldm_x4_trans(uint32_t (&r)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}
__device__ __forceinline__ void mma_16816(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                          uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__global__ void __launch_bounds__((kWgMma + 1) * 32, 1)
    k_conv3d_wgrad_tma(const __grid_constant__ CUtensorMap xmap, const __grid_constant__ CUtensorMap gmap,
                       const WgradParams p) {
  extern __shared__ __align__(1024) uint8_t wg_smem[];
  uint64_t* full = reinterpret_cast<uint64_t*>(wg_smem + kWgStages * kWgStage);
  uint64_t* empty = full + kWgStages;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cb = blockIdx.x % (p.Ci / 16) * 16, ob = blockIdx.x / (p.Ci / 16) * 16;   // first channels
  const int64_t t0 = static_cast<int64_t>(blockIdx.y) * p.per_block;
  const int64_t t1 = t0 + p.per_block < p.tiles ? t0 + p.per_block : p.tiles;
  if (threadIdx.x == 0) {
    for (int i = 0; i < kWgStages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kWgMma);
    }
    mbar_init_fence();
  }
  __syncthreads();

  if (warp == kWgMma) {   // ------------------------------------------------- copies
    if (lane == 0 && !p.debug_stall) {
      int k = 0;
      for (int64_t tile = t0; tile < t1; ++tile, ++k) {
        const int st = k % kWgStages;
        if (k >= kWgStages && !wait_spin(&empty[st], ((k / kWgStages) - 1) & 1, p.wait_limit)) {
          atomicOr(&g_conv_tc_err, 1);
          break;
        }
        const int tx = static_cast<int>(tile % p.tiles_x);
        int64_t r = tile / p.tiles_x;
        const int ty = static_cast<int>(r % p.tiles_y);
        r /= p.tiles_y;
        const int z0 = static_cast<int>(r % p.tiles_z) * kWgTZ, n = static_cast<int>(r / p.tiles_z);
        const uint32_t dst = smem_u32(wg_smem) + st * kWgStage;
        mbar_arrive_expect_tx(&full[st], kWgStage);
        for (int g = 0; g < 2; ++g) {
          tma_load_5d(dst + g * kWgAPitch, &xmap, cb + g * 8, tx * kTX - 1, ty * kTY - 1, z0 - 1, n,
                      &full[st]);
          tma_load_5d(dst + 2 * kWgAPitch + g * kWgGPitch, &gmap, ob + g * 8, tx * kTX, ty * kTY, z0, n,
                      &full[st]);
        }
      }
      await_copies(full, kWgStages, k);
    }
    return;
  }

  // ------------------------------------------------------------------------- MMAs
  const int wz = warp % 3, qy = warp / 3;      // tap plane dz + 1, quarter of the y rows
  const int mat = lane >> 3;
  // lane's row addresses inside a stage: A half fragments (channel group mat & 1, x row
  // mat >> 1 of a pair) and the B fragment (8-channel group lane >> 4, voxel lane & 15)
  const uint32_t a_lane = smem_u32(wg_smem) + (mat & 1) * kWgAPitch +
                          (wz * (kHX * kHY) + (4 * qy + (mat >> 1)) * kHX + (lane & 7)) * 16;
  const uint32_t b_lane = smem_u32(wg_smem) + 2 * kWgAPitch + (lane >> 4) * kWgGPitch + (qy * 32 + (lane & 15)) * 16;
  float acc[9][2][4];   // [3 dy + dx][output-channel half][fragment]
#pragma unroll
  for (int i = 0; i < 9; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) acc[i][j][0] = acc[i][j][1] = acc[i][j][2] = acc[i][j][3] = 0.f;

  int k = 0;
  for (int64_t tile = t0; tile < t1; ++tile, ++k) {
    const int st = k % kWgStages;
    if (!__all_sync(0xffffffffu, wait_spin(&full[st], (k / kWgStages) & 1, p.wait_limit))) {
      if (lane == 0) atomicOr(&g_conv_tc_err, 1);
      break;
    }
#pragma unroll
    for (int z = 0; z < kWgTZ; ++z) {
      const uint32_t a0 = a_lane + st * kWgStage + z * (kHX * kHY * 16);
      const uint32_t b0 = b_lane + st * kWgStage + z * (kTX * kTY * 16);
      uint32_t b[2][4];
      ldm_x4_trans(b[0], b0);
      ldm_x4_trans(b[1], b0 + 256);
#pragma unroll
      for (int dx = 0; dx < 3; ++dx) {
        uint32_t h[3][4];   // rows 2 i (registers 0, 1) and 2 i + 1 (2, 3) of the quarter's six
#pragma unroll
        for (int i = 0; i < 3; ++i) ldm_x4_trans(h[i], a0 + (2 * i * kHX + dx) * 16);
        auto row = [&](int y, int g) { return h[y >> 1][2 * (y & 1) + g]; };
#pragma unroll
        for (int dy = 0; dy < 3; ++dy) {
#pragma unroll
          for (int ks = 0; ks < 2; ++ks) {
            const int y = dy + 2 * ks;
#pragma unroll
            for (int j = 0; j < 2; ++j)
              mma_16816(acc[3 * dy + dx][j], row(y, 0), row(y, 1), row(y + 1, 0), row(y + 1, 1), b[ks][2 * j],
                        b[ks][2 * j + 1]);
          }
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(&empty[st]);
  }

  // quarters 1 ... 3 hand their sums to quarter 0 through the (drained) stages
  auto mma_sync_all = [] { asm volatile("bar.sync 1, %0;" ::"n"(kWgMma * 32) : "memory"); };
  float* part = reinterpret_cast<float*>(wg_smem);
  mma_sync_all();
  if (qy > 0) {
    float* dst = part + ((qy - 1) * 3 + wz) * (72 * 32) + lane;
#pragma unroll
    for (int i = 0; i < 9; ++i)
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 4; ++e) dst[((i * 2 + j) * 4 + e) * 32] = acc[i][j][e];
  }
  mma_sync_all();
  if (qy > 0) return;
#pragma unroll
  for (int i = 0; i < 9; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float* src = part + wz * (72 * 32) + ((i * 2 + j) * 4 + e) * 32 + lane;
        const float s = (acc[i][j][e] + src[0]) + (src[3 * 72 * 32] + src[6 * 72 * 32]);
        const int ci = cb + (lane >> 2) + 8 * (e >> 1);
        const int co = ob + 8 * j + 2 * (lane & 3) + (e & 1);
        atomicAdd(p.dw + (static_cast<int64_t>(wz * 9 + i) * p.Ci + ci) * p.Co + co, s);
      }
}
