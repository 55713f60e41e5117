// das_slices.cuh -- delay-and-sum for ensembles of up to four frames.
//
// With so few frames a term's evaluation and its two tap rows serve hardly anything else, so
// frames cannot fill the lanes.  A block of 8 warps beamforms a compact box of 32 voxels, one
// voxel per lane; warp w takes elements w, w + 8, ...  The voxels of a box sit within a few
// samples of one another for any one element, so a warp's gather touches two or three cache
// lines, and most elements outside the aperture are skipped by the whole warp.  (One voxel
// per 8 lanes with an element each, the mapping before, touched a line or two per lane: the
// L1's tag lookups, not the arithmetic, were the bound.)  The 8 partial sums of a voxel meet
// in shared memory, in the order of a pairwise tree.
// Bound now by the terms' evaluation (a rounded square root, window and phase per term serve
// one to four frames).  Before -> now, complex64, cold L2: 128 x 128 px, 128 elements, 3
// transmits, 1 frame 29.4 -> 23.2 us; 251 x 251 px, 1 transmit, 1 / 2 / 4 frames 39.6 -> 33.4,
// 39.6 -> 33.4, 51.8 -> 39.5 us; 64^3 voxels, 1024 elements, 3 transmits 1367 -> 945,
// 1447 -> 1123, 2048 -> 1377 us.  Same sums, bit for bit.
#pragma once

#include <cuda_runtime.h>
#include <cstdint>

#include "das_term.cuh"
#include "mach_internal.h"
#include "tap_mac.cuh"

namespace mach {

constexpr int kSlices = 8;     // element slices = warps of a block
constexpr int kSliceVox = 32;  // voxels of a block

// Both taps of F frames, row i0 at r0 (rows are F samples; F = 2 and 4 start on the vector grid).
template <class IQ, int F>
__device__ __forceinline__ void load_taps(const IQ* r0, float2 (&x0)[F], float2 (&x1)[F]) {
  constexpr int VEC = F == 4 ? 4 : F == 2 ? 2 : 1;
#pragma unroll
  for (int f = 0; f < F; f += VEC) {
    float2 a[VEC], b[VEC];
    load_vec<IQ, VEC, false>(r0 + f, a);
    load_vec<IQ, VEC, false>(r0 + F + f, b);
#pragma unroll
    for (int e = 0; e < VEC; ++e) {
      x0[f + e] = a[e];
      x1[f + e] = b[e];
    }
  }
}

// One block's 32 voxels; part: kSlices x F x 32 partial sums in shared memory.  Every thread of
// the block calls it.
template <class IQ, int F>
__device__ __forceinline__ void das_slices_tile(const DasParams& p, int64_t tile, float2* part) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t v = tile_voxel(p, tile, lane);
  const IQ* __restrict__ iq = static_cast<const IQ*>(p.iq);
  float2 acc[F];
#pragma unroll
  for (int f = 0; f < F; ++f) acc[f] = make_float2(0.f, 0.f);
  if (v >= 0) {
    const float4 vpos = p.vox[v];
    const float tx0 = __ldg(&p.tx[v]);
    for (int c = warp; c < p.C; c += kSlices) {
      const TermGeo geo = term_geometry(vpos, __ldg(&p.elem[c]), p);
      if (geo.a < 0.f) continue;
      for (int t = 0; t < p.T; ++t) {
        const float4 r = term_record(t == 0 ? tx0 : __ldg(&p.tx[static_cast<size_t>(t) * p.V + v]), geo, p);
        const int i0 = __float_as_int(r.w);
        if (i0 < 0) continue;
        const float4 cw = tap_weights(r);
        float2 x0[F], x1[F];
        load_taps<IQ, F>(iq + ((static_cast<size_t>(t) * p.C + c) * p.S + i0) * F, x0, x1);
#pragma unroll
        for (int f = 0; f < F; ++f) mac1(acc[f], cw.x, cw.y, cw.z, cw.w, x0[f], x1[f]);
      }
    }
  }
#pragma unroll
  for (int f = 0; f < F; ++f) part[(warp * F + f) * kSliceVox + lane] = acc[f];
  __syncthreads();
  if (warp != 0 || v < 0) return;
  float pw = 0.f;
#pragma unroll
  for (int f = 0; f < F; ++f) {
    float2 s[kSlices];
#pragma unroll
    for (int w = 0; w < kSlices; ++w) s[w] = part[(w * F + f) * kSliceVox + lane];
#pragma unroll
    for (int o = kSlices / 2; o > 0; o >>= 1)
#pragma unroll
      for (int w = 0; w < o; ++w) {
        s[w].x += s[w + o].x;
        s[w].y += s[w + o].y;
      }
    pw = fmaf(s[0].x, s[0].x, fmaf(s[0].y, s[0].y, pw));
    if (p.y) p.y[v * p.ystride + f] = s[0];
  }
  if (p.pd) p.pd[v] = pw;
}

}  // namespace mach
