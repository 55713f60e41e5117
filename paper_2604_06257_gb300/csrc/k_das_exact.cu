// k_das_exact.cu -- the staged delay-and-sum kernel for split complex64 rows when the
// ensemble fills the frame tile exactly (F = 8, 16, 32 or 64), with receive delays evaluated
// on the fly (Sec. 4.3's hybrid delays) and reused across the frames (Sec. 4.4); the same for
// the frame tiles of repacked ensembles, of one acquisition (launch_das_parts) or of many in
// one launch (launch_das_multi).
//
// Same work, order and arithmetic as k_das_staged<C64Planar, ...> (das_staged.cuh): the
// same producer warp stages each usable (element, transmit) pair's sample window into a
// shared-memory ring with one bulk copy, the same lanes evaluate the same terms, and every
// frame receives the same FMA sequence, so the outputs are bitwise equal.  What differs is
// the consumer's instruction stream, which bounds the generic kernel (about 84 thread
// instructions per 4 term-frames, 16 of them packed FMAs):
//  * the frame count is a compile-time constant, so a sample row is RB = 8 F bytes (F real
//    parts, then F imaginary parts) and the four tap loads of a term are one 32-bit shared
//    address plus constant offsets (0, F*4, RB, RB + F*4); no per-frame bounds tests;
//  * the lane that evaluates a term also forms its two complex tap weights and the byte
//    offset of its first tap row inside the staged window, so a consuming lane reads a
//    16-byte weight record and a 4-byte offset and adds one integer per term;
//  * all shared-memory traffic of the inner loop uses 32-bit shared addresses.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "das_staged.cuh"

namespace mach {
namespace {

// Shared memory: [ring slots][tap weights][row offsets][transmit-delay cache][slot metadata][barriers].
template <int NBUF>
struct ExactLayout {
  size_t slot_bytes, coef_bytes, offs_bytes, tx_bytes;
  __host__ __device__ ExactLayout(int rows_cap, int row_bytes, int T, int nwc)
      : slot_bytes((static_cast<size_t>(rows_cap) * row_bytes + 127) / 128 * 128),
        coef_bytes(static_cast<size_t>(nwc) * 32 * 16),
        offs_bytes(static_cast<size_t>(nwc) * 32 * 4),
        tx_bytes(T <= kTxCache ? static_cast<size_t>(nwc) * T * 32 * 4 : 0) {}
  __host__ __device__ size_t coef_off() const { return NBUF * slot_bytes; }
  __host__ __device__ size_t offs_off() const { return coef_off() + coef_bytes; }
  __host__ __device__ size_t tx_off() const { return offs_off() + offs_bytes; }
  __host__ __device__ size_t meta_off() const { return tx_off() + (tx_bytes + 15) / 16 * 16; }
  __host__ __device__ size_t bar_off() const { return meta_off() + NBUF * 32; }
  __host__ __device__ size_t total() const { return bar_off() + 2 * NBUF * 8; }
  // repacked tiles: two more rows, of zeros
  __host__ __device__ size_t zero_off() const { return (total() + 127) / 128 * 128; }
};

__device__ __forceinline__ float4 lds128(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds32(uint32_t a) {
  int v;
  asm volatile("ld.shared.b32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts128(uint32_t a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void sts32(uint32_t a, int v) {
  asm volatile("st.shared.b32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}

// One term into 4 frames of a lane (split rows): taps x0 = (re ar, im ai) at row i0 and
// x1 = (re br, im bi) at row i0 + 1, weights cw = (c0r, c0i, c1r, c1i).  Per frame the
// FMA sequence of tap_mac.cuh: re += c0r x0re - c0i x0im + c1r x1re - c1i x1im and
// im += c0r x0im + c0i x0re + c1r x1im + c1i x1re, two frames per packed FMA.
// acc[2h] = (re of frames 2h, 2h+1), acc[2h+1] = (im of frames 2h, 2h+1).
__device__ __forceinline__ void mac4(float2* acc, const float4 cw, const float4 ar, const float4 ai, const float4 br,
                                     const float4 bi) {
  const float2 C0R = make_float2(cw.x, cw.x), C0N = make_float2(-cw.y, -cw.y), C0I = make_float2(cw.y, cw.y);
  const float2 C1R = make_float2(cw.z, cw.z), C1N = make_float2(-cw.w, -cw.w), C1I = make_float2(cw.w, cw.w);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float2 x0r = h ? make_float2(ar.z, ar.w) : make_float2(ar.x, ar.y);
    const float2 x0i = h ? make_float2(ai.z, ai.w) : make_float2(ai.x, ai.y);
    const float2 x1r = h ? make_float2(br.z, br.w) : make_float2(br.x, br.y);
    const float2 x1i = h ? make_float2(bi.z, bi.w) : make_float2(bi.x, bi.y);
    float2& re = acc[2 * h];
    float2& im = acc[2 * h + 1];
    re = __ffma2_rn(C0R, x0r, re);
    re = __ffma2_rn(C0N, x0i, re);
    re = __ffma2_rn(C1R, x1r, re);
    re = __ffma2_rn(C1N, x1i, re);
    im = __ffma2_rn(C0R, x0i, im);
    im = __ffma2_rn(C0I, x0r, im);
    im = __ffma2_rn(C1R, x1i, im);
    im = __ffma2_rn(C1I, x1r, im);
  }
}

// Frame chunks of a lane: FPL / 4 chunks of 4 consecutive frames.  Chunk c of lane jl of
// lane group g starts at frame 4 (jl + FL (c ^ swz)), swz = g & 1 when FL = 4 and a lane
// holds two chunks: the two lane groups of a quarter warp then read opposite halves of
// their rows first, which keeps every 128-bit load free of bank conflicts.
// Rows of 8 and 16 frames leave several lane groups on the same banks (their real parts
// span 32 or 64 bytes), so every other group reads the imaginary parts first: it keeps its
// sums with real and imaginary parts exchanged and gets its weights with the imaginary
// parts negated (half_swap), which is the same FMA sequence.  With 8 frames per lane in
// rows of 16 the chunks alternate over pairs of groups, so a quarter warp's four groups read
// four different 32-byte pieces.
// Measured (256 x 256 px, 128 elements | 64^3 voxels, 1024 elements, 3 transmits): 16 frames,
// 4 x 2 per lane 101 -> 93 us | 4562 -> 4163 us; at 8 frames per lane 81 | 3840 us.
template <int FL, int FPL>
__device__ __forceinline__ int chunk_swizzle(int g) {
  return FPL == 8 ? (FL == 4 ? (g & 1) : FL <= 2 ? ((g >> 1) & 1) : 0) : 0;
}
template <int FT, int FPL>
constexpr bool kHalves = FT == 16 || (FT == 8 && FPL == 8);   // at 4 frames per lane in rows of 8 it gains nothing
template <int FT, int FPL>
__device__ __forceinline__ int half_swap(int g) {
  return kHalves<FT, FPL> ? (g & 1) : 0;
}

// Accumulators of one lane: VPG voxel slots x FPL frames, as packed pairs.
template <int VPG, int FPL>
struct Acc {
  float2 a[VPG][FPL];
};

// The terms of one pair when some kept term falls outside the staged window (delays beyond
// those that windows_hold covers): such terms read their taps from global memory.
// Out of line, with the accumulators passed and returned by value, so that neither its
// registers nor an address of the accumulators burden the hot loop.
template <int FT, int FPL, int VPG, int G>
__device__ __noinline__ Acc<VPG, FPL> outside_pair(const DasParams& p, Acc<VPG, FPL> acc, const SlotMeta m,
                                                   const unsigned char* wsrc, uint32_t cw_at, uint32_t of_at, int jl,
                                                   int order) {
  constexpr int RB = FT * 8, IMO = FT * 4, FL = FT / FPL;
  const int swz = kHalves<FT, FPL> ? order & 1 : order, hs = kHalves<FT, FPL> ? order >> 1 : 0;   // chunk and half orders
  const unsigned char* gsrc =
      static_cast<const unsigned char*>(p.iq) + ((static_cast<size_t>(m.t) * p.C + m.c) * p.S + m.lo) * RB + jl * 16;
#pragma unroll
  for (int k = 0; k < VPG; ++k) {
    const float4 cw = lds128(cw_at + k * G * 16);
    const int off = lds32(of_at + k * G * 4);
    const int rrow = off / RB;
    const unsigned char* src = (rrow >= 0 && rrow + 1 < m.rows ? wsrc : gsrc) + off;
#pragma unroll
    for (int c = 0; c < FPL / 4; ++c) {
      const unsigned char* x = src + (c ^ swz) * FL * 16 + hs * IMO;
      const unsigned char* z = src + (c ^ swz) * FL * 16 + (1 - hs) * IMO;
      mac4(&acc.a[k][4 * c], cw, *reinterpret_cast<const float4*>(x), *reinterpret_cast<const float4*>(z),
           *reinterpret_cast<const float4*>(x + RB), *reinterpret_cast<const float4*>(z + RB));
    }
  }
  return acc;
}

// FT: frames (= F); FPL frames per lane (4 or 8), FL = FT / FPL lanes per voxel, VPG voxel
// slots per lane group; NWC consumer warps + 1 producer warp; NBUF ring slots; MAXR
// registers per thread.
// FLAGS bit 0: consumers suspended in hardware while waiting for a window; bit 1: a warp
// releases each ring slot right after its last read instead of at the end of the round;
// bit 2: every kept term is known to lie in its staged window (windows_hold), so no term has to
// look for its taps elsewhere.
constexpr int kSleep = 1, kEarly = 2, kInside = 4;
// The plan decides that from the delays it has (DasParams::inside); the check and the
// out-of-line path behind it cost registers: 94 x 94 x 178 voxels, 32 frames 91.4 -> 89.7 ms
// without them.  Ensembles for which it does not hold are not repacked.
//
// PART: the launch covers frames p.f_first ... of an ensemble of p.f_total frames that the
// frame tiles need not fill.  A tile's rows (zero beyond the last
// frame) start p.iq_tile_bytes after the previous tile's, frames past the last one are not
// written, and Power Doppler leaves as one partial sum per tile when there are several.
// Dropped terms read two rows of zeros instead of the window's first two, so that an infinite
// or NaN sample reaches only the voxels whose kept terms touch it, as with the direct kernels
// that repacked ensembles would otherwise take.
//
// das_exact_block is one block's work.  W says what that is: voxel tile, frame tile and
// outputs, read where they are needed (a value kept across the hot loop costs registers that
// the 64 of a thread do not have: 1 % of a 94 x 94 x 178 volume, 6 % of a 25-frame run).
template <int FT, int FPL, int VPG, int NWC, int NBUF, int FLAGS, bool PART, class W>
__device__ __forceinline__ void das_exact_block(const DasParams& p, const W& w) {
  constexpr int FL = FT / FPL;
  constexpr int G = 32 / FL;
  constexpr int WV = G * VPG;
  constexpr int PB = 32 / WV;           // pairs whose terms one warp evaluates per round
  constexpr int RB = FT * 8;            // bytes per sample row
  constexpr int IMO = FT * 4;           // imaginary parts' offset inside a row
  static_assert(FPL == 4 || FPL == 8, "4 or 8 frames per lane");
  static_assert(WV * PB == 32, "a round must fill the warp");
  static_assert(NBUF >= PB && NBUF % PB == 0, "a round must fit in the ring");
  static_assert(!PART || (FLAGS & kInside) != 0, "outside_pair reads p.iq as one frame tile");
  extern __shared__ __align__(128) unsigned char smem[];
  const ExactLayout<NBUF> L(p.rows_cap, RB, p.T, NWC);
  SlotMeta* meta = reinterpret_cast<SlotMeta*>(smem + L.meta_off());
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + L.bar_off());
  uint64_t* empty = full + NBUF;
  const bool tx_cached = p.T <= kTxCache;
  float* txc_all = reinterpret_cast<float*>(smem + L.tx_off());

  const int lane = threadIdx.x & 31;
  const int warp = threadIdx.x >> 5;
  const int64_t tile = w.tile();

  if (threadIdx.x == 0) {
    for (int b = 0; b < NBUF; ++b) {
      mbar_init(&full[b], 1);
      mbar_init(&empty[b], NWC);
    }
    mbar_init_fence();
  }
  if constexpr (PART) {
    for (int i = threadIdx.x; i < 2 * RB / 16; i += (NWC + 1) * 32)
      sts128(smem_u32(smem) + static_cast<uint32_t>(L.zero_off()) + i * 16, make_float4(0.f, 0.f, 0.f, 0.f));
  }
  __syncthreads();

  if (warp == NWC) {   // producer
    int r = 0;
    const unsigned char* iq = static_cast<const unsigned char*>(p.iq);
    if constexpr (PART) iq += w.ftile() * p.iq_tile_bytes;
    const bool ok = produce_windows<NBUF>(p, iq, tile, lane, smem, L.slot_bytes, 8, meta, full, empty, r);
    if (lane == 0) finish_producer<NBUF, PB>(p, ok, r, meta, full, empty);
    return;
  }

  // ------------------------------------------------------------------ consumers
  // Lane group g (FL lanes) accumulates the frames of its chunks for the voxel slots
  // g VPG + k.  Each round lane group `sub` (WV lanes) evaluates the terms of pair r + sub
  // for the warp's WV voxels; the weights of voxel slot g VPG + k for pair i sit at entry
  // i WV + k G + g, so the G groups read G consecutive entries (conflict-free broadcast).
  const int g = lane / FL;
  const int jl = lane % FL;
  const int sub = lane / WV;
  const int q = lane % WV;
  const int swz = chunk_swizzle<FL, FPL>(g);
  const int hs = half_swap<FT, FPL>(g);
  const float im_sign = half_swap<FT, FPL>(q / VPG) ? -1.0f : 1.0f;   // of the group that reads this lane's terms
  float* txc = txc_all + warp * (p.T * 32);
  const int64_t v_term = tile_voxel_blocked(p, tile, warp * WV + q);
  const float4 vpos = v_term >= 0 ? p.vox[v_term] : make_float4(0.f, 0.f, 0.f, 0.f);
  const int store_at = sub * WV + (q % VPG) * G + (q / VPG);
  const uint32_t s0 = smem_u32(smem);
  const uint32_t coef_w = s0 + static_cast<uint32_t>(L.coef_off()) + warp * 32 * 16;
  const uint32_t offs_w = s0 + static_cast<uint32_t>(L.offs_off()) + warp * 32 * 4;
  const uint32_t slot_bytes = static_cast<uint32_t>(L.slot_bytes);
  const uint32_t lane_tap = s0 + jl * 16 + swz * FL * 16 + hs * IMO;   // chunk 0; chunk 1 at +/- FL * 16
  const uint32_t im_at = hs ? -IMO : IMO;                              // the other parts, from there
  if (tx_cached) {
    for (int t = 0; t < p.T; ++t) txc[t * 32 + lane] = v_term >= 0 ? p.tx[static_cast<size_t>(t) * p.V + v_term] : 0.f;
  }

  Acc<VPG, FPL> acc;
#pragma unroll
  for (int k = 0; k < VPG; ++k)
#pragma unroll
    for (int e = 0; e < FPL; ++e) acc.a[k][e] = make_float2(0.f, 0.f);

  int cur_c = -1;
  TermGeo geo;
  geo.rx = 0.f;
  geo.a = -1.f;
  bool ok = true, done = false;
  for (int r = 0; !done; r += PB) {
    const int mine = r + sub, my_slot = mine % NBUF;
    const bool got = (FLAGS & kSleep) ? mbar_wait_bounded_sleep(&full[my_slot], (mine / NBUF) & 1, p.wait_limit, 1000)
                              : mbar_wait_bounded(&full[my_slot], (mine / NBUF) & 1, p.wait_limit);
    if (__any_sync(0xffffffffu, !got)) {
      if (lane == 0) atomicOr(p.err, 1);
      ok = false;
      break;
    }
    const SlotMeta mm = meta[my_slot];
    float4 rec = make_float4(0.f, 0.f, 0.f, __int_as_float(-1));
    if (mm.c >= 0) {
      if (mm.c != cur_c) {
        cur_c = mm.c;
        geo.a = -1.f;
        if (v_term >= 0) geo = term_geometry(vpos, mm.e, p);
      }
      if (geo.a >= 0.f) {
        const float stx = tx_cached ? txc[mm.t * 32 + lane] : __ldg(&p.tx[static_cast<size_t>(mm.t) * p.V + v_term]);
        rec = term_record(stx, geo, p);
      }
    }
    // dropped terms: zero weights (rec.x = rec.y = rec.z = 0) and row 0 of the window
    const int i0 = __float_as_int(rec.w);
    const bool active = i0 >= 0;
    const int row = active ? i0 - mm.lo : 0;
    bool outside = false;
    if constexpr ((FLAGS & kInside) == 0) outside = active && (row < 0 || row + 1 >= mm.rows);
    float4 tw = tap_weights(rec);
    if constexpr (kHalves<FT, FPL>) {   // exact
      tw.y *= im_sign;
      tw.w *= im_sign;
    }
    sts128(coef_w + store_at * 16, tw);
    int off = row * RB;
    if constexpr (PART) {
      if (!active) off = static_cast<int>(L.zero_off()) - my_slot * static_cast<int>(slot_bytes);
    }
    sts32(offs_w + store_at * 4, off);
    const unsigned act = __ballot_sync(0xffffffffu, active);
    unsigned outm = 0u;
    if constexpr ((FLAGS & kInside) == 0) outm = __ballot_sync(0xffffffffu, outside);
    const unsigned ended = __ballot_sync(0xffffffffu, mm.c < 0);
    __syncwarp();
#pragma unroll
    for (int i = 0; i < PB; ++i) {
      const unsigned gm = WV == 32 ? 0xffffffffu : (((1u << (WV & 31)) - 1u) << (i * WV));
      if (ended & gm) {   // end marker: every later pair of the round is one too
        done = true;
        break;
      }
      const int slot = (r + i) % NBUF;
      if (!(act & gm)) {
        if constexpr ((FLAGS & kEarly) != 0) {
          if (lane == 0) mbar_arrive(&empty[slot]);
        }
        continue;
      }
      const uint32_t win = lane_tap + slot * slot_bytes;
      const uint32_t cw_at = coef_w + (i * WV + g) * 16;
      const uint32_t of_at = offs_w + (i * WV + g) * 4;
      if ((FLAGS & kInside) || !(outm & gm)) {
        // every kept term lies in the staged window: branch-free over the voxels
#pragma unroll
        for (int k = 0; k < VPG; ++k) {
          const float4 cw = lds128(cw_at + k * G * 16);
          const uint32_t a = win + lds32(of_at + k * G * 4);
#pragma unroll
          for (int c = 0; c < FPL / 4; ++c) {
            // chunk c lies (c ^ swz - swz) FL * 16 bytes from chunk 0's lane address
            const uint32_t b = a + ((c ^ swz) - swz) * FL * 16;
            if constexpr (kHalves<FT, FPL>) {
              const uint32_t z = b + im_at;
              mac4(&acc.a[k][4 * c], cw, lds128(b), lds128(z), lds128(b + RB), lds128(z + RB));
            } else {
              mac4(&acc.a[k][4 * c], cw, lds128(b), lds128(b + IMO), lds128(b + RB), lds128(b + RB + IMO));
            }
          }
        }
      } else {
        acc = outside_pair<FT, FPL, VPG, G>(p, acc, meta[slot], smem + slot * slot_bytes + jl * 16, cw_at, of_at,
                                            jl, kHalves<FT, FPL> ? swz | hs << 1 : swz);
      }
      if constexpr ((FLAGS & kEarly) != 0) {   // every lane has read the slot: release it
        __syncwarp();
        if (lane == 0) mbar_arrive(&empty[slot]);
      }
    }
    if constexpr ((FLAGS & kEarly) == 0) {
      __syncwarp();
      if (lane < PB) mbar_arrive(&empty[(r + lane) % NBUF]);
    }
  }
  if (!ok) return;

  // epilogue: complex frames and sum_f |y|^2 (Sec. 5), reduced over the FL lanes
#pragma unroll
  for (int k = 0; k < VPG; ++k) {
    const int64_t v = tile_voxel_blocked(p, tile, warp * WV + g * VPG + k);
    float pw = 0.f;
    if (hs) {   // sums kept with real and imaginary parts exchanged
#pragma unroll
      for (int e = 0; e < FPL; e += 2) {
        const float2 t = acc.a[k][e];
        acc.a[k][e] = acc.a[k][e + 1];
        acc.a[k][e + 1] = t;
      }
    }
#pragma unroll
    for (int c = 0; c < FPL / 4; ++c) {
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 a = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], e);
        pw = fmaf(a.x, a.x, fmaf(a.y, a.y, pw));
      }
      if (v >= 0 && w.y()) {
        const int f0 = 4 * (jl + FL * (c ^ swz));
        if constexpr (PART) {
          const int f = p.f_first + static_cast<int>(w.ftile()) * FT + f0;
          float2* dst = w.y() + v * p.ystride + f;
#pragma unroll
          for (int e = 0; e < 4; e += 2) {
            const float2 a = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], e), b = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], e + 1);
            if (p.ystride % 2 == 0) {   // even rows: pairs of frames on the 16-byte grid
              if (f + e < p.f_total) *reinterpret_cast<float4*>(dst + e) = make_float4(a.x, a.y, b.x, b.y);
            } else {
              if (f + e < p.f_total) dst[e] = a;
              if (f + e + 1 < p.f_total) dst[e + 1] = b;
            }
          }
          continue;
        }
        float2* dst = w.y() + v * p.ystride + f0;
        const float2 a0 = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], 0), a1 = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], 1);
        const float2 a2 = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], 2), a3 = acc_frame<C64Planar, 4>(&acc.a[k][4 * c], 3);
        *reinterpret_cast<float4*>(dst) = make_float4(a0.x, a0.y, a1.x, a1.y);
        *reinterpret_cast<float4*>(dst + 2) = make_float4(a2.x, a2.y, a3.x, a3.y);
      }
    }
#pragma unroll
    for (int o = FL / 2; o > 0; o >>= 1) pw += __shfl_xor_sync(0xffffffffu, pw, o);
    if (jl == 0 && v >= 0 && w.pd()) {
      if (PART && p.frame_tiles > 1)
        p.pd_part[static_cast<int64_t>(p.f_tile + static_cast<int>(w.ftile())) * p.V + v] = pw;
      else
        w.pd()[v] = pw;
    }
  }
}

// Work of a block of one acquisition's launch: the last tiles (deepest rows of the grid, the
// widest apertures: the most pairs) start first, so that the light shallow tiles fill the
// tail of the launch.
struct GridWork {
  const DasParams& p;
  __device__ __forceinline__ int64_t tile() const { return static_cast<int64_t>(gridDim.x) - 1 - blockIdx.x; }
  __device__ __forceinline__ unsigned ftile() const { return blockIdx.y; }
  __device__ __forceinline__ float2* y() const { return p.y; }
  __device__ __forceinline__ float* pd() const { return p.pd; }
};

template <int FT, int FPL, int VPG, int NWC, int NBUF, int MAXR, int FLAGS, bool PART = false>
__global__ void __launch_bounds__((NWC + 1) * 32) __maxnreg__(MAXR) k_das_exact(const DasParams p) {
  das_exact_block<FT, FPL, VPG, NWC, NBUF, FLAGS, PART>(p, GridWork{p});
}

// Many acquisitions in one launch: block b works on items[b] = (frame tile << 16 | entry of
// a.p, voxel tile).  The entries' tables and tilings travel as kernel parameters (read through
// the constant cache, like a single acquisition's); the bound output buffers are read from
// the instance table, so that a captured launch follows a later bind.
struct ItemWork {
  const MultiArgs& a;
  const int2* items;
  __device__ __forceinline__ int2 item() const { return items[blockIdx.x]; }
  __device__ __forceinline__ int entry() const { return item().x & 0xffff; }
  __device__ __forceinline__ int64_t tile() const { return item().y; }
  __device__ __forceinline__ unsigned ftile() const { return static_cast<unsigned>(item().x) >> 16; }
  __device__ __forceinline__ float2* y() const { return a.insts[a.inst[entry()]].p.y; }
  __device__ __forceinline__ float* pd() const { return a.insts[a.inst[entry()]].p.pd; }
};

template <int FT, int FPL, int VPG, int NWC, int NBUF, int MAXR, int FLAGS>
__global__ void __launch_bounds__((NWC + 1) * 32) __maxnreg__(MAXR)
    k_das_exact_multi(const __grid_constant__ MultiArgs a, const int2* items) {
  const ItemWork w{a, items};
  das_exact_block<FT, FPL, VPG, NWC, NBUF, FLAGS, true>(a.p[w.entry()], w);
}

}  // namespace

size_t repacked_smem_bytes(Variant v, int rows_cap, int T) {
  const VariantShape& sh = variant_shape(v);
  const int rb = sh.frame_tile * 8;
  return ExactLayout<8>(rows_cap, rb, T, sh.warps).zero_off() + 2 * rb;   // every such shape has 8 slots
}

size_t exact_smem_bytes(Variant v, int rows_cap, int T) {
  const VariantShape& sh = variant_shape(v);
  const int rb = sh.frame_tile * 8;
  switch (sh.ring_slots) {
    case 4: return ExactLayout<4>(rows_cap, rb, T, sh.warps).total();
    case 8: return ExactLayout<8>(rows_cap, rb, T, sh.warps).total();
    case 12: return ExactLayout<12>(rows_cap, rb, T, sh.warps).total();
    default: return ExactLayout<16>(rows_cap, rb, T, sh.warps).total();
  }
}

cudaError_t launch_das_exact(const DasParams& p, Variant v, cudaStream_t s) {
  if (p.F != variant_shape(v).frame_tile || p.frame_tiles != 1) return cudaErrorInvalidValue;
  const size_t sm = exact_smem_bytes(v, p.rows_cap, p.T);
  switch (v) {
    //                                        FT FPL VPG NWC NBUF MAXR FLAGS
    case V_SX32_C64P: case V_SX32_C64P_T8X14: return go_staged(k_das_exact<32, 4, 4, 7, 4, 64, 0>, 7, p, sm, s);
    case V_SX32_F4V2W7: return go_staged(k_das_exact<32, 4, 2, 7, 8, 64, 0>, 7, p, sm, s);
    case V_SX32_F8V1W7: return go_staged(k_das_exact<32, 8, 1, 7, 8, 64, 0>, 7, p, sm, s);
    case V_SX32_F4V2W15: return go_staged(k_das_exact<32, 4, 2, 15, 8, 64, 0>, 15, p, sm, s);
    case V_SX32_F8V1W15: case V_SX32_F8V1W15T24: case V_SX32_F8V1W15T40:
      return go_staged(k_das_exact<32, 8, 1, 15, 8, 64, 0>, 15, p, sm, s);
    case V_SX32_F8V1W15T24S: return go_staged(k_das_exact<32, 8, 1, 15, 8, 64, kSleep>, 15, p, sm, s);
    case V_SX32_F8V1W7T14: return go_staged(k_das_exact<32, 8, 1, 7, 8, 64, 0>, 7, p, sm, s);
    case V_SX32_F8V1W7T14E: case V_SX32_F8V1W7_T8X7E:
      return p.inside ? go_staged(k_das_exact<32, 8, 1, 7, 8, 64, kEarly | kInside>, 7, p, sm, s)
                      : go_staged(k_das_exact<32, 8, 1, 7, 8, 64, kEarly>, 7, p, sm, s);
    case V_SX32_F4V2W7T14: return go_staged(k_das_exact<32, 4, 2, 7, 8, 64, 0>, 7, p, sm, s);
    case V_SX32_F8V1W15T30R12: return go_staged(k_das_exact<32, 8, 1, 15, 12, 64, 0>, 15, p, sm, s);
    case V_SX32_F8V1W15T30R12E: return go_staged(k_das_exact<32, 8, 1, 15, 12, 64, kEarly>, 15, p, sm, s);
    case V_SX64_C64P: case V_SX64_C64P_T16: case V_SX64_C64P_T8X8:
      return p.inside ? go_staged(k_das_exact<64, 4, 4, 8, 8, 72, kInside>, 8, p, sm, s)
                      : go_staged(k_das_exact<64, 4, 4, 8, 8, 72, 0>, 8, p, sm, s);
    case V_SX64_C64P_T16E: return go_staged(k_das_exact<64, 4, 4, 8, 8, 72, kEarly>, 8, p, sm, s);
    case V_SX64_C64PS: return go_staged(k_das_exact<64, 4, 4, 8, 8, 72, kSleep>, 8, p, sm, s);
    case V_SX64_C64PE: return go_staged(k_das_exact<64, 4, 4, 8, 8, 72, kEarly>, 8, p, sm, s);
    case V_SX64_F8V2: return go_staged(k_das_exact<64, 8, 2, 8, 8, 72, 0>, 8, p, sm, s);
    case V_SX16_F4V2W7: case V_SX16_F4V2W7_T8X14:
      return p.inside ? go_staged(k_das_exact<16, 4, 2, 7, 8, 64, kEarly | kInside>, 7, p, sm, s)
                      : go_staged(k_das_exact<16, 4, 2, 7, 8, 64, kEarly>, 7, p, sm, s);
    case V_SX16_F8V1W7: return go_staged(k_das_exact<16, 8, 1, 7, 8, 64, kEarly>, 7, p, sm, s);
    case V_SX16_F8V1W4: return go_staged(k_das_exact<16, 8, 1, 4, 8, 64, kEarly>, 4, p, sm, s);
    case V_SX8_F8V1W4: return go_staged(k_das_exact<8, 8, 1, 4, 8, 64, kEarly>, 4, p, sm, s);
    case V_SX16_F4V1W7: return go_staged(k_das_exact<16, 4, 1, 7, 8, 64, kEarly>, 7, p, sm, s);
    case V_SX8_F4V1W7: case V_SX8_F4V1W7_T8X14: return go_staged(k_das_exact<8, 4, 1, 7, 8, 64, kEarly>, 7, p, sm, s);
    default: return cudaErrorInvalidValue;
  }
}

// The kernels of a repacked ensemble (see mach_internal.h): the exact-frame shapes above, one
// launch per run of equal frame tiles.
cudaError_t launch_das_parts(const DasParams& p, Variant v, int tiles, cudaStream_t s) {
  DasParams q = p;
  const size_t sm = repacked_smem_bytes(v, p.rows_cap, p.T);
  auto go = [&](auto* kernel, int nwc) -> cudaError_t {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kStagedSmemCap));
    if (e != cudaSuccess) return e;
    const int64_t blocks = static_cast<int64_t>(p.tiles_x) * p.tiles_y * p.tiles_z;
    kernel<<<dim3(static_cast<unsigned>(blocks), static_cast<unsigned>(tiles)), (nwc + 1) * 32, sm, s>>>(q);
    return cudaGetLastError();
  };
  switch (v) {
    case V_SX32_F8V1W7T14E: case V_SX32_F8V1W7_T8X7E: return go(k_das_exact<32, 8, 1, 7, 8, 64, kEarly | kInside, true>, 7);
    case V_SX16_F8V1W7: return go(k_das_exact<16, 8, 1, 7, 8, 64, kEarly | kInside, true>, 7);
    case V_SX16_F8V1W4: return go(k_das_exact<16, 8, 1, 4, 8, 64, kEarly | kInside, true>, 4);
    case V_SX16_F4V1W7: return go(k_das_exact<16, 4, 1, 7, 8, 64, kEarly | kInside, true>, 7);
    case V_SX8_F8V1W4: return go(k_das_exact<8, 8, 1, 4, 8, 64, kEarly | kInside, true>, 4);
    case V_SX8_F4V1W7: return go(k_das_exact<8, 4, 1, 7, 8, 64, kEarly | kInside, true>, 7);
    default: return cudaErrorInvalidValue;
  }
}

cudaError_t launch_das_multi(const MultiArgs& a, Variant v, const int2* items, int n_items, cudaStream_t s) {
  size_t sm = 0;
  for (int k = 0; k < a.n; ++k) sm = std::max(sm, repacked_smem_bytes(v, a.p[k].rows_cap, a.p[k].T));
  auto go = [&](auto* kernel, int nwc) -> cudaError_t {
    const cudaError_t e =
        cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kStagedSmemCap));
    if (e != cudaSuccess) return e;
    kernel<<<static_cast<unsigned>(n_items), (nwc + 1) * 32, sm, s>>>(a, items);
    return cudaGetLastError();
  };
  switch (v) {
    case V_SX32_F8V1W7T14E: case V_SX32_F8V1W7_T8X7E: return go(k_das_exact_multi<32, 8, 1, 7, 8, 64, kEarly | kInside>, 7);
    case V_SX16_F8V1W7: return go(k_das_exact_multi<16, 8, 1, 7, 8, 64, kEarly | kInside>, 7);
    case V_SX16_F8V1W4: return go(k_das_exact_multi<16, 8, 1, 4, 8, 64, kEarly | kInside>, 4);
    case V_SX16_F4V1W7: return go(k_das_exact_multi<16, 4, 1, 7, 8, 64, kEarly | kInside>, 7);
    case V_SX8_F8V1W4: return go(k_das_exact_multi<8, 8, 1, 4, 8, 64, kEarly | kInside>, 4);
    case V_SX8_F4V1W7: return go(k_das_exact_multi<8, 4, 1, 7, 8, 64, kEarly | kInside>, 7);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mach
