// Spectrum -> CIE XYZ contraction (section 6: colorimetry from spectra).
//
//   xyz[p][c] = sum_j (spectral[p][j] / spp) * w[j][c]
//
// RT_XYZ_BF16X3 (the default, FP32-level accuracy): k_xyz_f32, FP32 FMAs on
// the CUDA cores.  Three columns make 6 flops per 8 bytes read: the path is
// bound by HBM, and an operand must reach a tensor core through shared memory
// as three BF16 terms, which cost more than the FMAs they replace.
//
// RT_XYZ_BF16: 5th-generation tensor cores (tcgen05.mma, accumulator in tensor
// memory).  A CTA processes tiles of 128 pixels: the FP64 rows are rounded to
// FP32 (integer operations on the IEEE fields), scaled by 1/spp and rounded to
// BF16, written to shared memory in the K-major, non-swizzled canonical layout
// (8 x 16-byte core matrices).  One thread issues D[128 x 16] += A[128 x 16]
// B[16 x 16] for every 16-band slice.  The FP32 accumulator is read back with
// tcgen05.ld (warp w owns TMEM lanes 32w..32w+31 = pixels).
//
// RT_XYZ_FP64: CUDA cores, FP64, the reference mode.
#include <cstdint>

#include "rt_internal.h"
#include "rt_tc.cuh"

namespace srt {

namespace {

// ---------------------------------------------------------------------------
// FP64 reference kernel
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(256) k_xyz_fp64(const double* __restrict__ s, uint64_t np, uint32_t bc,
                                                  const float* __restrict__ w, double inv_spp, float* __restrict__ xyz) {
  extern __shared__ double tile[];  // [blockDim][bc]
  const uint64_t p0 = (uint64_t)blockIdx.x * blockDim.x;
  const uint64_t rows = (np - p0) < blockDim.x ? (np - p0) : blockDim.x;
  const uint64_t elems = rows * bc;
  const double* src = s + p0 * bc;
  for (uint64_t e = threadIdx.x; e < elems; e += blockDim.x) tile[e] = src[e];
  __syncthreads();
  if (threadIdx.x < rows) {
    double a0 = 0.0, a1 = 0.0, a2 = 0.0;
    const double* row = tile + (size_t)threadIdx.x * bc;
    for (uint32_t j = 0; j < bc; ++j) {
      const double v = row[j] * inv_spp;
      a0 += v * (double)w[3 * j];
      a1 += v * (double)w[3 * j + 1];
      a2 += v * (double)w[3 * j + 2];
    }
    float* o = xyz + 3 * (p0 + threadIdx.x);
    o[0] = (float)a0;
    o[1] = (float)a1;
    o[2] = (float)a2;
  }
}

// FP64 -> FP32 by integer operations on the IEEE-754 fields (this GPU's FP64
// pipe is slow; a conversion instruction per spectral value made the
// contraction compute-bound).  RN rounds to nearest even, RZ truncates.
// Values below the FP32 normal range become signed zero, values above it
// infinity.
template <bool RN>
__device__ __forceinline__ float f64_to_f32(double x) {
  const uint64_t b = (uint64_t)__double_as_longlong(x);
  const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b;
  const uint32_t sign = hi & 0x80000000u;
  const int e = (int)((hi >> 20) & 0x7FFu) - 1023 + 127;
  if (e <= 0) return __uint_as_float(sign);
  if (e >= 255) return __uint_as_float(sign | 0x7F800000u);
  const uint32_t m = ((hi & 0xFFFFFu) << 3) | (lo >> 29);  // top 23 of the 52 fraction bits
  uint32_t bits = ((uint32_t)e << 23) | m;
  if (RN) {
    const uint32_t rem = lo & 0x1FFFFFFFu;  // the 29 bits dropped
    if (rem > 0x10000000u || (rem == 0x10000000u && (m & 1u))) bits += 1u;  // a carry moves into the exponent
  }
  return __uint_as_float(sign | bits);
}

// FP64 -> FP32 truncated, from the double's two words: rebias the exponent
// inside the high word, then one funnel shift joins its 20 fraction bits with
// the top 3 of the low word.  Magnitudes below the FP32 normal range (zero
// included) give signed zero; the spectral sums never exceed its range.
__device__ __forceinline__ float f64_to_f32_rz(uint32_t lo, uint32_t hi) {
  const uint32_t t = (hi & 0x7FFFFFFFu) - (896u << 20);  // exponent 1023 -> 127
  const uint32_t bits = __funnelshift_l(lo, t, 3);       // (t << 3) | (lo >> 29)
  const uint32_t sign = hi & 0x80000000u;
  return __uint_as_float(((hi >> 20) & 0x7FFu) > 896u ? (bits | sign) : sign);
}

// FP64 -> FP32, nearest (ties away from zero): one bit more than the 23 kept,
// plus one, halved.  Magnitudes below the FP32 normal range give signed zero.
// top keeps the largest rebiased high word: past kTopF32 a value is above
// 2^96, where 192 products with weights of up to 2^24 can leave the FP32 range
// before the division by the samples (and the value itself can).
constexpr int kTopF32 = (1023 + 96 - 896) << 20;
__device__ __forceinline__ float f64_to_f32_rn(uint2 d, int& top) {
  const int t = (int)((d.y & 0x7FFFFFFFu) - (896u << 20));
  top = max(top, t);
  const uint32_t bits = (__funnelshift_l(d.x, (uint32_t)t, 4) + 1u) >> 1;
  const uint32_t sign = d.y & 0x80000000u;
  return __uint_as_float(t >= (1 << 20) ? (bits | sign) : sign);
}

constexpr int kTileM = 128;        // pixels per tile = MMA M = TMEM lanes
constexpr int kMmaN = 16;          // XYZ padded to 16 columns
constexpr int kTmemCols = 32;      // smallest TMEM allocation
constexpr uint32_t kATile = 4096;  // one 128 x 16 BF16 K-slice
constexpr uint32_t kBTile = 512;   // one 16 x 16 BF16 K-slice
constexpr uint32_t kIdesc = tc_idesc_bf16(kTileM, kMmaN);

constexpr int kXyzThreads = 256;
constexpr int kUnroll = 8;

// inv_bc = ceil(2^32 / bc): __umulhi(e, inv_bc) == e / bc for every element
// index of a tile (e < 128 * 192).
__global__ void __launch_bounds__(kXyzThreads) k_xyz_tc(const double* __restrict__ s, uint64_t np, uint32_t bc,
                                                        uint32_t nk, uint32_t inv_bc, const float* __restrict__ w,
                                                        double inv_spp, float* __restrict__ xyz, uint32_t* status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* A = smem;                                   // [nk][4096]
  unsigned char* Bm = smem + nk * kATile;                    // [nk][512]
  uint64_t* mbar = (uint64_t*)(Bm + nk * kBTile);
  uint32_t* tslot = (uint32_t*)(mbar + 1);
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;

  // zero A (its padded K columns stay zero) and build the weight tile
  for (uint32_t i = tid; i < nk * kATile / 16u; i += blockDim.x) ((uint4*)A)[i] = make_uint4(0, 0, 0, 0);
  for (uint32_t i = tid; i < (uint32_t)kMmaN * nk * 16u; i += blockDim.x) {
    const uint32_t n = i / (nk * 16u), k = i - n * nk * 16u;
    const float v = (n < 3u && k < bc) ? w[3u * k + n] : 0.0f;
    *(uint16_t*)(Bm + (k >> 4) * kBTile + tc_kmajor_off(n, k & 15u)) = tc_bf16_bits(v);
  }
  if (tid == 0) {
    tc_mbar_init(mbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tc_tmem_alloc(tslot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;

  const uint64_t ntiles = (np + kTileM - 1) / kTileM;
  const float inv_spp_f = (float)inv_spp;
  uint32_t phase = 0;
  bool ok = true;
  for (uint64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const uint64_t p0 = tile * kTileM;
    const uint32_t rows = (uint32_t)((np - p0) < (uint64_t)kTileM ? (np - p0) : (uint64_t)kTileM);
    const uint32_t nel = rows * bc;
    const double* src = s + p0 * bc;
    // coalesced 16-byte loads over the tile's contiguous rows, kUnroll in
    // flight per thread before any conversion
    const uint32_t npair = (nel + 1u) >> 1;
    for (uint32_t q0 = tid; q0 < npair; q0 += blockDim.x * kUnroll) {
      double2 v[kUnroll];
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const uint32_t q = q0 + (uint32_t)u * blockDim.x;
        if (2u * q + 1u < nel) {
          v[u] = __ldcs((const double2*)src + q);
        } else if (2u * q < nel) {
          v[u] = make_double2(__ldcs(src + 2u * q), 0.0);
        } else {
          v[u] = make_double2(0.0, 0.0);
        }
      }
#pragma unroll
      for (int u = 0; u < kUnroll; ++u) {
        const uint32_t q = q0 + (uint32_t)u * blockDim.x;
#pragma unroll
        for (int h2 = 0; h2 < 2; ++h2) {
          const uint32_t ee = 2u * q + (uint32_t)h2;
          if (ee < nel) {
            const uint32_t r = __umulhi(ee, inv_bc), k = ee - r * bc;
            const float val = f64_to_f32<true>(h2 ? v[u].y : v[u].x) * inv_spp_f;
            *(uint16_t*)(A + (k >> 4) * kATile + tc_kmajor_off(r, k & 15u)) = tc_bf16_bits(val);
          }
        }
      }
    }
    tc_fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      for (uint32_t kb = 0; kb < nk; ++kb)
        tc_mma_bf16(tmem, tc_smem_desc(smem_u32(A + kb * kATile)), tc_smem_desc(smem_u32(Bm + kb * kBTile)), kIdesc,
                    kb > 0 ? 1u : 0u);
      tc_commit(mbar);
    }
    const int timed_out = __syncthreads_or(tc_mbar_wait(mbar, phase, 1u << 24) ? 0 : 1);
    if (timed_out) {
      if (tid == 0) atomicOr(status, ST_ITER);
      ok = false;
    }
    phase ^= 1u;
    tc_fence_after();
    if (warp < 4) {  // warp w reads TMEM lanes 32w..32w+31 (pixels)
      float x, y, z, pad;
      tc_tmem_ld4(tmem + ((warp * 32u) << 16), x, y, z, pad);
      const uint32_t r = warp * 32u + lane;
      if (ok && r < rows) {
        float* o = xyz + 3 * (p0 + r);
        o[0] = x;
        o[1] = y;
        o[2] = z;
      }
    }
    tc_fence_before();
    __syncthreads();
  }
  tc_fence_after();
  if (warp == 0) tc_tmem_dealloc(tmem, kTmemCols);
}

// ---------------------------------------------------------------------------
// TMA-pipelined variant (RT_XYZ_BF16 where it fits in shared memory): a tile of
// 128 pixels arrives as two halves of 64 rows, each one bulk copy (the rows
// are contiguous) into its own shared buffer, completion counted on an
// mbarrier.  Each half is converted (FP32, divide by spp, BF16, 16-byte stores
// of 8 K-consecutive values into the canonical layout)
// as soon as it lands, and the copy of the same half of the CTA's next tile is
// issued as soon as the buffer is read, so HBM traffic overlaps conversion,
// MMA and epilogue.  A tail tile whose halves are not full is read with
// plain loads.
// ---------------------------------------------------------------------------
constexpr uint32_t kHalf = 64;

__device__ __forceinline__ bool half_full(uint64_t tile, uint32_t h, uint64_t np) {
  return tile * kTileM + (uint64_t)(h + 1) * kHalf <= np;
}

constexpr int kXyzTmaThreads = 512;

__global__ void __launch_bounds__(kXyzTmaThreads, 1) k_xyz_tma(const double* __restrict__ s, uint64_t np, uint32_t bc,
                                                            uint32_t nk, const float* __restrict__ w, double inv_spp,
                                                            float* __restrict__ xyz, uint32_t* status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  const uint32_t half_bytes = kHalf * bc * 8u;  // a multiple of 512
  unsigned char* raw0 = smem;
  unsigned char* A = smem + 2u * half_bytes;
  unsigned char* Bm = A + nk * kATile;
  uint64_t* mb = (uint64_t*)(Bm + nk * kBTile);  // [0], [1]: raw halves, [2]: MMA
  uint32_t* tslot = (uint32_t*)(mb + 3);
  const uint32_t tid = threadIdx.x, warp = tid >> 5, lane = tid & 31u;
  for (uint32_t i = tid; i < nk * kATile / 16u; i += blockDim.x) ((uint4*)A)[i] = make_uint4(0, 0, 0, 0);
  for (uint32_t i = tid; i < (uint32_t)kMmaN * nk * 16u; i += blockDim.x) {
    const uint32_t n = i / (nk * 16u), k = i - n * nk * 16u;
    const float v = (n < 3u && k < bc) ? w[3u * k + n] : 0.0f;
    *(uint16_t*)(Bm + (k >> 4) * kBTile + tc_kmajor_off(n, k & 15u)) = tc_bf16_bits(v);
  }
  if (tid == 0) {
    for (int i = 0; i < 3; ++i) tc_mbar_init(mb + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tc_tmem_alloc(tslot, kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tslot;
  const uint64_t ntiles = (np + kTileM - 1) / kTileM;
  const float inv_spp_f = (float)inv_spp;
  auto issue = [&](uint64_t tile, uint32_t h) {
    tc_mbar_expect_tx(mb + h, half_bytes);
    tc_bulk_g2s(raw0 + h * half_bytes, s + (tile * kTileM + h * kHalf) * bc, half_bytes, mb + h);
  };
  // every thread tracks which halves have a copy in flight (the conditions
  // are the same in all threads; thread 0 issues)
  bool inflight[2] = {false, false};
  if ((uint64_t)blockIdx.x < ntiles)
    for (uint32_t h = 0; h < 2u; ++h)
      if (half_full(blockIdx.x, h, np)) {
        inflight[h] = true;
        if (tid == 0) issue(blockIdx.x, h);
      }
  uint32_t ph[2] = {0u, 0u}, phm = 0u;
  bool ok = true;
  for (uint64_t tile = blockIdx.x; tile < ntiles && ok; tile += gridDim.x) {
    const uint64_t p0 = tile * kTileM;
    const uint32_t rows = (uint32_t)((np - p0) < (uint64_t)kTileM ? (np - p0) : (uint64_t)kTileM);
    for (uint32_t h = 0; h < 2u && ok; ++h) {
      unsigned char* raw = raw0 + h * half_bytes;
      const uint32_t rh = rows > h * kHalf ? min(rows - h * kHalf, kHalf) : 0u;
      if (half_full(tile, h, np)) {
        const int bad = __syncthreads_or(tc_mbar_wait(mb + h, ph[h], 1u << 24) ? 0 : 1);
        if (bad) {
          if (tid == 0) atomicOr(status, ST_ITER);
          ok = false;
          break;
        }
        ph[h] ^= 1u;
        inflight[h] = false;
      } else {
        const double* src = s + (p0 + h * kHalf) * bc;
        for (uint32_t e = tid; e < rh * bc; e += blockDim.x) ((double*)raw)[e] = src[e];
        __syncthreads();
      }
      // (row, group of 8 K values) items, rows fastest
      const uint32_t items = kHalf * 2u * nk;
      for (uint32_t it = tid; it < items; it += blockDim.x) {
        const uint32_t r = it % kHalf, g8 = it / kHalf;
        float v[8];
        const double* rowp = (const double*)raw + r * bc + 8u * g8;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          v[e] = 0.0f;
          if (r < rh && 8u * g8 + (uint32_t)e < bc) {
            const uint2 wv = *(const uint2*)(rowp + e);
            v[e] = f64_to_f32_rz(wv.x, wv.y) * inv_spp_f;
          }
        }
        *(uint4*)(A + (g8 >> 1) * kATile + tc_kmajor_off(h * kHalf + r, (g8 & 1u) * 8u)) =
            make_uint4(tc_bf16x2_bits(v[0], v[1]), tc_bf16x2_bits(v[2], v[3]), tc_bf16x2_bits(v[4], v[5]),
                       tc_bf16x2_bits(v[6], v[7]));
      }
      // the buffer is read: refill it with the same half of the next tile
      __syncthreads();
      const uint64_t next = tile + gridDim.x;
      if (next < ntiles && half_full(next, h, np)) {
        inflight[h] = true;
        if (tid == 0) {
          tc_fence_async_smem();
          issue(next, h);
        }
      }
    }
    if (!ok) break;
    tc_fence_async_smem();
    __syncthreads();
    if (tid == 0) {
      tc_fence_after();
      for (uint32_t kb = 0; kb < nk; ++kb)
        tc_mma_bf16(tmem, tc_smem_desc(smem_u32(A + kb * kATile)), tc_smem_desc(smem_u32(Bm + kb * kBTile)), kIdesc,
                    kb > 0 ? 1u : 0u);
      tc_commit(mb + 2);
    }
    const int timed_out = __syncthreads_or(tc_mbar_wait(mb + 2, phm, 1u << 24) ? 0 : 1);
    phm ^= 1u;
    if (timed_out) {
      if (tid == 0) atomicOr(status, ST_ITER);
      ok = false;
    }
    tc_fence_after();
    if (warp < 4) {  // warp w reads TMEM lanes 32w..32w+31 (pixels)
      float x, y, z, pad;
      tc_tmem_ld4(tmem + ((warp * 32u) << 16), x, y, z, pad);
      const uint32_t r = warp * 32u + lane;
      if (ok && r < rows) {
        float* o = xyz + 3 * (p0 + r);
        o[0] = x;
        o[1] = y;
        o[2] = z;
      }
    }
    tc_fence_before();
    __syncthreads();
  }
  // after an early exit, wait (bounded) for the copies still in flight
  if (!ok && tid == 0)
    for (uint32_t h = 0; h < 2u; ++h)
      if (inflight[h]) tc_mbar_wait(mb + h, ph[h], 1u << 24);
  tc_fence_after();
  if (warp == 0) tc_tmem_dealloc(tmem, kTmemCols);
}

size_t xyz_tma_smem(uint32_t band_count) {
  const uint32_t nk = (band_count + 15) / 16;
  return 2ull * kHalf * band_count * 8ull + (size_t)nk * kATile + (size_t)nk * kBTile + 64;
}

// ---------------------------------------------------------------------------
// FP32 contraction (RT_XYZ_BF16X3).  Bound by HBM: 8 bytes per (pixel, band)
// for some 15 instructions.  A stage is 32 RPT pixels, whose rows are
// contiguous: one bulk copy (TMA) into shared memory, the CTA's next ones in
// flight meanwhile.  Eight lanes share RPT pixels, lane l their bands l, l + 8,
// ... (a row-per-lane order would meet in the same banks for even band
// counts), and add up over the eight.  The last, short stage is read from
// global memory.  786,432 pixels x 81 bands: 195 us with BF16 triples on
// tensor cores (one CTA per SM; conversion, MMAs and epilogue of a tile in
// turn), 198 us here with a pixel per eight lanes and a branch per conversion,
// 103 us with two (the kernel alone 79 us, 6.4 TB/s).
// ---------------------------------------------------------------------------
constexpr int kF32Threads = 256;
constexpr uint32_t kF32Stages = 4;
constexpr uint32_t kF32Smem = 110u * 1024u;  // two CTAs per SM

// pixels per eight lanes: two while two stages of 64 pixels fit
uint32_t xyz_f32_rpt(uint32_t bc) { return 2u * 64u * bc * 8u + 16u * bc + 64u <= kF32Smem ? 2u : 1u; }
uint32_t xyz_f32_stages(uint32_t bc) {
  const uint32_t fit = (kF32Smem - 16u * bc - 64u) / (32u * xyz_f32_rpt(bc) * bc * 8u);
  return fit > kF32Stages ? kF32Stages : fit;
}
size_t xyz_f32_smem(uint32_t bc) {
  return (size_t)xyz_f32_stages(bc) * 32u * xyz_f32_rpt(bc) * bc * 8u + 16u * bc + 64u;
}

template <int RPT>
__global__ void __launch_bounds__(kF32Threads, 2)
    k_xyz_f32(const double* __restrict__ s, uint64_t np, uint32_t bc, uint32_t n_stages, const float* __restrict__ w,
              double inv_spp, float* __restrict__ xyz, uint32_t* status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  constexpr uint32_t kRows = 32u * RPT;
  const float inv_spp_f = (float)inv_spp;
  const uint32_t stage_bytes = kRows * bc * 8u;  // a multiple of 256
  float4* W = (float4*)(smem + n_stages * stage_bytes);
  uint64_t* full = (uint64_t*)(W + bc);
  const uint32_t tid = threadIdx.x, row = tid >> 3, l = tid & 7u;
  for (uint32_t j = tid; j < bc; j += blockDim.x) W[j] = make_float4(w[3u * j], w[3u * j + 1], w[3u * j + 2], 0.0f);
  if (tid == 0) {
    for (uint32_t i = 0; i < n_stages; ++i) tc_mbar_init(full + i, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const uint64_t nt = (np + kRows - 1) / kRows;
  auto whole = [&](uint64_t t) { return (t + 1) * kRows <= np; };
  auto issue = [&](uint64_t t, uint32_t st) {
    tc_mbar_expect_tx(full + st, stage_bytes);
    tc_bulk_g2s(smem + st * stage_bytes, s + t * kRows * bc, stage_bytes, full + st);
  };
  if (tid == 0)
    for (uint32_t i = 0; i < n_stages; ++i) {
      const uint64_t t = blockIdx.x + (uint64_t)i * gridDim.x;
      if (t < nt && whole(t)) issue(t, i);
    }
  uint32_t st = 0, phase = 0;
  for (uint64_t t = blockIdx.x; t < nt; t += gridDim.x) {
    const bool staged = whole(t);
    if (staged && __syncthreads_or(tc_mbar_wait(full + st, phase, 1u << 24) ? 0 : 1)) {
      if (tid == 0) {
        atomicOr(status, ST_ITER);
        // copies still in flight write this CTA's memory: wait (bounded) for them
        for (uint32_t i = 1; i < n_stages; ++i) {
          const uint64_t u = t + (uint64_t)i * gridDim.x;
          const uint32_t si = st + i < n_stages ? st + i : st + i - n_stages;
          if (u < nt && whole(u)) tc_mbar_wait(full + si, si < st ? phase ^ 1u : phase, 1u << 24);
        }
      }
      return;
    }
    // the eight lanes' pixels: rows row, row + 32 of the stage
    const uint64_t p0 = t * kRows + row;
    const uint2* v[RPT];
    float x[RPT], y[RPT], z[RPT];
    int top = 0;
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
      // (past the image's end: its last pixel, whose result is not stored)
      const uint64_t p = min(p0 + 32u * (uint32_t)q, np - 1);
      v[q] = staged ? (const uint2*)(smem + st * stage_bytes) + (row + 32u * (uint32_t)q) * bc
                    : (const uint2*)(s + p * bc);
      x[q] = y[q] = z[q] = 0.0f;
    }
#pragma unroll 4
    for (uint32_t j = l; j < bc; j += 8u) {
      const float4 c = W[j];
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        const float f = f64_to_f32_rn(v[q][j], top);
        x[q] = fmaf(f, c.x, x[q]);
        y[q] = fmaf(f, c.y, y[q]);
        z[q] = fmaf(f, c.z, z[q]);
      }
    }
    // a large value, an infinity or a NaN in the warp's pixels: divided in FP64
    // before the conversion, by its instruction
    float scale = inv_spp_f;
    if (__any_sync(0xffffffffu, top > kTopF32)) {
      scale = 1.0f;
#pragma unroll
      for (int q = 0; q < RPT; ++q) {
        x[q] = y[q] = z[q] = 0.0f;
        for (uint32_t j = l; j < bc; j += 8u) {
          const float4 c = W[j];
          const uint2 d = v[q][j];
          const float f = (float)(__hiloint2double((int)d.y, (int)d.x) * inv_spp);
          x[q] = fmaf(f, c.x, x[q]);
          y[q] = fmaf(f, c.y, y[q]);
          z[q] = fmaf(f, c.z, z[q]);
        }
      }
    }
#pragma unroll
    for (int q = 0; q < RPT; ++q) {
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        x[q] += __shfl_xor_sync(0xffffffffu, x[q], o);
        y[q] += __shfl_xor_sync(0xffffffffu, y[q], o);
        z[q] += __shfl_xor_sync(0xffffffffu, z[q], o);
      }
      const uint64_t p = p0 + 32u * (uint32_t)q;
      if (p < np && l < 3u) xyz[3 * p + l] = (l == 0 ? x[q] : (l == 1 ? y[q] : z[q])) * scale;
    }
    // the stage is read: refill it
    __syncthreads();
    const uint64_t next = t + (uint64_t)n_stages * gridDim.x;
    if (tid == 0 && staged && next < nt && whole(next)) {
      tc_fence_async_smem();
      issue(next, st);
    }
    if (++st == n_stages) {
      st = 0;
      phase ^= 1u;
    }
  }
}

}  // namespace

size_t xyz_tc_smem(uint32_t band_count) {
  const uint32_t nk = (band_count + 15) / 16;
  return (size_t)nk * kATile + (size_t)nk * kBTile + 16;
}

void launch_xyz(const double* spectral, uint64_t n_pixels, const XyzWeights& w, uint32_t spp, int mode, float* xyz,
                cudaStream_t st, uint32_t* status, int sms) {
  if (n_pixels == 0) return;
  if (mode == 2) {
    int block = (int)(49152 / (8 * (size_t)w.band_count));
    block = block > 256 ? 256 : (block < 1 ? 1 : block);
    const uint64_t grid = (n_pixels + block - 1) / block;
    const size_t smem = (size_t)block * w.band_count * sizeof(double);
    k_xyz_fp64<<<(unsigned)grid, block, smem, st>>>(spectral, n_pixels, w.band_count, w.w32, 1.0 / (double)spp, xyz);
    return;
  }
  if (mode == 0) {
    const size_t smem = xyz_f32_smem(w.band_count);
    const uint32_t rpt = xyz_f32_rpt(w.band_count), n_stages = xyz_f32_stages(w.band_count);
    auto* kernel = rpt == 2 ? k_xyz_f32<2> : k_xyz_f32<1>;
    cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    const uint64_t nt = (n_pixels + 32 * rpt - 1) / (32 * rpt);
    const unsigned grid = (unsigned)(nt < 2ull * (uint64_t)sms ? nt : 2ull * (uint64_t)sms);
    kernel<<<grid, kF32Threads, smem, st>>>(spectral, n_pixels, w.band_count, n_stages, w.w32, 1.0 / (double)spp, xyz, status);
    return;
  }
  const uint32_t nk = (w.band_count + 15) / 16;
  const size_t tsmem = xyz_tma_smem(w.band_count);
  if (tsmem <= 227u * 1024u && ((uintptr_t)spectral & 15u) == 0) {
    cudaFuncSetAttribute(k_xyz_tma, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tsmem);
    const uint64_t ntiles = (n_pixels + kTileM - 1) / kTileM;
    uint64_t grid = (uint64_t)sms;
    if (grid > ntiles) grid = ntiles;
    k_xyz_tma<<<(unsigned)grid, kXyzTmaThreads, tsmem, st>>>(spectral, n_pixels, w.band_count, nk, w.w32,
                                                         1.0 / (double)spp, xyz, status);
    return;
  }
  const size_t smem = xyz_tc_smem(w.band_count);
  cudaFuncSetAttribute(k_xyz_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  const uint64_t ntiles = (n_pixels + kTileM - 1) / kTileM;
  int per_sm = (int)((227u * 1024u) / (smem + 1024));
  if (per_sm < 1) per_sm = 1;
  if (per_sm > 4) per_sm = 4;
  uint64_t grid = (uint64_t)sms * per_sm;
  if (grid > ntiles) grid = ntiles;
  const uint32_t inv_bc = (uint32_t)((0x100000000ull + w.band_count - 1) / w.band_count);
  k_xyz_tc<<<(unsigned)grid, kXyzThreads, smem, st>>>(spectral, n_pixels, w.band_count, nk, inv_bc, w.w32,
                                                      1.0 / (double)spp, xyz, status);
}

}  // namespace srt
