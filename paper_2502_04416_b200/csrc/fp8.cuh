// FP8 weight-only quantisation of the expert weights (the paper, Section 6, only states that the
// restructured FFN composes with post-training quantisation; the format is this library's choice):
// OCP E4M3 codes (bias 7, 3 mantissa bits, subnormals, largest value 448) with one power-of-two
// scale per output channel.  Because the scale is a power of two, w / scale is exact, the code
// is the round-to-nearest-even encoding of an exactly known number, and code * scale is exactly
// representable in bf16.
#pragma once

#include "common.cuh"

namespace cmoe {

// Two floats -> two E4M3 codes (round to nearest even, saturating): `lo` in bits 0..7.
__device__ __forceinline__ uint16_t f32x2_to_e4m3x2(float lo, float hi) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(hi), "f"(lo));
  return r;
}
// Two E4M3 codes -> two floats (exact).
__device__ __forceinline__ float2 e4m3x2_to_f32x2(uint16_t v) {
  uint32_t h2;
  asm("cvt.rn.f16x2.e4m3x2 %0, %1;" : "=r"(h2) : "h"(v));
  return __half22float2(*reinterpret_cast<const __half2*>(&h2));
}

// Smallest e with amax * 2^-e <= 448 = 0.875 * 2^9 (0 for amax == 0).
__device__ __forceinline__ int pow2_scale_exponent(float amax) {
  if (!(amax > 0.0f)) return 0;
  int p;
  const float f = frexpf(amax, &p);                       // amax = f * 2^p, f in [0.5, 1)
  return f <= 0.875f ? p - 9 : p - 8;
}

// One block per row of a bf16 matrix [rows, cols] (leading dimension ld elements): the row's
// scale 2^e, its E4M3 codes, and (when deq != nullptr, which may alias w) the dequantised row.
__global__ void __launch_bounds__(256)
quantise_rows_fp8_kernel(const bf16* w, int rows, int cols, long long ld, uint8_t* __restrict__ codes,
                         long long ld_codes, float* __restrict__ scale, bf16* deq) {
  const int r = blockIdx.x;
  if (r >= rows) return;
  const bf16* src = w + (size_t)r * ld;
  __shared__ float red[8];
  __shared__ float sh_amax;
  float amax = 0.0f;
  for (int c = threadIdx.x; c < cols; c += 256) {
    const float v = fabsf(__bfloat162float(src[c]));
    amax = (v > amax) ? v : amax;                          // NaN weights never raise the maximum
  }
  amax = warp_max(amax);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
  __syncthreads();
  if (threadIdx.x == 0) {
    float m = red[0];
    for (int i = 1; i < 8; ++i) m = fmaxf(m, red[i]);
    sh_amax = m;
  }
  __syncthreads();
  const int e = pow2_scale_exponent(sh_amax);
  if (threadIdx.x == 0) scale[r] = ldexpf(1.0f, e);
  uint8_t* dst = codes + (size_t)r * ld_codes;
  bf16* dq = deq ? deq + (size_t)r * ld : nullptr;
  for (int c = 2 * threadIdx.x; c < cols; c += 512) {
    const float v0 = ldexpf(__bfloat162float(src[c]), -e);
    const bool two = c + 1 < cols;
    const float v1 = two ? ldexpf(__bfloat162float(src[c + 1]), -e) : 0.0f;
    const uint16_t q = f32x2_to_e4m3x2(v0, v1);
    dst[c] = (uint8_t)(q & 0xFF);
    if (two) dst[c + 1] = (uint8_t)(q >> 8);
    if (dq) {
      const float2 back = e4m3x2_to_f32x2(q);
      dq[c] = __float2bfloat16_rn(ldexpf(back.x, e));
      if (two) dq[c + 1] = __float2bfloat16_rn(ldexpf(back.y, e));
    }
  }
}

constexpr int kSplitThreads = 256;         // threads per token row of the split
// Threads per (token row, expert) in split_groups_e4m3_kernel.  More of them leave the down kernel, which comes in under the split, less
// room on the SMs: 7B-shaped FP8 layer, 48 rows, 48.1 us with 256, 47.1 with 128 (46.8 with one scale and block per row).
constexpr int kSplitGroupThreads = 128;

// Splits bf16 rows into two E4M3 planes for the FP8 tensor-core path: with the row's power-of-two
// scale 2^e (largest magnitude brought to at most 448), hi = E4M3(v / 2^e) and lo = E4M3(16 (v / 2^e - hi)).
// A bf16 value has 8 significant bits, hi keeps the top 4 and the remainder is a multiple of the
// value's last place not above 8 of them, so lo holds it exactly unless it falls below E4M3's range
// (values under 2^-13 of the row's maximum): v = (hi + lo / 16) 2^e.  One block per row.
template <int THREADS>
__device__ __forceinline__ void split_row_e4m3(const bf16* __restrict__ row, int cols, uint8_t* __restrict__ h,
                                               uint8_t* __restrict__ l, float* __restrict__ scale_out) {
  constexpr int kKeep = 6;                   // chunks of 8 per thread held between the two passes
  __shared__ float red[THREADS / 32];
  uint4 raw[kKeep];
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    const int c = 8 * (threadIdx.x + i * THREADS);
    raw[i] = c < cols ? __ldcg(reinterpret_cast<const uint4*>(row + c)) : make_uint4(0u, 0u, 0u, 0u);
  }
  float amax = 0.0f;
  auto unpack = [](const uint4& r, float (&v)[8]) {
    const uint32_t w[4] = {r.x, r.y, r.z, r.w};
#pragma unroll
    for (int i = 0; i < 4; ++i) { v[2 * i] = __uint_as_float(w[i] << 16); v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u); }
  };
  auto take_max = [&](const uint4& r) {
    float v[8];
    unpack(r, v);
#pragma unroll
    for (int q = 0; q < 8; ++q) { const float a = fabsf(v[q]); amax = (a > amax) ? a : amax; }
  };
#pragma unroll
  for (int i = 0; i < kKeep; ++i) take_max(raw[i]);
#pragma unroll 1
  for (int c = 8 * (threadIdx.x + kKeep * THREADS); c < cols; c += 8 * THREADS)
    take_max(__ldcg(reinterpret_cast<const uint4*>(row + c)));
  amax = warp_max(amax);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = amax;
  __syncthreads();
#pragma unroll
  for (int i = 0; i < THREADS / 32; ++i) amax = fmaxf(amax, red[i]);
  const int e = pow2_scale_exponent(amax);
  if (threadIdx.x == 0) *scale_out = ldexpf(1.0f, e);
  // 2^-e as two factors (2^-e itself may be out of range): every product is exact or far below the codes' range
  const float f0 = ldexpf(1.0f, -(e / 2)), f1 = ldexpf(1.0f, -(e - e / 2));
  auto convert = [&](const uint4& r, int c) {
    float v[8];
    unpack(r, v);
    uint32_t hw[2], lw[2];
#pragma unroll
    for (int q = 0; q < 8; q += 2) {
      const float v0 = v[q] * f0 * f1, v1 = v[q + 1] * f0 * f1;
      const uint16_t hq = f32x2_to_e4m3x2(v0, v1);
      const float2 back = e4m3x2_to_f32x2(hq);
      const uint16_t lq = f32x2_to_e4m3x2((v0 - back.x) * 16.0f, (v1 - back.y) * 16.0f);
      hw[q >> 2] = (q & 2) ? (hw[q >> 2] | ((uint32_t)hq << 16)) : (uint32_t)hq;
      lw[q >> 2] = (q & 2) ? (lw[q >> 2] | ((uint32_t)lq << 16)) : (uint32_t)lq;
    }
    *reinterpret_cast<uint2*>(h + c) = make_uint2(hw[0], hw[1]);
    *reinterpret_cast<uint2*>(l + c) = make_uint2(lw[0], lw[1]);
  };
#pragma unroll
  for (int i = 0; i < kKeep; ++i) {
    const int c = 8 * (threadIdx.x + i * THREADS);
    if (c < cols) convert(raw[i], c);
  }
#pragma unroll 1
  for (int c = 8 * (threadIdx.x + kKeep * THREADS); c < cols; c += 8 * THREADS)
    convert(__ldcg(reinterpret_cast<const uint4*>(row + c)), c);
}

// One segment of rows: src [rows, cols] bf16 (leading dimension ld) -> planes [2][plane_rows][cols], scales [rows].
struct SplitSegment {
  const bf16* src;
  int rows, cols;
  long long ld;
  uint8_t* planes;
  long long plane_rows;
  float* scale;
};

// Blocks 0 .. a.rows-1 split the rows of segment a, the next b.rows blocks those of segment b (b.rows may be 0).
__global__ void __launch_bounds__(kSplitThreads) split_rows_e4m3_kernel(const SplitSegment a, const SplitSegment b) {
  grid_dep_wait();
  grid_dep_trigger();
  int r = blockIdx.x;
  const SplitSegment& sg = r < a.rows ? a : b;
  if (r >= a.rows) r -= a.rows;
  if (r >= sg.rows) return;
  uint8_t* hi = sg.planes + (size_t)r * sg.cols;
  split_row_e4m3<kSplitThreads>(sg.src + (size_t)r * sg.ld, sg.cols, hi, hi + (size_t)sg.plane_rows * sg.cols, sg.scale + r);
}

// The same for rows that hold the activations of several experts side by side: the shared experts' columns, then m per routed
// expert.  Every (row, expert) gets a scale of its own, so that an expert with small activations keeps its precision beside one with
// large ones.  Block (row, expert).  Columns of experts without rows hold what an earlier forward left; nothing reads their planes.
struct SplitGroups {
  const bf16* src;             // [rows][ld]
  uint8_t* planes;             // [2][plane_rows][ld]
  float* scale;                // [1 + experts][plane_rows]
  int shared_w, m;
  long long ld, plane_rows;
};
__global__ void __launch_bounds__(kSplitGroupThreads) split_groups_e4m3_kernel(const SplitGroups p) {
  grid_dep_wait();
  grid_dep_trigger();
  const int r = blockIdx.x, g = blockIdx.y, cols = g == 0 ? p.shared_w : p.m;
  if (cols == 0) return;
  const size_t at = (size_t)r * p.ld + (g == 0 ? 0 : p.shared_w + (size_t)(g - 1) * p.m);
  split_row_e4m3<kSplitGroupThreads>(p.src + at, cols, p.planes + at, p.planes + (size_t)p.plane_rows * p.ld + at,
                                     p.scale + (size_t)g * p.plane_rows + r);
}

}  // namespace cmoe
