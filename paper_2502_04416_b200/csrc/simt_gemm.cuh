// Plain SIMT grouped expert GEMMs (fp32 FMA, fp32 accumulate).  They serve the
// fp32 storage type and every shape the tensor-core path does not take, and give
// a second, structurally different implementation to check the tensor path against.
//
//   GEMM-1: H[r, n] = Swish(sum_k A[r,k] Wg[n,k]) * (sum_k A[r,k] Wu[n,k])   (Eq. ori_ffn_method)
//   GEMM-2: Y[r, c] = sum_n H[r,n] Wd[c,n]
// per group g (one shared expert per outer expert, then every routed expert), on the
// group's rows [row0, row0+count) of its row space.
#pragma once

#include "common.cuh"

namespace cmoe {

constexpr int kSimtTile = 64;
constexpr int kSimtBK = 32;
// Small tiles for grids that would leave most SMs idle: 16 rows x 32 columns, 128 threads with 2 x 2 outputs each.
// With the row router, the mask permutation and chained launches: fp32 forward of 64 rows, d = 256, 8 x 128 neurons 69.5 ->
// 25.5 us (a 64 x 64 tile kept 28 SMs busy for 16 dependent load-compute steps per GEMM).
constexpr int kSimtSmallM = 16, kSimtSmallN = 32, kSimtSmallThreads = 128;

template <typename T>
__device__ __forceinline__ void load_seg(const T* row_ptr, int k, int K, bool vec, float (&v)[8]) {
  if (row_ptr == nullptr) {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = 0.0f;
  } else if (vec && k + 8 <= K) {
    load8(row_ptr + k, v);
  } else {
#pragma unroll
    for (int q = 0; q < 8; ++q) v[q] = (k + q < K) ? to_float(__ldcg(row_ptr + k + q)) : 0.0f;
  }
}

// One 64x64 tile of C = A B^T (and, if DUAL, of A B2^T) into acc / acc2.
// A: M x K (lda), B/B2: N x K (ldb); (m0, n0) tile origin.  256 threads.
template <typename T, bool DUAL>
__device__ __forceinline__ void simt_tile(const T* __restrict__ A, int lda, int M, const T* __restrict__ B,
                                          const T* __restrict__ B2, int ldb, int N, int K, int m0, int n0,
                                          bool vec_a, bool vec_b, float (&acc)[4][4], float (&acc2)[4][4]) {
  __shared__ float As[kSimtBK][kSimtTile + 1];
  __shared__ float Bs[kSimtBK][kSimtTile + 1];
  __shared__ float Bs2[DUAL ? kSimtBK : 1][kSimtTile + 1];
  const int tid = threadIdx.x;
  const int lrow = tid >> 2, kseg = (tid & 3) * 8;
  const int ty = tid >> 4, tx = tid & 15;
  const T* a_row = (m0 + lrow < M) ? A + (size_t)(m0 + lrow) * lda : nullptr;
  const T* b_row = (n0 + lrow < N) ? B + (size_t)(n0 + lrow) * ldb : nullptr;
  const T* b2_row = (DUAL && n0 + lrow < N) ? B2 + (size_t)(n0 + lrow) * ldb : nullptr;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) { acc[i][j] = 0.0f; acc2[i][j] = 0.0f; }

  for (int k0 = 0; k0 < K; k0 += kSimtBK) {
    float va[8], vb[8], vb2[8];
    load_seg(a_row, k0 + kseg, K, vec_a, va);
    load_seg(b_row, k0 + kseg, K, vec_b, vb);
    if (DUAL) load_seg(b2_row, k0 + kseg, K, vec_b, vb2);
#pragma unroll
    for (int q = 0; q < 8; ++q) {
      As[kseg + q][lrow] = va[q];
      Bs[kseg + q][lrow] = vb[q];
      if (DUAL) Bs2[kseg + q][lrow] = vb2[q];
    }
    __syncthreads();
#pragma unroll 8
    for (int kk = 0; kk < kSimtBK; ++kk) {
      float a[4], b[4], b2[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty * 4 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        b[j] = Bs[kk][tx * 4 + j];
        b2[j] = DUAL ? Bs2[kk][tx * 4 + j] : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
          if (DUAL) acc2[i][j] = fmaf(a[i], b2[j], acc2[i][j]);
        }
    }
    __syncthreads();
  }
}

__device__ __forceinline__ float4 load4f(const float* p) {
  const uint4 r = ld_dep16(p);
  return make_float4(__uint_as_float(r.x), __uint_as_float(r.y), __uint_as_float(r.z), __uint_as_float(r.w));
}
__device__ __forceinline__ float4 load4f(const bf16* p) {
  uint2 r;
  asm volatile("ld.global.v2.u32 {%0, %1}, [%2];" : "=r"(r.x), "=r"(r.y) : "l"(p));
  return make_float4(__uint_as_float(r.x << 16), __uint_as_float(r.x & 0xffff0000u), __uint_as_float(r.y << 16),
                     __uint_as_float(r.y & 0xffff0000u));
}
// Four k values of a row (null: zeros) from k on, zeros past K.
template <typename T>
__device__ __forceinline__ float4 load_quad(const T* row_ptr, int k, int K, bool vec) {
  if (row_ptr == nullptr) return make_float4(0.f, 0.f, 0.f, 0.f);
  if (vec && k + 4 <= K) return load4f(row_ptr + k);
  float v[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) v[q] = k + q < K ? to_float(__ldcg(row_ptr + k + q)) : 0.0f;
  return make_float4(v[0], v[1], v[2], v[3]);
}

// One 16 x 32 tile of A B^T (DUAL: and of A B2^T): rows 2 ty, 2 ty + 1 and columns tx, tx + 16 per thread.  a_rows(i): row
// i of A or null.  Bound by latency and by issue: k quads are read from shared memory 16 bytes at a time (row-major, so
// six reads feed 32 multiply-adds), and the next k step's global loads are in flight during a step.  Sums run over k in
// ascending order, as in simt_tile.
template <typename T, bool DUAL, typename ARows>
__device__ __forceinline__ void simt_tile_small(ARows a_rows, const T* __restrict__ B, const T* __restrict__ B2, int ldb, int N,
                                                int K, int n0, bool vec_a, bool vec_b, float (&acc)[2][2], float (&acc2)[2][2]) {
  constexpr int kLd = kSimtBK + 4, kNB = DUAL ? 2 : 1;
  __shared__ __align__(16) float As[2][kSimtSmallM][kLd];
  __shared__ __align__(16) float Bs[2][kNB][kSimtSmallN][kLd];
  const int tid = threadIdx.x, lrow = tid >> 3, kq = (tid & 7) * 4;         // loads: 16 rows x 8 quads per pass
  const int ty = tid >> 4, tx = tid & 15;
  const T* a_row = a_rows(lrow);
  const T* b_row[kNB][2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int n = n0 + lrow + 16 * h;
    b_row[0][h] = n < N ? B + (size_t)n * ldb : nullptr;
    if (DUAL) b_row[kNB - 1][h] = n < N ? B2 + (size_t)n * ldb : nullptr;
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) { acc[i][j] = 0.0f; acc2[i][j] = 0.0f; }
  float4 va, vb[kNB][2];
  auto fetch = [&](int k0) {
    va = load_quad(a_row, k0 + kq, K, vec_a);
#pragma unroll
    for (int b = 0; b < kNB; ++b)
#pragma unroll
      for (int h = 0; h < 2; ++h) vb[b][h] = load_quad(b_row[b][h], k0 + kq, K, vec_b);
  };
  fetch(0);
  int buf = 0;
#pragma unroll 1
  for (int k0 = 0; k0 < K; k0 += kSimtBK, buf ^= 1) {
    *reinterpret_cast<float4*>(&As[buf][lrow][kq]) = va;
#pragma unroll
    for (int b = 0; b < kNB; ++b)
#pragma unroll
      for (int h = 0; h < 2; ++h) *reinterpret_cast<float4*>(&Bs[buf][b][lrow + 16 * h][kq]) = vb[b][h];
    __syncthreads();                                  // the other buffer is free: its readers passed this barrier's predecessor
    if (k0 + kSimtBK < K) fetch(k0 + kSimtBK);
#pragma unroll
    for (int k = 0; k < kSimtBK; k += 4) {
      float4 a[2], b[kNB][2];
#pragma unroll
      for (int i = 0; i < 2; ++i) a[i] = *reinterpret_cast<const float4*>(&As[buf][2 * ty + i][k]);
#pragma unroll
      for (int q = 0; q < kNB; ++q)
#pragma unroll
        for (int j = 0; j < 2; ++j) b[q][j] = *reinterpret_cast<const float4*>(&Bs[buf][q][tx + 16 * j][k]);
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          acc[i][j] = fmaf(a[i].x, b[0][j].x, acc[i][j]); acc[i][j] = fmaf(a[i].y, b[0][j].y, acc[i][j]);
          acc[i][j] = fmaf(a[i].z, b[0][j].z, acc[i][j]); acc[i][j] = fmaf(a[i].w, b[0][j].w, acc[i][j]);
          if (DUAL) {
            acc2[i][j] = fmaf(a[i].x, b[kNB - 1][j].x, acc2[i][j]); acc2[i][j] = fmaf(a[i].y, b[kNB - 1][j].y, acc2[i][j]);
            acc2[i][j] = fmaf(a[i].z, b[kNB - 1][j].z, acc2[i][j]); acc2[i][j] = fmaf(a[i].w, b[kNB - 1][j].w, acc2[i][j]);
          }
        }
    }
  }
}

template <typename T>
struct SimtGemmArgs {
  const GroupStatic* gs;
  const GroupRows* gr;
  const T* a_shared;   // GEMM-1: outer rows of x [R, d];            GEMM-2: H_s [R, shared width]
  const T* a_routed;   // GEMM-1: permuted rows of x [R*N_k, d];     GEMM-2: H_r [R*N_k, m]
  const int32_t* row_token;   // small tiles, GEMM-1: outer row of every routed row (gathered from a_shared)
  const T* w_gate;     // GEMM-1: packed W_gate [rows, d];           GEMM-2: packed W_down
  const T* w_up;       // GEMM-1: packed W_up
  T* c_shared;         // GEMM-1: H_s;  GEMM-2: Y_s [R, d]
  T* c_routed;         // GEMM-1: H_r;  GEMM-2: Y_r [R*N_k, d]
  int d;
  int shared_width, routed_width;
};

// grid = (row tiles, column tiles, groups)
template <typename T>
__global__ void __launch_bounds__(256) simt_gemm1_kernel(const SimtGemmArgs<T> p) {
  grid_dep_wait();
  grid_dep_trigger();
  const GroupStatic g = p.gs[blockIdx.z];
  const GroupRows r = p.gr[blockIdx.z];
  const int m0 = blockIdx.x * kSimtTile, n0 = blockIdx.y * kSimtTile;
  if (m0 >= r.count || n0 >= g.width) return;
  const int ldc = g.is_shared ? p.shared_width : p.routed_width;
  const T* A = (g.is_shared ? p.a_shared : p.a_routed) + (size_t)r.row0 * p.d;
  const T* Bg = p.w_gate + (size_t)g.w_row0 * p.d;
  const T* Bu = p.w_up + (size_t)g.w_row0 * p.d;
  T* C = (g.is_shared ? p.c_shared : p.c_routed) + (size_t)r.row0 * ldc;
  float acc_g[4][4], acc_u[4][4];
  simt_tile<T, true>(A, p.d, r.count, Bg, Bu, p.d, g.width, p.d, m0, n0, true, true, acc_g, acc_u);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = m0 + ty * 4 + i;
    if (row >= r.count) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n < g.width) C[(size_t)row * ldc + n] = from_float<T>(silu_accurate(acc_g[i][j]) * acc_u[i][j]);
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) simt_gemm2_kernel(const SimtGemmArgs<T> p) {
  grid_dep_wait();
  grid_dep_trigger();
  const GroupStatic g = p.gs[blockIdx.z];
  const GroupRows r = p.gr[blockIdx.z];
  const int m0 = blockIdx.x * kSimtTile, n0 = blockIdx.y * kSimtTile;
  if (m0 >= r.count || n0 >= p.d || g.width == 0) return;
  const int lda = g.is_shared ? p.shared_width : p.routed_width;
  const T* A = (g.is_shared ? p.a_shared : p.a_routed) + (size_t)r.row0 * lda;
  const T* B = p.w_gate + g.wd_offset;                     // [d, width], ld = width
  T* C = (g.is_shared ? p.c_shared : p.c_routed) + (size_t)r.row0 * p.d;
  const bool vec = (g.width % 8 == 0) && (lda % 8 == 0) && (g.wd_offset % 8 == 0);
  float acc[4][4], unused[4][4];
  simt_tile<T, false>(A, lda, r.count, B, nullptr, g.width, p.d, g.width, m0, n0, vec, vec, acc, unused);
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const int row = m0 + ty * 4 + i;
    if (row >= r.count) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int c = n0 + tx * 4 + j;
      if (c < p.d) C[(size_t)row * p.d + c] = from_float<T>(acc[i][j]);
    }
  }
}

// The two GEMMs on small tiles.  SECOND = false: gate/up, routed rows gathered from x; true: down.
template <typename T, bool SECOND>
__global__ void __launch_bounds__(kSimtSmallThreads) simt_small_kernel(const SimtGemmArgs<T> p) {
  grid_dep_wait();
  grid_dep_trigger();
  const GroupStatic g = p.gs[blockIdx.z];
  const GroupRows r = p.gr[blockIdx.z];
  const int m0 = blockIdx.x * kSimtSmallM, n0 = blockIdx.y * kSimtSmallN;
  const int N = SECOND ? p.d : g.width, K = SECOND ? g.width : p.d;
  if (m0 >= r.count || n0 >= N || g.width == 0) return;
  const int width = g.is_shared ? p.shared_width : p.routed_width;
  const int lda = SECOND ? width : p.d, ldc = SECOND ? p.d : width;
  const T* A = (g.is_shared || !SECOND ? p.a_shared : p.a_routed);
  auto a_rows = [&](int i) -> const T* {
    if (m0 + i >= r.count) return nullptr;
    const int row = r.row0 + m0 + i;
    return A + (size_t)(!SECOND && !g.is_shared ? __ldcg(p.row_token + row) : row) * lda;
  };
  const T* B = p.w_gate + (SECOND ? (size_t)g.wd_offset : (size_t)g.w_row0 * p.d);
  const T* B2 = SECOND ? nullptr : p.w_up + (size_t)g.w_row0 * p.d;
  const bool vec_a = lda % 4 == 0, vec_b = SECOND ? (g.width % 4 == 0 && g.wd_offset % 4 == 0) : true;     // d is a multiple of 8
  float acc[2][2], acc2[2][2];
  simt_tile_small<T, !SECOND>(a_rows, B, B2, K, N, K, n0, vec_a, vec_b, acc, acc2);
  T* C = (g.is_shared ? p.c_shared : p.c_routed) + (size_t)r.row0 * ldc;
  const int ty = threadIdx.x >> 4, tx = threadIdx.x & 15;
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int row = m0 + 2 * ty + i, n = n0 + tx + 16 * j;
      if (row < r.count && n < N)
        C[(size_t)row * ldc + n] = from_float<T>(SECOND ? acc[i][j] : silu_accurate(acc[i][j]) * acc2[i][j]);
    }
}

}  // namespace cmoe
