// fp32 layers of a few rows, in three launches with the router: everything is latency, so the gate/up product needs nothing of the
// routing and runs beside the router, and the down product, the combine and the permutation are one launch.
//
//   small_up_kernel:   H[t, n] = Swish(w_gate[n] . x_t) (w_up[n] . x_t) for ALL rows and neurons (Eq. ori_ffn_method), ahead of the
//       wait for the router.  Tiles of 16 rows x 16 neurons, four warps that take 64 k each in turn.
//   small_down_kernel: out[t, c] = sum over the shared expert and the experts that t selected of g (W_down[c] . H[t])  (Eq. moe_output).
//       Tiles of 8 rows x 16 channels; eight warps take 64 neurons of one expert each in turn, add them times the gate where the row
//       selected the expert (a select, not a zero gate: an unselected expert's Inf or NaN goes no further), and meet in shared memory in
//       warp order.  The first weights are fetched ahead of the wait.  One more block writes the permutation, which only
//       cmoe_get_routing and the utilisation read.
// Forwards back to back, 64 rows, d = 256, 8 x 128 neurons: 26.0 us in five launches (router, permutation, two GEMMs, combine), 14.7 in three; 1 / 128 /
// 256 rows 22.0 / 27.8 / 38.1 -> 15.4 / 16.2 / 29.1; d = 512, 8 x 192 neurons, 8 / 64 / 128 rows 33.8 / 48.8 / 56.1 -> 15.2 / 22.0 / 43.5.
// A warp fetches its whole 64-wide slice at once (coalesced 16-byte loads, all in flight) into its own part of shared memory: no
// block barrier inside the sums.  Unselected experts' products are computed in vain, so the host takes this path only where that is
// expected to be cheaper than two more launches (small_fp32_takes).
#pragma once

#include <cmath>

#include "common.cuh"
#include "permute.cuh"

namespace cmoe {

constexpr int kSmKC = 64, kSmLd = kSmKC + 4;         // k per slice; row stride in shared memory (conflict-free 16-byte reads)
constexpr int kSmUpM = 16, kSmUpN = 16, kSmUpWarps = 4;
constexpr int kSmDnM = 8, kSmDnN = 16, kSmDnWarps = 8;
constexpr int kSmMaxRows = 256;
constexpr double kSmMaxWork = 400e6;                 // multiply-adds of all experts: 302 M 43.5 against 56.1 us, even on both paths at 440 to 600 M
constexpr int kSmUpSmem = kSmUpWarps * (kSmUpM + 2 * kSmUpN) * kSmLd * 4;
constexpr int kSmDnSmem = kSmDnWarps * (kSmDnM + kSmDnN) * kSmLd * 4;
static_assert(kSmMaxRows <= kMaskRows && kMaxRouted <= kMaskGroups && kSmMaxRows * kMaxTopK <= kMaskPairs, "one block permutes");
static_assert(kMaskBytes <= kSmDnSmem && kSmDnWarps * 32 == kMaskThreads, "the permutation runs in a block of the down kernel");

struct SmallArgs {
  const float *x, *w_gate, *w_up, *w_down;           // packed
  float* h;                                          // [rows][d_ff]
  float* out;
  const int32_t* topk_idx;
  const float* topk_gate;
  int n_rows, d, d_ff, shared_w, m, n_r, n_k;
  PermuteOut perm;
};

// Lanes 4 x 8: rows ty, ty + 4, ... of A against rows tx, tx + 8, ... of B, both [row][kSmLd] in shared memory.
template <int MA, int NB>
__device__ __forceinline__ void small_slice(const float* A, const float* B, int lane, float (&acc)[MA][NB]) {
  const float *a0 = A + (lane >> 3) * kSmLd, *b0 = B + (lane & 7) * kSmLd;
#pragma unroll 4
  for (int k = 0; k < kSmKC; k += 4) {
    float4 a[MA], b[NB];
#pragma unroll
    for (int i = 0; i < MA; ++i) a[i] = *reinterpret_cast<const float4*>(a0 + 4 * i * kSmLd + k);
#pragma unroll
    for (int j = 0; j < NB; ++j) b[j] = *reinterpret_cast<const float4*>(b0 + 8 * j * kSmLd + k);
#pragma unroll
    for (int i = 0; i < MA; ++i)
#pragma unroll
      for (int j = 0; j < NB; ++j) {
        acc[i][j] = fmaf(a[i].x, b[j].x, acc[i][j]); acc[i][j] = fmaf(a[i].y, b[j].y, acc[i][j]);
        acc[i][j] = fmaf(a[i].z, b[j].z, acc[i][j]); acc[i][j] = fmaf(a[i].w, b[j].w, acc[i][j]);
      }
  }
}
// This lane's pieces of ROWS rows of a slice (row r: quads of `row(r)` + k, null and past `width`: zeros).
template <int ROWS> struct SmallTile {
  float4 v[ROWS / 2];
  template <typename Row> __device__ __forceinline__ void load(Row row, int k, int width, int lane) {
    const int q = 4 * (lane & 15);
#pragma unroll
    for (int i = 0; i < ROWS / 2; ++i) {
      const float* p = row(2 * i + (lane >> 4));
      uint4 r = make_uint4(0u, 0u, 0u, 0u);
      if (p && k + q < width) r = ld_dep16(p + k + q);
      v[i] = make_float4(__uint_as_float(r.x), __uint_as_float(r.y), __uint_as_float(r.z), __uint_as_float(r.w));
    }
  }
  __device__ __forceinline__ void store(float* dst, int lane) const {
#pragma unroll
    for (int i = 0; i < ROWS / 2; ++i) *reinterpret_cast<float4*>(dst + (2 * i + (lane >> 4)) * kSmLd + 4 * (lane & 15)) = v[i];
  }
};

// grid (neuron tiles, row tiles)
__global__ void __launch_bounds__(32 * kSmUpWarps) small_up_kernel(const SmallArgs p) {
  extern __shared__ __align__(16) float small_smem[];
  grid_dep_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * kSmUpN, t0 = blockIdx.y * kSmUpM;
  float* A = small_smem + warp * (kSmUpM + 2 * kSmUpN) * kSmLd;
  float* B = A + kSmUpM * kSmLd;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  auto x_row = [&](int r) { return t0 + r < p.n_rows ? p.x + (size_t)(t0 + r) * p.d : nullptr; };
  auto w_row = [&](int r) {                           // 16 gate rows, then 16 up rows
    const int n = n0 + (r & 15);
    return n < p.d_ff ? (r < 16 ? p.w_gate : p.w_up) + (size_t)n * p.d : nullptr;
  };
  // the router, ahead in the stream, lets this kernel start after its own wait: x is final
#pragma unroll 1
  for (int k = warp * kSmKC; k < p.d; k += kSmUpWarps * kSmKC) {
    SmallTile<kSmUpM> a;
    SmallTile<2 * kSmUpN> b;
    a.load(x_row, k, p.d, lane);
    b.load(w_row, k, p.d, lane);
    __syncwarp();
    a.store(A, lane);
    b.store(B, lane);
    __syncwarp();
    small_slice<4, 4>(A, B, lane, acc);
  }
  __syncthreads();
  float* red = small_smem;                            // [warp][16][32]
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) red[(warp * 16 + 4 * i + j) * 32 + lane] = acc[i][j];
  __syncthreads();
  grid_dep_wait();                                    // whatever read H before has ended
#pragma unroll
  for (int o = threadIdx.x; o < kSmUpM * kSmUpN; o += 32 * kSmUpWarps) {
    const int n = o & 15, t = o >> 4;
    const int from = 4 * (t >> 2) + (n >> 3), at = 8 * (t & 3) + (n & 7);       // accumulator and lane
    float g = 0.0f, u = 0.0f;
#pragma unroll
    for (int w = 0; w < kSmUpWarps; ++w) { g += red[(w * 16 + from) * 32 + at]; u += red[(w * 16 + from + 2) * 32 + at]; }
    if (t0 + t < p.n_rows && n0 + n < p.d_ff) p.h[(size_t)(t0 + t) * p.d_ff + n0 + n] = silu_accurate(g) * u;
  }
}

// grid (channel tiles x row tiles + 1): the last block permutes
__global__ void __launch_bounds__(32 * kSmDnWarps) small_down_kernel(const SmallArgs p) {
  extern __shared__ __align__(16) float small_smem[];
  __shared__ float gate[kSmDnM][kMaxRouted];
  __shared__ uint32_t picked[kSmDnM];
  grid_dep_trigger();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (blockIdx.x == gridDim.x - 1) {
    grid_dep_wait();
    permute_from_selections(p.topk_idx, p.perm, reinterpret_cast<uint8_t*>(small_smem));
    return;
  }
  const int c_tiles = (p.d + kSmDnN - 1) / kSmDnN;
  const int c0 = blockIdx.x % c_tiles * kSmDnN, t0 = blockIdx.x / c_tiles * kSmDnM;
  float* A = small_smem + warp * (kSmDnM + kSmDnN) * kSmLd;
  float* B = A + kSmDnM * kSmLd;
  const int slices_s = (p.shared_w + kSmKC - 1) / kSmKC, slices_m = (p.m + kSmKC - 1) / kSmKC;
  const int n_slices = slices_s + p.n_r * slices_m;
  // slice s: expert (-1 shared), first neuron inside it, its width, its first column of H
  int e = -1, k = 0, width = 0, col0 = 0;
  auto slice = [&](int s) {
    if (s < slices_s) { e = -1; k = s * kSmKC; width = p.shared_w; col0 = 0; }
    else { e = (s - slices_s) / slices_m; k = (s - slices_s - e * slices_m) * kSmKC; width = p.m; col0 = p.shared_w + e * p.m; }
  };
  auto w_row = [&](int r) {
    return c0 + r < p.d ? p.w_down + (size_t)(e < 0 ? 0 : col0) * p.d + (size_t)(c0 + r) * width : nullptr;
  };
  auto h_row = [&](int r) { return t0 + r < p.n_rows ? p.h + (size_t)(t0 + r) * p.d_ff + col0 : nullptr; };
  SmallTile<kSmDnM> a;
  SmallTile<kSmDnN> b;
  int s = warp;
  if (s < n_slices) { slice(s); b.load(w_row, k, width, lane); }          // the layer's own
  grid_dep_wait();
  if (threadIdx.x < kSmDnM) {
    uint32_t mask = 0;
    const size_t t = (size_t)t0 + threadIdx.x;
    if (t < (size_t)p.n_rows) {
      int idx[kMaxTopK];
      float g[kMaxTopK];
#pragma unroll
      for (int i = 0; i < kMaxTopK; ++i) {
        idx[i] = i < p.n_k ? __ldcg(p.topk_idx + t * p.n_k + i) : 0;
        g[i] = i < p.n_k ? __ldcg(p.topk_gate + t * p.n_k + i) : 0.0f;
      }
#pragma unroll
      for (int i = 0; i < kMaxTopK; ++i)
        if (i < p.n_k) { gate[threadIdx.x][idx[i]] = g[i]; mask |= 1u << idx[i]; }
    }
    picked[threadIdx.x] = mask;
  }
  if (s < n_slices) a.load(h_row, k, width, lane);
  __syncthreads();
  const int ty = lane >> 3;
  const uint32_t mine[2] = {picked[ty], picked[ty + 4]};
  float sum[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
#pragma unroll 1
  for (; s < n_slices; s += kSmDnWarps) {
    __syncwarp();
    a.store(A, lane);
    b.store(B, lane);
    __syncwarp();
    const int now = e;
    if (s + kSmDnWarps < n_slices) {                                      // the next slice is on its way meanwhile
      slice(s + kSmDnWarps);
      b.load(w_row, k, width, lane);
      a.load(h_row, k, width, lane);
    }
    float acc[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
    small_slice<2, 2>(A, B, lane, acc);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const bool on = now < 0 || ((mine[i] >> now) & 1u);
      const float g = now < 0 ? 1.0f : on ? gate[ty + 4 * i][now] : 0.0f;
#pragma unroll
      for (int j = 0; j < 2; ++j) sum[i][j] = on ? fmaf(g, acc[i][j], sum[i][j]) : sum[i][j];
    }
  }
  __syncthreads();
  float* red = small_smem;                                                // [warp][4][32]
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 2; ++j) red[(warp * 4 + 2 * i + j) * 32 + lane] = sum[i][j];
  __syncthreads();
  if (threadIdx.x < kSmDnM * kSmDnN) {
    const int c = threadIdx.x & 15, t = threadIdx.x >> 4;
    const int from = 2 * (t >> 2) + (c >> 3), at = 8 * (t & 3) + (c & 7);
    float y = 0.0f;
#pragma unroll
    for (int w = 0; w < kSmDnWarps; ++w) y += red[(w * 4 + from) * 32 + at];
    if (t0 + t < p.n_rows && c0 + c < p.d) p.out[(size_t)(t0 + t) * p.d + c0 + c] = y;
  }
}

// Whether a plain fp32 layer's forward of so many rows takes this path: 16-byte rows, and less time expected here than in the five
// launches of the general path, which multiplies the selected experts only.  Both times (us) are fits to 40 shapes (d 64 to 4096, 2 to 34
// experts of 32 to 1376 neurons, top-1 to 8) at 1 to 256 rows, chained forwards on one B200, good to about 17 %.
//   Here: rounds of up blocks (four per SM) times the slices of d that a warp takes, the slices of all experts that a warp of a down block
// takes, alone and times the down blocks per SM, and all experts' weights.
//   There: the length of the two k loops, the down tiles' slices per SM (16 x 32 tiles of the rows that an expert is expected to get), and the
// weights of the experts that at least one row is expected to select.
// Choosing by them costs 0.5 % over the better path (geometric mean over these and 14 more shapes; the factor 1.05 is the best of 0.95 to
// 1.1).  Here / there, us: 8 x 128 neurons, d = 256, top-2 64 rows 12.4 / 25.8, 256 rows 29.4 / 37.4; 34 x 128 neurons, d = 256, 1 / 64 / 96
// rows 26 / 43 / 50 against 28 / 38 / 40; 34 x 256 neurons, d = 128, 16 rows 57 / 34; d = 2048, 34 x 256 neurons, one row 210 / 130; d = 2048,
// 8 x 688 neurons, one row 98 / 166.
inline bool small_fp32_takes(int rows, int d, int d_ff, int shared_w, int m, int n_r, int n_k, int n_sms) {
  if (rows < 1 || rows > kSmMaxRows || n_r < 1 || n_k < 1 || m % 4 || shared_w % 4) return false;
  if ((double)rows * 3.0 * d * d_ff > kSmMaxWork) return false;
  auto cut = [](double v, double by) { return ceil(v / by); };
  const double mb = 12e-6 * d * d_ff;                                            // all experts' weights
  const double slices = cut(shared_w, kSmKC) + n_r * cut(m, kSmKC), per_warp = cut(slices, kSmDnWarps);
  const double up_rounds = cut(cut(d_ff, kSmUpN) * cut(rows, kSmUpM), 4 * n_sms), down_blocks = cut(d, kSmDnN) * cut(rows, kSmDnM);
  const double here = 4.5 + 3.6 * up_rounds * cut(d, kSmUpWarps * kSmKC) + 1.6 * per_warp + 1.5 * per_warp * down_blocks / n_sms + 0.38 * mb;
  const double hit = n_r * (1.0 - pow(1.0 - (double)n_k / n_r, rows));           // experts with rows
  const double each = (double)rows * n_k / n_r > 1.0 ? (double)rows * n_k / n_r : 1.0;
  const double touched = mb * (shared_w + hit * m) / d_ff;
  const double tiles = cut(d, 32) * (cut(rows, 16) * cut(shared_w, 64) + hit * cut(each, 16) * cut(m, 64));
  const double there = 11.0 + 2.7 * d / 64 + (shared_w > m ? shared_w : m) / 64.0 + 1.4 * tiles / n_sms + 0.43 * touched;
  if (mb > 30.0 && mb > 3.0 * touched) return false;                             // weights from DRAM: not three times as many
  return here < 1.05 * there;
}

inline cudaError_t small_fp32_allow() {
  const cudaError_t e = allow_smem(small_up_kernel, kSmUpSmem);
  return e == cudaSuccess ? allow_smem(small_down_kernel, kSmDnSmem) : e;
}

inline cudaError_t small_fp32_forward(const SmallArgs& a, bool dep, cudaStream_t st, cudaEvent_t mid) {
  const dim3 up((a.d_ff + kSmUpN - 1) / kSmUpN, (a.n_rows + kSmUpM - 1) / kSmUpM);
  cudaError_t e = launch_kernel(dep, small_up_kernel, up, dim3(32 * kSmUpWarps), kSmUpSmem, st, a);
  if (mid) cudaEventRecord(mid, st);
  const int tiles = (a.d + kSmDnN - 1) / kSmDnN * ((a.n_rows + kSmDnM - 1) / kSmDnM);
  if (e == cudaSuccess) e = launch_kernel(dep, small_down_kernel, dim3(tiles + 1), dim3(32 * kSmDnWarps), kSmDnSmem, st, a);
  return e;
}

}  // namespace cmoe
