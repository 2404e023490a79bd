// bf16 router for up to kRcMaxRows rows (Eq. router, Eq. final_gate) with the permutation of small batches in the
// same launch.  Bound: latency.  The contraction [16 rows, d] x [d, 2 N_r] is tiny, but its operands come from DRAM
// and everything downstream waits for it, so the kernel is one chain that is kept short:
//   - a cluster of 8 CTAs owns a tile of 16 rows; its 64 warps split K (32-wide slices, mma.sync.m16n8k16), so every
//     16-byte load of a d = 4096 layer is in flight at once;
//   - each CTA adds its 8 warps' sums and pushes two rows each to its peers' shared memory, and after one cluster
//     barrier every CTA adds the eight contributions of its own two rows in rank order (deterministic) and runs their gate
//     logic, one warp per row;
//   - rank 0 collects the selections the same way and, with one row tile, permutes at once; with more, the tile that
//     takes the last ticket permutes the batch: per group a bit mask of its rows, population counts for ranks and counts.
// A hierarchical layer runs it twice, for the outer experts and for the inner ones; the second pass reads every outer row
// from its token and writes the layer's copy of the rows as it goes (8 x 7B-shaped layer, 7 / 128 / 700 tokens, against a block per 16
// tokens, a permutation and a copy kernel: 288.8 / 512.4 / 594.2 -> 266.8 / 491.7 / 575.9 us).  Against K slices over independent blocks
// that met in global memory, the last block alone doing the gate logic: 7B-shaped layer 1 / 16 / 64 rows 40.5 / 67.4 / 74.1 -> 35.0 /
// 62.1 / 69.1 us.  Alone and with cold caches a launch takes 9 us at 16 and 11 at 300 rows.  Where tensor-core tiles take over:
// router_takes_tiles.
#pragma once

#include "common.cuh"
#include "permute.cuh"
#include "router.cuh"
#include "router_mma.cuh"

namespace cmoe {

constexpr int kRcThreads = 256;
constexpr int kRcCluster = 8;
constexpr int kRcRows = 16;                 // rows of a cluster's tile
constexpr int kRcMaxRows = 1024;            // rows of a batch this kernel takes
static_assert(kRcMaxRows <= kMaskRows && kRcThreads == kMaskThreads, "the fused permutation is permute_by_masks");

__device__ __forceinline__ void rc_cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void rc_cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
// Address of a shared variable of this CTA in the shared memory of cluster CTA `rank`.
__device__ __forceinline__ uint32_t rc_peer(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"((uint32_t)__cvta_generic_to_shared(p)), "r"(rank));
  return r;
}
__device__ __forceinline__ void rc_push(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void rc_push(uint32_t addr, int v) {
  asm volatile("st.shared::cluster.s32 [%0], %1;" ::"r"(addr), "r"(v) : "memory");
}

struct RouterArgs {
  const bf16* x;
  const int32_t* row_src;          // hierarchical: the token of every outer row; x_copy takes the row in passing
  bf16* x_copy;
  int n_rows, d, n_r, n_rp, n_k;   // top-level router: n_r = outer experts, n_k = those of a token
  const bf16* w_rep;
  const float *u, *b;
  const int32_t* outer_off;        // hierarchical: row ranges of the outer experts
  int n_outer;
  int32_t* ticket;                 // zero between launches
  float *scores, *keys;            // top-level router: scores = logits, topk_gate = weights
  int32_t* topk_idx;
  float* topk_gate;
  int late_wait;                   // the preceding kernel of the forward is the split of the token rows, which this one does not read
  int fuse_permute, n_groups;
  int32_t *counts, *offsets, *row_token, *row_of;
  GroupPlanOut po;
};

// MAXT: tiles of 8 router columns at most (2 N_r rounded up); NB: outer experts whose representative rows are held in
// flight at once when a tile's rows belong to several (1 for a plain layer).  OUTER: the top-level router of a
// hierarchical layer, one column per outer expert.
template <int MAXT, int NB, bool OUTER = false>
__global__ void __cluster_dims__(kRcCluster, 1, 1) __launch_bounds__(kRcThreads, MAXT * NB <= 2 ? 3 : 2)
router_cluster_kernel(const RouterArgs p) {
  constexpr int kCols = MAXT * 8, kStride = kCols + 8;
  constexpr int kUnr = 16 / (MAXT * NB) >= 2 ? 2 : 1;                // k slices in flight per warp
  constexpr int kPartBytes = 8 * kRcRows * kStride * 4;
  __shared__ __align__(16) uint8_t scratch[kPartBytes > kMaskBytes ? kPartBytes : kMaskBytes];
  float (*part)[kRcRows][kStride] = reinterpret_cast<float (*)[kRcRows][kStride]>(scratch);   // [warp]
  __shared__ float recv[kRcCluster][2][kCols];                       // [source CTA][row 2 rank + i][column]
  __shared__ int sel_recv[kRcRows * kMaxTopK];                       // rank 0: the tile's selections
  __shared__ int row_group[kRcRows], g_list[kRcRows];
  __shared__ int n_list, is_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = blockIdx.x;                                  // the grid's x extent is one cluster
  const int row_base = blockIdx.y * kRcRows;
  const int n_rows = min(kRcRows, p.n_rows - row_base);
  rc_cluster_arrive();                                               // the peers have started: waited for before the push
  const int g = lane >> 2, t = lane & 3;
  const int n2 = OUTER ? p.n_r : 2 * p.n_rp, n_tiles = (n2 + 7) >> 3;
  const int n_slices = (p.d + 31) >> 5, s0 = (int)rank * 8 + warp;
  const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
  uint4 w[kUnr][NB][MAXT];
  // representative rows of expert list entries i0 .. i0 + NB - 1, k slices s, s + 64 ..
  auto load_w = [&](int s, int i0, int nl) {
#pragma unroll
    for (int q = 0; q < kUnr; ++q) {
      const int k = (s + 64 * q) * 32 + 8 * t;
#pragma unroll
      for (int i = 0; i < NB; ++i) {
        const bool have = k < p.d && (NB == 1 || i0 + i < nl);
        const bf16* wr = p.w_rep + ((size_t)(NB > 1 && have ? g_list[i0 + i] : 0) * n2 + g) * p.d + k;
#pragma unroll
        for (int nt = 0; nt < MAXT; ++nt)
          w[q][i][nt] = (have && (OUTER ? nt * 8 + g < n2 : nt < n_tiles)) ? __ldg(reinterpret_cast<const uint4*>(wr + (size_t)nt * 8 * p.d)) : zero;
      }
    }
  };
  if (NB == 1) load_w(s0, 0, 1);          // the layer's own rows: fetched while the preceding kernel of the stream drains
  // The split lets this kernel start after its own wait, so x is final; what follows reads the planes and starts after it.
  // FP8 layers, waiting first / late: 8B-shaped 4 rows 42.7 / 40.0 us, 7B-shaped 2 rows 38.2 / 37.3, even from 16 rows on.
  const bool late = NB == 1 && !OUTER && p.late_wait;
  if (!late) { grid_dep_wait(); grid_dep_trigger(); }
  if (NB > 1 && warp == 0) {
    const int go = (p.outer_off && lane < kRcRows) ? find_outer(p.outer_off, p.n_outer, row_base + min(lane, n_rows - 1)) : 0;
    const int prev = __shfl_up_sync(0xffffffffu, go, 1);
    const bool first = lane == 0 || (lane < kRcRows && go != prev);  // rows are sorted by outer expert
    const uint32_t m = __ballot_sync(0xffffffffu, first);
    if (lane < kRcRows) row_group[lane] = go;
    if (first) g_list[__popc(m & ((1u << lane) - 1u))] = go;
    if (lane == 0) n_list = __popc(m);
  }
  if (NB > 1) __syncthreads();
  // u and b of this warp's gate row (warps 0 and 1), fetched ahead of the sums
  const int my_row = 2 * (int)rank + warp;
  const bool gate_warp = warp < 2 && my_row < n_rows;
  float u_pre = 0.0f, b_pre = 0.0f;
  int go_mine = 0;
  if (!OUTER && gate_warp) {
    if (NB > 1) go_mine = row_group[my_row];
    if (lane < p.n_r) { u_pre = __ldcg(p.u + go_mine * p.n_r + lane); b_pre = __ldcg(p.b + go_mine * p.n_r + lane); }
  }
  // ---- partial sums over this warp's k slices
  const int r_lo = min(g, n_rows - 1), r_hi = min(g + 8, n_rows - 1);
  const bf16* x_lo = p.x + (size_t)(NB > 1 ? __ldcg(p.row_src + row_base + r_lo) : row_base + r_lo) * p.d + 8 * t;
  const bf16* x_hi = p.x + (size_t)(NB > 1 ? __ldcg(p.row_src + row_base + r_hi) : row_base + r_hi) * p.d + 8 * t;
  const int nl = NB > 1 ? n_list : 1;
#pragma unroll 1
  for (int i0 = 0; i0 < nl; i0 += NB) {
    float acc[NB][MAXT][4];
#pragma unroll
    for (int i = 0; i < NB; ++i)
#pragma unroll
      for (int nt = 0; nt < MAXT; ++nt)
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][nt][q] = 0.0f;
#pragma unroll 1
    for (int s = s0; s < n_slices; s += 64 * kUnr) {
      uint4 a_lo[kUnr], a_hi[kUnr];
#pragma unroll
      for (int q = 0; q < kUnr; ++q) {
        const int k = (s + 64 * q) * 32;
        const bool in = k + 8 * t < p.d;
        a_lo[q] = in ? ld_dep16(x_lo + k) : zero;
        a_hi[q] = in ? ld_dep16(x_hi + k) : zero;
      }
      if (NB > 1 || s != s0) load_w(s, i0, nl);
      if (NB > 1 && i0 == 0) {                                       // the outer rows, for the GEMMs
#pragma unroll
        for (int q = 0; q < kUnr; ++q) {
          const int k = (s + 64 * q) * 32 + 8 * t;
          if (k < p.d) {
            if (g < n_rows) *reinterpret_cast<uint4*>(p.x_copy + (size_t)(row_base + g) * p.d + k) = a_lo[q];
            if (g + 8 < n_rows) *reinterpret_cast<uint4*>(p.x_copy + (size_t)(row_base + g + 8) * p.d + k) = a_hi[q];
          }
        }
      }
#pragma unroll
      for (int q = 0; q < kUnr; ++q)
#pragma unroll
        for (int i = 0; i < NB; ++i)
#pragma unroll
          for (int nt = 0; nt < MAXT; ++nt)
            if (nt < n_tiles) {
              mma_bf16_16816(acc[i][nt], a_lo[q].x, a_hi[q].x, a_lo[q].y, a_hi[q].y, w[q][i][nt].x, w[q][i][nt].y);
              mma_bf16_16816(acc[i][nt], a_lo[q].z, a_hi[q].z, a_lo[q].w, a_hi[q].w, w[q][i][nt].z, w[q][i][nt].w);
            }
    }
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      if (NB > 1 && i0 + i >= nl) break;
      const int go = NB > 1 ? g_list[i0 + i] : 0;
      const bool take_lo = NB == 1 || row_group[g] == go, take_hi = NB == 1 || row_group[g + 8] == go;
#pragma unroll
      for (int nt = 0; nt < MAXT; ++nt)
        if (nt < n_tiles) {
          float* lo = &part[warp][g][nt * 8 + 2 * t];
          float* hi = &part[warp][g + 8][nt * 8 + 2 * t];
          if (take_lo) { lo[0] = acc[i][nt][0]; lo[1] = acc[i][nt][1]; }
          if (take_hi) { hi[0] = acc[i][nt][2]; hi[1] = acc[i][nt][3]; }
        }
    }
  }
  if (late) { grid_dep_wait(); grid_dep_trigger(); }
  __syncthreads();
  rc_cluster_wait();
#pragma unroll 1
  for (int i = threadIdx.x; i < kRcRows * n2; i += kRcThreads) {     // this CTA's sums, each to the CTA of its row
    const int r = i / n2, c = i - r * n2;
    float s = 0.0f;
#pragma unroll
    for (int w = 0; w < 8; ++w) s += part[w][r][c];
    rc_push(rc_peer(&recv[rank][r & 1][c], r >> 1), s);
  }
  rc_cluster_arrive();
  rc_cluster_wait();
  // ---- gate logic, one warp per row
  if (gate_warp) {
    float a = 0.0f, v = 0.0f;
    if (lane < p.n_r)
#pragma unroll
      for (int q = 0; q < kRcCluster; ++q) { a += recv[q][warp][lane]; if (!OUTER) v += recv[q][warp][p.n_rp + lane]; }
    const size_t row = (size_t)row_base + my_row;
    int sel = 0;
    if (OUTER)
      outer_row_redux(lane, p.n_r, p.n_k, a, p.scores + row * p.n_r, p.topk_idx + row * p.n_k, p.topk_gate + row * p.n_k, sel);
    else
      gate_row_redux(lane, p.n_r, p.n_k, a, v, u_pre, b_pre, go_mine * p.n_r, row, p.scores, p.keys, p.topk_idx, p.topk_gate, sel);
    if (p.fuse_permute && lane < p.n_k) rc_push(rc_peer(&sel_recv[my_row * p.n_k + lane], 0), sel);
  }
  if (!p.fuse_permute) return;
  rc_cluster_arrive();
  rc_cluster_wait();
  if (rank != 0) return;
  // ---- permutation
  uint8_t* sel = scratch;                                             // [n_rows * n_k <= kMaskPairs]
  if (gridDim.y == 1) {
#pragma unroll 1
    for (int i = threadIdx.x; i < n_rows * p.n_k; i += kRcThreads) sel[i] = (uint8_t)sel_recv[i];
  } else {
    if (threadIdx.x == 0) {                                           // the tile's selections are ordered before the ticket
      __threadfence();
      is_last = atomicAdd(p.ticket, 1) == (int)gridDim.y - 1;
      if (is_last) *p.ticket = 0;
      __threadfence();
    }
    __syncthreads();
    if (!is_last) return;
    const int pairs = p.n_rows * p.n_k;
#pragma unroll 1
    for (int i0 = threadIdx.x; i0 < pairs; i0 += 8 * kRcThreads) {    // eight loads in flight per thread
      int v[8];
#pragma unroll
      for (int q = 0; q < 8; ++q) v[q] = i0 + q * kRcThreads < pairs ? __ldcg(p.topk_idx + i0 + q * kRcThreads) : 0;
#pragma unroll
      for (int q = 0; q < 8; ++q)
        if (i0 + q * kRcThreads < pairs) sel[i0 + q * kRcThreads] = (uint8_t)v[q];
    }
  }
  __syncthreads();
  permute_by_masks(PermuteOut{p.n_rows, p.n_k, p.n_groups, p.counts, p.offsets, p.row_token, p.row_of, p.po}, scratch);
}

inline bool router_cluster_fuses(int n_rows, int n_k, int n_groups) {
  return n_rows <= kRcMaxRows && permute_masks_fit(n_rows, n_k, n_groups);
}

// Top-level router of a hierarchical layer with its permutation (router_cluster_fuses(n_tokens, outer_k, n_outer)).
inline cudaError_t outer_router_cluster_launch(const RouterArgs& a, bool dep, cudaStream_t st) {
  const dim3 grid(kRcCluster, (a.n_rows + kRcRows - 1) / kRcRows), block(kRcThreads);
  if (a.n_r <= 8) return launch_kernel(dep, router_cluster_kernel<1, 1, true>, grid, block, 0, st, a);
  return launch_kernel(dep, router_cluster_kernel<4, 1, true>, grid, block, 0, st, a);
}

inline cudaError_t router_cluster_launch(const RouterArgs& a, bool hier, bool dep, bool all_smem, cudaStream_t st) {
  const dim3 grid(kRcCluster, (a.n_rows + kRcRows - 1) / kRcRows), block(kRcThreads);
  const int tiles = 2 * a.n_rp / 8;
  if (hier) {                                                         // a.row_src and a.x_copy are set
    if (tiles <= 2) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<2, 4>, grid, block, 0, st, a);
    if (tiles <= 4) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<4, 2>, grid, block, 0, st, a);
    return launch_kernel_smem(dep, all_smem, router_cluster_kernel<8, 2>, grid, block, 0, st, a);
  }
  if (tiles <= 2) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<2, 1>, grid, block, 0, st, a);
  if (tiles <= 4) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<4, 1>, grid, block, 0, st, a);
  return launch_kernel_smem(dep, all_smem, router_cluster_kernel<8, 1>, grid, block, 0, st, a);
}

}  // namespace cmoe
