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
// Against K slices over independent blocks (partial sums and a ticket through global memory, the last block alone
// doing the gate logic and a block-wide scan; the permutation in kernels of its own above 128 rows), whole forwards: 7B-shaped
// layer 1 / 16 / 64 / 128 / 512 rows 40.5 / 67.4 / 74.1 / 86.9 / 114.0 -> 35.0 / 62.1 / 69.1 / 80.0 / 109.3 us, 8B-shaped 32 /
// 256 / 512 rows 88.2 / 112.3 / 140.9 -> 80.7 / 102.0 / 121.8, hierarchical 7 rows 295 -> 278.  Against the 128-row
// tensor-core tiles of umma_grouped_kernel<3>: 8B-shaped 700 / 1000 / 2048 rows 143.7 / 181.4 / 237.6 -> 129.5 / 170.3 /
// 240.7, 7B-shaped 600 / 1000 / 2048 rows 121.0 / 186.8 / 257.9 -> 117.9 / 179.3 / 269.3: every tile re-reads the
// representative rows, so the line is drawn at 1024 rows.
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
constexpr int kRcFuseGroups = 64;           // routed groups up to which the permutation runs in the same launch
// ... and selections (fused against the permutation kernels: 8B-shaped 700 rows x 4: 129.5 against 131.4 us, 7B-shaped 1000 x 2:
// 179.3 against 184.6, 8B-shaped 1000 x 4: 174.9 against 170.3)
constexpr int kRcFusePairs = 3072;
constexpr int kRcPermBytes = kRcFusePairs + kRcFuseGroups * (kRcMaxRows / 32) * 6 + kRcFuseGroups * 8;

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

// A float's bits mapped so that unsigned order is numeric order (-0 counts as +0).
__device__ __forceinline__ uint32_t ordered_bits(float v) {
  const uint32_t b = __float_as_uint(v + 0.0f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// gate_row with u and b already in registers and the arg-max by one warp-wide integer reduction and a ballot (the
// same order: larger key first, equal keys by index).  Lane i < n_k returns its selection in `sel`.
__device__ __forceinline__ void gate_row_redux(int lane, int n_r, int n_k, float a, float v, float u, float b, int group_base,
                                               float* __restrict__ scores_row, float* __restrict__ keys_row,
                                               int32_t* __restrict__ idx_row, float* __restrict__ gates_row, int& sel) {
  const bool live = lane < n_r;
  const float s = live ? silu_accurate(a) * v : -INFINITY;            // Eq. router
  const float s_max = warp_max(s);
  const float e = live ? expf(s - s_max) : 0.0f;
  const float s_prime = e / warp_sum(e);                               // Softmax over all N_r
  const float key = live ? s_prime + b : -INFINITY;
  if (live) { scores_row[lane] = s; keys_row[lane] = key; }
  const float gate = 1.0f + s_prime * u;                               // 1 + s'_i u_i
  const float rank_key = (key != key) ? -INFINITY : key;               // NaN ranks last
  uint32_t bits = live ? ordered_bits(rank_key) : 0u;                  // every live key is above 0
  float my_gate = 0.0f;
#pragma unroll 1
  for (int i = 0; i < n_k; ++i) {
    const uint32_t best = __reduce_max_sync(0xffffffffu, bits);
    const int who = __ffs(__ballot_sync(0xffffffffu, bits == best)) - 1;
    const float g = __shfl_sync(0xffffffffu, gate, who);
    if (lane == who) bits = 0u;
    if (lane == i) { sel = group_base + who; my_gate = g; }
  }
  if (lane < n_k) { idx_row[lane] = sel; gates_row[lane] = my_gate; }
}

struct RouterArgs {
  const bf16* x;
  int n_rows, d, n_r, n_rp, n_k;
  const bf16* w_rep;
  const float *u, *b;
  const int32_t* outer_off;        // hierarchical: row ranges of the outer experts
  int n_outer;
  int32_t* ticket;                 // zero between launches
  float *scores, *keys;
  int32_t* topk_idx;
  float* topk_gate;
  int fuse_permute, n_groups;
  int32_t *counts, *offsets, *row_token, *row_of;
  GroupPlanOut po;
};

// Histogram, scan and stable permutation of at most kRcFusePairs selections over at most kRcFuseGroups groups, by one
// block.  sel[i]: selection of pair i = row * n_k + j, already in shared memory.  mask[g][w]: which of the rows
// 32 w .. 32 w + 31 selected group g; before[g][w]: how many rows ahead of those did.
__device__ __forceinline__ void permute_by_masks(const RouterArgs& p, const uint8_t* sel, uint32_t* mask, uint16_t* before,
                                                 int32_t* count, int32_t* offs) {
  const int words = (p.n_rows + 31) >> 5, pairs = p.n_rows * p.n_k;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
#pragma unroll 1
  for (int i = threadIdx.x; i < p.n_groups * words; i += kRcThreads) mask[i] = 0;
  __syncthreads();
#pragma unroll 1
  for (int row = threadIdx.x; row < p.n_rows; row += kRcThreads)
#pragma unroll 1
    for (int j = 0; j < p.n_k; ++j) atomicOr(&mask[sel[row * p.n_k + j] * words + (row >> 5)], 1u << (row & 31));
  __syncthreads();
#pragma unroll 1
  for (int g = warp; g < p.n_groups; g += kRcThreads / 32) {           // lane: word (at most kRcMaxRows / 32 = 32)
    const int c = lane < words ? __popc(mask[g * words + lane]) : 0;
    int incl = c;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    if (lane < words) before[g * words + lane] = (uint16_t)(incl - c);
    if (lane == 31) count[g] = incl;
  }
  __syncthreads();
  if (warp == 0) {                                                     // lane l: groups 2l and 2l + 1
    int c[2];
#pragma unroll
    for (int q = 0; q < 2; ++q) c[q] = 2 * lane + q < p.n_groups ? count[2 * lane + q] : 0;
    int incl = c[0] + c[1];
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    int run = incl - c[0] - c[1];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int g = 2 * lane + q;
      if (g < p.n_groups) {
        offs[g] = run;
        p.counts[g] = c[q];
        p.offsets[g] = run;
        if (p.po.gr) { GroupRows r; r.row0 = run; r.count = c[q]; p.po.gr[p.po.n_outer + g] = r; }
        run += c[q];
        if (g == p.n_groups - 1) p.offsets[p.n_groups] = run;
      }
    }
  } else if (p.po.gr) {
#pragma unroll 1
    for (int g = threadIdx.x - 32; g < p.po.n_outer; g += kRcThreads - 32) {
      GroupRows r;
      r.row0 = p.po.outer_off ? p.po.outer_off[g] : 0;
      r.count = p.po.outer_off ? p.po.outer_off[g + 1] - r.row0 : p.po.n_tokens;
      p.po.gr[g] = r;
    }
  }
  __syncthreads();
#pragma unroll 1
  for (int row = threadIdx.x; row < p.n_rows; row += kRcThreads) {
    const int w = row >> 5;
    const uint32_t below = (1u << (row & 31)) - 1u;
#pragma unroll 1
    for (int j = 0; j < p.n_k; ++j) {
      const int g = sel[row * p.n_k + j];
      const int pos = offs[g] + before[g * words + w] + __popc(mask[g * words + w] & below);
      p.row_token[pos] = row;
      p.row_of[row * p.n_k + j] = pos;
    }
  }
}

// MAXT: tiles of 8 router columns at most (2 N_r rounded up); NB: outer experts whose representative rows are held in
// flight at once when a tile's rows belong to several (1 for a plain layer).
template <int MAXT, int NB>
__global__ void __cluster_dims__(kRcCluster, 1, 1) __launch_bounds__(kRcThreads, MAXT * NB <= 2 ? 3 : 2)
router_cluster_kernel(const RouterArgs p) {
  constexpr int kCols = MAXT * 8, kStride = kCols + 8;
  constexpr int kUnr = 16 / (MAXT * NB) >= 2 ? 2 : 1;                // k slices in flight per warp
  constexpr int kPartBytes = 8 * kRcRows * kStride * 4;
  __shared__ __align__(16) uint8_t scratch[kPartBytes > kRcPermBytes ? kPartBytes : kRcPermBytes];
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
  const int n2 = 2 * p.n_rp, n_tiles = n2 >> 3;
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
          w[q][i][nt] = (have && nt < n_tiles) ? __ldg(reinterpret_cast<const uint4*>(wr + (size_t)nt * 8 * p.d)) : zero;
      }
    }
  };
  if (NB == 1) load_w(s0, 0, 1);          // the layer's own rows: fetched while the preceding kernel of the stream drains
  grid_dep_wait();
  grid_dep_trigger();
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
  if (gate_warp) {
    if (NB > 1) go_mine = row_group[my_row];
    if (lane < p.n_r) { u_pre = __ldg(p.u + go_mine * p.n_r + lane); b_pre = __ldg(p.b + go_mine * p.n_r + lane); }
  }
  // ---- partial sums over this warp's k slices
  const int r_lo = min(g, n_rows - 1), r_hi = min(g + 8, n_rows - 1);
  const bf16* x_lo = p.x + (size_t)(row_base + r_lo) * p.d + 8 * t;
  const bf16* x_hi = p.x + (size_t)(row_base + r_hi) * p.d + 8 * t;
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
        a_lo[q] = in ? __ldg(reinterpret_cast<const uint4*>(x_lo + k)) : zero;
        a_hi[q] = in ? __ldg(reinterpret_cast<const uint4*>(x_hi + k)) : zero;
      }
      if (NB > 1 || s != s0) load_w(s, i0, nl);
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
      for (int q = 0; q < kRcCluster; ++q) { a += recv[q][warp][lane]; v += recv[q][warp][p.n_rp + lane]; }
    const size_t row = (size_t)row_base + my_row;
    int sel = 0;
    gate_row_redux(lane, p.n_r, p.n_k, a, v, u_pre, b_pre, go_mine * p.n_r, p.scores + row * p.n_r, p.keys + row * p.n_r,
                   p.topk_idx + row * p.n_k, p.topk_gate + row * p.n_k, sel);
    if (p.fuse_permute && lane < p.n_k) rc_push(rc_peer(&sel_recv[my_row * p.n_k + lane], 0), sel);
  }
  if (!p.fuse_permute) return;
  rc_cluster_arrive();
  rc_cluster_wait();
  if (rank != 0) return;
  // ---- permutation
  uint8_t* sel = scratch;                                             // [n_rows * n_k <= kRcFusePairs]
  int32_t* count = reinterpret_cast<int32_t*>(sel + kRcFusePairs);     // [n_groups], then the exclusive scan
  int32_t* offs = count + kRcFuseGroups;
  uint32_t* mask = reinterpret_cast<uint32_t*>(offs + kRcFuseGroups);
  uint16_t* before = reinterpret_cast<uint16_t*>(mask + kRcFuseGroups * (kRcMaxRows / 32));
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
  permute_by_masks(p, sel, mask, before, count, offs);
}

inline bool router_cluster_fuses(int n_rows, int n_k, int n_groups) {
  return n_groups <= kRcFuseGroups && n_rows <= kRcMaxRows && (long long)n_rows * n_k <= kRcFusePairs;
}

inline cudaError_t router_cluster_launch(const RouterArgs& a, bool hier, bool dep, bool all_smem, cudaStream_t st) {
  const dim3 grid(kRcCluster, (a.n_rows + kRcRows - 1) / kRcRows), block(kRcThreads);
  const int tiles = 2 * a.n_rp / 8;
  if (hier) {
    if (tiles <= 2) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<2, 4>, grid, block, 0, st, a);
    if (tiles <= 4) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<4, 2>, grid, block, 0, st, a);
    return launch_kernel_smem(dep, all_smem, router_cluster_kernel<8, 2>, grid, block, 0, st, a);
  }
  if (tiles <= 2) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<2, 1>, grid, block, 0, st, a);
  if (tiles <= 4) return launch_kernel_smem(dep, all_smem, router_cluster_kernel<4, 1>, grid, block, 0, st, a);
  return launch_kernel_smem(dep, all_smem, router_cluster_kernel<8, 1>, grid, block, 0, st, a);
}

}  // namespace cmoe
