// bf16 routers for large batches: the top-level and the analytical router (Eq. router, Eq. final_gate) on tcgen05 tiles of
// 64 rows, and the permutation that follows them.
//
// The contraction [rows, d] x [d, at most 64] is bound by reading x once; a tile per CTA left most SMs idle and every tile a
// chain of 64 k blocks, partial sums and a ticket through global memory, and a gate stage of one thread per row (a serial
// chain over up to 32 experts).  Here a cluster of 1, 2, 4 or 8 CTAs owns a tile:
//   - every CTA multiplies its slice of k (TMA, tcgen05.mma, sums in tensor memory) and lays its sums out in its shared memory;
//   - after one cluster barrier it adds the slices of its share of the tile's rows in rank order (deterministic) straight
//     from its peers' shared memory and runs their gate logic, one warp per row;
//   - with the selections it writes, per 32 rows and expert, the bit mask of the rows that chose the expert.
// The permutation is then one launch over those masks (population counts; the whole batch's masks are a few ten KB).
// Against 128-row tiles of one to four CTAs with partial sums and tickets in global memory, a gate stage of one thread per row and a
// permutation in two launches: 8B-shaped 2048 rows 241.8 -> 217.8 us, 7B-shaped 269.3 -> 261.3.  Of the 18.5 us from the start to the
// GEMM at 2048 rows of the 8B-shaped layer the contraction takes 5, the sums of the cluster 3, the gates 3, the permutation 5.
#pragma once

#include "permute.cuh"
#include "router.cuh"
#include "router_cluster.cuh"
#include "umma_gemm.cuh"

namespace cmoe {

constexpr int kRtThreads = 256;                // warp 0 TMA, warp 1 MMA, warps 4 and 5 read tensor memory, all eight gate
constexpr int kRtTile = 64;                    // rows of a tile (the multiply takes 128; the upper half is not read back)
constexpr int kRtStages = 6;                   // two CTAs on an SM: alone on theirs, clusters of 8 found no place at once
constexpr int kRtABytes = kRtTile * kUmmaBK * 2;
constexpr int kRtRows = 4;                     // rows whose gate logic a warp runs at once (times 8 warps: one 32-row mask)

struct RouterTileArgs {
  int n_rows, d, n_r, n_rp, n_k, n_cols;       // n_cols: columns of a tile, a multiple of 16; top-level: n_r = outer experts
  int ks;                                      // CTAs of a tile's cluster; the grid's one extent is ks x tiles (2^31 - 1 at most)
  int n_outer;
  const int32_t* outer_off;                    // row ranges of the outer experts, or null (one range [0, n_rows))
  const float *u, *b;
  float *scores, *keys;                        // top-level: scores = logits, topk_gate = weights
  int32_t* topk_idx;
  float* topk_gate;
  uint32_t* words;                             // [2 tile + half][n_r] row masks
  int32_t* err;
};

// Tiles of every outer expert's row range, one expert per lane: lane o < n_outer returns its exclusive
// prefix and the range; `total` takes the sum.
__device__ __forceinline__ int outer_tile_prefix(const int32_t* outer_off, int n_outer, int n_rows, int lane, int& row0, int& count,
                                                 int& total) {
  row0 = 0; count = 0;
  if (lane < n_outer) {
    row0 = outer_off ? __ldcg(outer_off + lane) : 0;
    count = outer_off ? __ldcg(outer_off + lane + 1) - row0 : n_rows;
  }
  const int tiles = (count + kRtTile - 1) / kRtTile;
  int incl = tiles;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  total = __shfl_sync(0xffffffffu, incl, 31);
  return incl - tiles;
}

__device__ __forceinline__ float4 ld_peer4(uint32_t addr, uint32_t rank) {
  float4 v;
  asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %4, %5;\n\tld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [a];\n\t}"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr), "r"(rank) : "memory");
  return v;
}

template <bool OUTER>
__global__ void __launch_bounds__(kRtThreads)
router_tile_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w, const RouterTileArgs p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  __shared__ __align__(8) uint64_t bar_mem[2 * kRtStages + 1];
  __shared__ uint32_t tmem_slot, mask[kRtTile / 32][32];
  __shared__ int abort_mem;
  volatile int* abort_flag = &abort_mem;
  const uint32_t full0 = smem_u32(bar_mem), empty0 = full0 + 8 * kRtStages, accf = full0 + 16 * kRtStages;
  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int ks = p.ks, tile = blockIdx.x / ks, rank = blockIdx.x - tile * ks;
  const uint32_t b_bytes = (uint32_t)p.n_cols * kUmmaBK * 2, stage_bytes = kRtABytes + b_bytes;
  const uint32_t tmem_cols = p.n_cols <= 32 ? 32 : 64;
  const int k_blocks = (p.d + kUmmaBK - 1) / kUmmaBK;
  const int kb_lo = rank * k_blocks / ks, n_kb = (rank + 1) * k_blocks / ks - kb_lo;
  if (threadIdx.x < kRtTile) mask[threadIdx.x >> 5][lane] = 0;
  if (threadIdx.x == 0) {
    for (int s = 0; s < kRtStages; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    mbar_init(accf, 1);
    abort_mem = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(&tmem_slot), tmem_cols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;
  // the layer's own rows (known before the preceding kernel of the stream has ended) go ahead of x
  const int n_early = p.outer_off ? 0 : min(kRtStages, n_kb);
  if (warp == 0) {
#pragma unroll 1
    for (int i = 0; i < n_early; ++i) {
      if (elect_one()) {
        mbar_expect_tx(full0 + 8 * i, stage_bytes);
        tma_load_3d(base + i * stage_bytes + kRtABytes, &tm_w, full0 + 8 * i, (kb_lo + i) * kUmmaBK, 0, 0);
      }
      __syncwarp();
    }
  }
  grid_dep_wait();
  grid_dep_trigger();
  int go = 0, row0, count, total_tiles;
  {
    const int first = outer_tile_prefix(p.outer_off, p.n_outer, p.n_rows, lane, row0, count, total_tiles);
    const uint32_t m = __ballot_sync(0xffffffffu, lane < p.n_outer && first <= tile && count > 0);
    go = m ? 31 - __clz(m) : 0;                                       // the last expert whose tiles begin at or before this one
    const int mt = tile - __shfl_sync(0xffffffffu, first, go);
    row0 = __shfl_sync(0xffffffffu, row0, go) + mt * kRtTile;
    count = min(__shfl_sync(0xffffffffu, count, go) - mt * kRtTile, kRtTile);
  }
  const bool live = tile < total_tiles;                               // the same for the whole cluster
  if (live && warp == 0) {
    // ------------------------------------------------------------ TMA producer
#pragma unroll 1
    for (int i = 0; i < n_kb; ++i) {
      const uint32_t s = i % kRtStages, n = i / kRtStages;
      if (!mbar_wait_warp(empty0 + 8 * s, (n & 1) ^ 1, abort_flag, p.err, kErrWaitEmpty)) {
        for (int w = 0; w < 200; ++w) __nanosleep(1000);              // let copies in flight land
        break;
      }
      const uint32_t fb = full0 + 8 * s, sa = base + s * stage_bytes;
      if (elect_one()) {
        if (i >= n_early) {
          mbar_expect_tx(fb, stage_bytes);
          tma_load_3d(sa + kRtABytes, &tm_w, fb, (kb_lo + i) * kUmmaBK, 0, go);
        }
        tma_load_2d(sa, &tm_x, fb, (kb_lo + i) * kUmmaBK, row0);
      }
      __syncwarp();
    }
  } else if (live && warp == 1) {
    // ------------------------------------------------------------ MMA issuer
    const uint32_t idesc = umma_idesc(p.n_cols);
    bool ok = true;
#pragma unroll 1
    for (int i = 0; i < n_kb; ++i) {
      const uint32_t s = i % kRtStages, n = i / kRtStages;
      if (!mbar_wait_warp(full0 + 8 * s, n & 1, abort_flag, p.err, kErrWaitFull)) { ok = false; break; }
      tc_fence_after();
      const uint32_t sa = base + s * stage_bytes, sb = sa + kRtABytes;   // "rows" 64..127 of A: the bytes that follow
      if (elect_one()) {
#pragma unroll
        for (int k = 0; k < kUmmaBK / 16; ++k)
          umma_bf16(tmem, umma_smem_desc(sa + k * 32), umma_smem_desc(sb + k * 32), idesc, (i != 0 || k != 0) ? 1u : 0u);
        umma_commit(empty0 + 8 * s);
      }
      __syncwarp();
    }
    if (ok && elect_one()) umma_commit(accf);
    __syncwarp();
  } else if (live && (warp == 4 || warp == 5)) {
    // ------------------------------------------------------------ sums to shared memory, over the consumed operands
    if (mbar_wait_warp(accf, 0, abort_flag, p.err, kErrWaitAccFull)) {
      tc_fence_after();
      const int quad = warp & 3;
      float* dst = reinterpret_cast<float*>(gen) + (quad * 32 + lane) * (p.n_cols + 4);
#pragma unroll 1
      for (int c = 0; c < p.n_cols; c += 32) {
        float v[32];
        const bool two = c + 16 < p.n_cols;
        tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + c, v);
        if (two) tmem_ld16(tmem + ((uint32_t)(quad * 32) << 16) + c + 16, v + 16);
        tmem_ld_wait();
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (q < 4 || two) *reinterpret_cast<float4*>(dst + c + 4 * q) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
      }
      tc_fence_before();
    }
  }
  const bool have = lane < p.n_r;
  const float u = !OUTER && have ? __ldcg(p.u + go * p.n_r + lane) : 0.0f, b = !OUTER && have ? __ldcg(p.b + go * p.n_r + lane) : 0.0f;
  rc_cluster_arrive();
  rc_cluster_wait();
  const int per = kRtTile / ks, ld = p.n_cols + 4;
  float* sums = reinterpret_cast<float*>(gen) + rank * per * ld;      // this CTA's rows: no peer reads them here
  // ---- the slices' sums of this CTA's rows (a peer's shared memory is read at about 10 bytes a cycle)
  if (ks > 1) {
#pragma unroll 1
    for (int i = threadIdx.x; i < per * 16; i += kRtThreads) {
      const int r = i >> 4, c = (i & 15) * 4;
      if (c < p.n_cols) {
        const uint32_t at = smem_u32(sums + r * ld + c);
        float4 t = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        float4 v[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) v[q] = q < ks ? ld_peer4(at, q) : t;
#pragma unroll
        for (int q = 0; q < 8; ++q) { t.x += v[q].x; t.y += v[q].y; t.z += v[q].z; t.w += v[q].w; }
        *reinterpret_cast<float4*>(sums + r * ld + c) = t;
      }
    }
  }
  rc_cluster_arrive();                                                // done with the peers' shared memory
  __syncthreads();
  // ---- gate logic: a warp per row, kRtRows rows at a time (their reductions overlap)
#pragma unroll 1
  for (int i0 = warp; live && i0 < per; i0 += 8 * kRtRows) {
    float a[kRtRows], v[kRtRows];
    size_t row[kRtRows];
    bool row_live[kRtRows];
    int sel[kRtRows];
#pragma unroll
    for (int i = 0; i < kRtRows; ++i) {
      const int r = i0 + 8 * i;
      sel[i] = go * p.n_r;
      row[i] = (size_t)row0 + rank * per + r;
      row_live[i] = r < per && rank * per + r < count;
      a[i] = row_live[i] && have ? sums[r * ld + lane] : 0.0f;
      v[i] = !OUTER && row_live[i] && have ? sums[r * ld + p.n_rp + lane] : 0.0f;
    }
    if (OUTER) {
#pragma unroll
      for (int i = 0; i < kRtRows; ++i)
        if (row_live[i])
          outer_row_redux(lane, p.n_r, p.n_k, a[i], p.scores + row[i] * p.n_r, p.topk_idx + row[i] * p.n_k, p.topk_gate + row[i] * p.n_k, sel[i]);
    } else {
      gate_rows_redux<kRtRows>(lane, p.n_r, p.n_k, a, v, u, b, go * p.n_r, row, row_live, p.scores, p.keys, p.topk_idx, p.topk_gate, sel);
    }
    uint32_t mine = 0;                                                // lane = expert: which of these rows chose it
#pragma unroll
    for (int i = 0; i < kRtRows; ++i) {
      const uint32_t m = __reduce_or_sync(0xffffffffu, row_live[i] && lane < p.n_k ? 1u << (sel[i] - go * p.n_r) : 0u);
      mine |= ((m >> lane) & 1u) << ((i0 + 8 * i) & 31);
    }
    if (mine) atomicOr(&mask[i0 >> 5][lane], mine);                   // kRtRows * 8 = 32: the batch lies in one chunk
  }
  __syncthreads();
  // ---- row masks per expert
  if (live && warp * 32 < per && lane < p.n_r) {
    const uint32_t m = mask[warp][lane];
    uint32_t* dst = p.words + (size_t)(tile * 2 + (rank * per >> 5) + warp) * p.n_r + lane;
    if (per >= 32) *dst = m;
    else if (per == 16) reinterpret_cast<uint16_t*>(dst)[rank & 1] = (uint16_t)m;
    else reinterpret_cast<uint8_t*>(dst)[rank & 3] = (uint8_t)m;
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, tmem_cols);
  }
  rc_cluster_wait();                                                  // no CTA leaves while a peer still reads its sums
}

// Permutation of a batch from the row masks of router_tile_kernel: a block places 8 chunks of 32 rows and counts the masks of
// all chunks itself.
constexpr int kWordsMax = 32768;               // masks of a batch (every block reads them: 128 KB at most)
inline int router_tile_count(int n_rows, int n_outer) { return (n_rows + kRtTile - 1) / kRtTile + (n_outer > 1 ? n_outer - 1 : 0); }
inline size_t router_tile_words(int n_rows, int n_r, int n_outer) { return (size_t)2 * router_tile_count(n_rows, n_outer) * n_r; }

__global__ void __launch_bounds__(256)
permute_words_kernel(const uint32_t* __restrict__ words, const int32_t* __restrict__ topk_idx, int n_r, int n_outer,
                     const int32_t* __restrict__ outer_off, const PermuteOut p) {
  extern __shared__ int32_t sm[];
  int32_t* total = sm;                         // [G], then the exclusive scan
  int32_t* before = total + p.n_groups;        // [G] rows in chunks ahead of this block's
  __shared__ uint32_t bw[8][32];
  __shared__ int32_t bo[8], c_start[33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c0 = blockIdx.x * 8, c = c0 + warp;
#pragma unroll 1
  for (int g = threadIdx.x; g < 2 * p.n_groups; g += 256) sm[g] = 0;
  grid_dep_trigger();                          // the gate/up GEMM may start on what needs no permutation
  grid_dep_wait();
  int row0, count, total_tiles;
  const int first = outer_tile_prefix(outer_off, n_outer, p.n_rows, lane, row0, count, total_tiles);
  if (c0 >= total_tiles * 2 && blockIdx.x != 0) return;
  const bool live = c < total_tiles * 2;
  const uint32_t m = __ballot_sync(0xffffffffu, lane < n_outer && first <= (c >> 1) && count > 0);
  const int go = m ? 31 - __clz(m) : 0;
  const int in_group = (c - 2 * __shfl_sync(0xffffffffu, first, go)) * 32 + lane;
  const int row = __shfl_sync(0xffffffffu, row0, go) + in_group;
  const bool row_ok = live && in_group < __shfl_sync(0xffffffffu, count, go);
  int sel[kMaxTopK];
#pragma unroll
  for (int j = 0; j < kMaxTopK; ++j) sel[j] = row_ok && j < p.n_k ? __ldcg(topk_idx + (size_t)row * p.n_k + j) : -1;
  if (lane < n_r) bw[warp][lane] = live ? __ldcg(words + (size_t)c * n_r + lane) : 0u;
  if (lane == 0) bo[warp] = go;
  if (warp == 0) {
    c_start[lane] = 2 * first;
    if (lane == 0) c_start[32] = 2 * total_tiles;
  }
  __syncthreads();
  // ---- counts: thread = (expert of an outer expert, slice of its chunks)
  const int slices = 256 / n_r, sl = threadIdx.x / n_r, gl = threadIdx.x - sl * n_r;
  if (sl < slices) {
#pragma unroll 1
    for (int o = 0; o < n_outer; ++o) {
      const int end = c_start[o + 1 < 32 ? o + 1 : 32];
      int all = 0, ahead = 0;
#pragma unroll 1
      for (int cc = c_start[o] + sl; cc < end; cc += 8 * slices) {    // eight loads in flight
        uint32_t w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = cc + q * slices < end ? __ldcg(words + (size_t)(cc + q * slices) * n_r + gl) : 0u;
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          all += __popc(w[q]);
          ahead += cc + q * slices < c0 ? __popc(w[q]) : 0;
        }
      }
      if (all) atomicAdd(&total[o * n_r + gl], all);
      if (ahead) atomicAdd(&before[o * n_r + gl], ahead);
    }
  }
  __syncthreads();
  if (warp == 0) {                                                    // exclusive scan over the groups
    const int each = (p.n_groups + 31) / 32, lo = lane * each, hi = min(lo + each, p.n_groups);
    int sum = 0;
    for (int g = lo; g < hi; ++g) sum += total[g];
    int incl = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int up = __shfl_up_sync(0xffffffffu, incl, o);
      if (lane >= o) incl += up;
    }
    int run = incl - sum;
    for (int g = lo; g < hi; ++g) {
      const int n = total[g];
      before[g] += run;
      if (blockIdx.x == 0) {
        p.counts[g] = n;
        p.offsets[g] = run;
        if (p.po.gr) { GroupRows r; r.row0 = run; r.count = n; p.po.gr[p.po.n_outer + g] = r; }
      }
      run += n;
    }
    if (blockIdx.x == 0 && lane == 31) p.offsets[p.n_groups] = incl;
  } else if (warp == 1 && blockIdx.x == 0 && p.po.gr && lane < p.po.n_outer) {
    GroupRows r; r.row0 = row0; r.count = count;
    p.po.gr[lane] = r;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kMaxTopK; ++j) {
    if (sel[j] < 0) continue;
    const int l = sel[j] - go * n_r;
    int pos = before[sel[j]] + __popc(bw[warp][l] & ((1u << lane) - 1u));
#pragma unroll
    for (int w = 0; w < 7; ++w) pos += (w < warp && bo[w] == go) ? __popc(bw[w][l]) : 0;
    p.row_token[pos] = row;
    p.row_of[(size_t)row * p.n_k + j] = pos;
  }
}

// ----------------------------------------------------------------------------- host
// Rows from which this router is the better one (below: router_cluster_kernel, whose 16-row tiles each read all representative
// rows).  Whole forwards with either router, cluster / tiles: more than 16 columns, 8B-shaped 500 / 600 / 700 / 850 rows 103 / 115 / 111 /
// 129 against 103 / 108 / 103 / 119 us, 13B-shaped 600 rows 154 against 149; 16 columns, 7B-shaped 500 / 700 / 850 / 1000 rows 91 / 108 / 133 / 158
// against 89 / 108 / 135 / 147: even up to 850.  Outer rows: the clustered router copies them as well.
inline bool router_takes_tiles(int n_rows, int n_rp, bool hier) { return n_rows > (!hier && n_rp > 8 ? 512 : kRcMaxRows); }

inline cudaError_t router_tile_allow() {
  const int most = 1024 + kRtStages * (kRtABytes + 64 * kUmmaBK * 2) + kRtABytes;
  const cudaError_t e = allow_smem(router_tile_kernel<false>, most);
  return e == cudaSuccess ? allow_smem(router_tile_kernel<true>, most) : e;
}

// Top-level router rows [n_outer, d]: box of 64 k x n_cols rows (rows past n_outer are zero-filled).
inline bool router_tile_encode_outer(UmmaPlan* P, CUtensorMap* tm, const void* w, int n_outer, int d, int n_cols) {
  const cuuint64_t dims[3] = {(cuuint64_t)d, (cuuint64_t)n_outer, 1};
  const cuuint64_t str[2] = {(cuuint64_t)d * 2, (cuuint64_t)n_outer * d * 2};
  const cuuint32_t box[3] = {kUmmaBK, (cuuint32_t)n_cols, 1};
  return umma_encode(P, tm, w, 3, dims, str, box, "top-level router");
}

// Router and permutation; a.words holds router_tile_words(n_rows, n_r, n_outer) masks.  Returns launches, or -1.
template <bool OUTER>
inline int router_tile_forward(const CUtensorMap& tm_x, const CUtensorMap& tm_w, RouterTileArgs a, PermuteOut out, int32_t* scratch,
                               int n_sms, bool dep, cudaStream_t st, cudaEvent_t mid = nullptr) {
  // CTAs per tile: as many as keep the grid within one wave of two CTAs per SM, and two k blocks each
  const int tiles = router_tile_count(a.n_rows, a.n_outer), kb = (a.d + kUmmaBK - 1) / kUmmaBK;
  int ks = 8;
  while (ks > 1 && (tiles * ks > 2 * n_sms || 2 * ks > kb)) ks >>= 1;
  cudaLaunchConfig_t cfg = {};
  a.ks = ks;
  cfg.gridDim = dim3(ks * tiles); cfg.blockDim = dim3(kRtThreads); cfg.stream = st;
  cfg.dynamicSmemBytes = 1024 + (size_t)kRtStages * (kRtABytes + a.n_cols * kUmmaBK * 2) + kRtABytes /* read past the last A */;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = ks; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = dep ? 2 : 1;
  if (cudaLaunchKernelEx(&cfg, router_tile_kernel<OUTER>, tm_x, tm_w, (const RouterTileArgs)a) != cudaSuccess) return -1;
  if (mid) cudaEventRecord(mid, st);
  if (router_tile_words(a.n_rows, a.n_r, a.n_outer) > kWordsMax)
    return 1 + launch_token_permute(a.topk_idx, a.n_rows, a.n_k, out.n_groups, out.counts, out.offsets, out.row_token, out.row_of,
                                    scratch, st, out.po, dep);
  const cudaError_t e = launch_kernel(dep, permute_words_kernel, dim3((2 * tiles + 7) / 8), dim3(256), 2 * out.n_groups * sizeof(int32_t),
                                      st, (const uint32_t*)a.words, (const int32_t*)a.topk_idx, a.n_r, a.n_outer, a.outer_off, out);
  return e == cudaSuccess ? 2 : -1;
}

}  // namespace cmoe
