// Expert FFN of a plain layer for small batches: two weight streamers that read every active weight once and write the
// layer's output themselves (no partial outputs per expert, no combine kernel).
//
// Bound: HBM, the active experts' weight bytes.  Weight rows sit on the M side of the tcgen05 MMA, tokens on the N side,
// so the tensor core takes 160-400 cycles of the ~900 that an SM's share of the DRAM stream leaves for a block.
//
//   stream_up_kernel:   a tile is `tile_rows` neurons of one group (gate and up rows, two accumulators); it is computed for
//       ALL rows of the batch, and the epilogue writes gate * Swish(g . x) * (u . x) (Eq. ori_ffn_method, Eq. final_gate) for
//       the tokens that selected the expert and 0 for the others, into one dense matrix Hd [rows][d_ff].  The tile height is
//       chosen per launch so that the expected tiles fill whole rounds of the SMs.
//   stream_down_kernel: out[t, c] = sum over the active groups' neurons of W_down[c, n] Hd[t, n] (Eq. moe_output): with
//       the gates folded into Hd the sum over experts is part of the contraction, a tile is 128 output channels and its K range
//       runs through all active groups.  The 64-wide k blocks of all tiles are numbered through and every CTA takes an equal
//       run; a tile that spans several CTAs leaves fp32 partial sums in scratch, each epilogue warp takes a ticket for its
//       part, and the one with the last ticket adds the parts in CTA order (a fixed order: deterministic).  Nothing ever
//       waits for another CTA.
//
// What the up kernel needs of the router is only the epilogue's gates when (nearly) every expert is expected to be active
// (`dense`): then it streams from its first cycle, under the router's latency.  Otherwise the shared expert's tiles go
// first and the routed ones follow once the router is done.  The down kernel fetches its first ring of weights before it
// waits for the up kernel.
//
// W8 = true streams FP8 (E4M3) codes, half the bytes, into kind::f8f6f4 MMAs.  The token rows are E4M3 planes hi and lo (see
// split_rows_e4m3_kernel), both multiplied by one MMA (N = 2 x token rows); the planes of x are written ahead of the router,
// those of Hd by a split launch between the two kernels.  The scales of a down weight row and of a token's Hd differ from expert
// to expert, so the down kernel accumulates one group at a time and its epilogue adds them up in registers.
//
// Registers and shared memory are sized so that the router, the up and the down kernel fit one SM
// pairwise: otherwise the successor's CTAs start when the predecessor's end, and the streams pause in between.  Loops
// whose trip count is not fixed are not unrolled: the weight streams push the code out of L2 between two forwards, and
// every line of it that a short kernel needs is a miss to DRAM.
//
// Against the kernels of umma_decode.cuh followed by the combine kernel (cmoe_layer_set_gemm_path 0 / 2, chained forwards): 7B-shaped layer
// 2 / 16 / 64 rows 50.8 / 53.9 / 63.1 against 52.1 / 58.4 / 64.8 us, 8B-shaped 4 / 32 / 64 rows 48.5 / 69.5 / 75.3 against 51.8 / 78.7 / 81.5,
// 13B-shaped 16 / 64 rows 76.5 / 88.8 against 87.2 / 94.3; FP8 weights, 7B-shaped 2 / 16 / 48 rows 36.8 / 38.8 / 47.0 against 37.8 / 45.6 /
// 58.6, 8B-shaped 8 / 32 / 64 rows 44.2 / 50.6 / 58.9 against 50.0 / 69.2 / 83.0, 13B-shaped 16 / 48 rows 52.5 / 60.7 against 64.4 / 83.2.
// In a forward of 16 rows of the 7B-shaped layer (270 MB of weights, 42 us at the copy rate) the up kernel streams for 31 us from its start
// under the router, its slowest CTA and the hand-over cost 4, the down kernel streams for 13 and its sums take 3.  (The sums are one chain of latencies: stores,
// release, ticket, loads.  With a fence per lane beside lane 0's release and six of seven contributions in flight 16 rows took 56.1
// instead of 55.4 us, 8B-shaped 32 rows 69.8 instead of 69.3.)  A single row stays on the
// CUDA-core kernels of gemv.cuh (30.6 us against 42.3).  Fetching the down kernel's weights into L2 at the end of the up kernel was slower
// (it delays the up kernel's last CTAs), equal runs of k blocks instead of tiles in the up kernel as well (the partial sums).
#pragma once

#include <cmath>

#include "fp8.cuh"
#include "umma_gemm.cuh"

namespace cmoe {

constexpr int kStreamThreads = 320;          // warp 0 TMA, warp 1 MMA, warps 2..9 epilogue (two per TMEM quadrant)
constexpr int kStreamMaxRows = 64;
constexpr int kStreamMaxGrid = 160;
constexpr int kStreamMinRun = 4;             // k blocks a CTA of the down kernel takes at least
constexpr int kStreamUnselected = 0x7fc0dead;  // a NaN that no computed gate has: the token did not select the expert
constexpr int kStreamTail = 512;             // barriers and the active list in front of the ring

struct StreamArgs {
  const GroupRows* gr;         // row ranges of the groups (written by the router / permutation): which are active
  int has_s, n_r, n_k;
  int n_rows, d, shared_w, m;
  int dense;                   // up: every routed expert is treated as active
  int tile_rows;               // up: neurons per tile (a multiple of 8)
  int tok_rows;                // rows of the token boxes: n_rows rounded up to 16
  int stages;
  const int32_t* topk_idx;     // [rows][n_k] selected routed expert
  const float* topk_gate;
  bf16* h;                     // Hd
  int ld_h;
  bf16* out;                   // down: [rows][d]
  float* part;                 // down: [2 * CTAs] slots of 128 x NT fp32
  int32_t* ticket;             // down: [tiles][8], zero between launches
  int32_t* err;
  // FP8 weights: power-of-two scales of the token planes and of the weight rows
  const float* tok_scale;      // up: [rows] of x; down: [1 + n_r][kStreamMaxRows] of Hd
  const float* scale_gu;       // [2][rows_w]: gate plane, then up plane, packed neuron order
  const float* scale_d;        // [1 + n_r][d]: per group and output channel
  long long rows_w;
};

__device__ __forceinline__ int atom_inc_acq_rel(int32_t* p) {
  int v;
  asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// 8 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float* v) {
  uint32_t r[8];
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// Active routed experts, ascending, by one warp.
__device__ __forceinline__ void stream_list_active(const StreamArgs& p, bool all, int* active, int* n_active) {
  const int lane = threadIdx.x & 31;
  const bool on = lane < p.n_r && p.n_k > 0 && (all || __ldcg(&p.gr[1 + lane].count) > 0);
  const uint32_t mask = __ballot_sync(0xffffffffu, on);
  if (on) active[__popc(mask & ((1u << lane) - 1u))] = lane;
  if (lane == 0) *n_active = __popc(mask);
  __syncwarp();
}

// Position in the ring: stage index and the parity of its barriers.
struct RingPos {
  int s = 0;
  uint32_t ph = 0;
  __device__ __forceinline__ void next(int stages) { if (++s == stages) { s = 0; ph ^= 1; } }
};

// Place in the down kernel's work: tile, group (-1 shared, else index into the active list), k block inside the group.
struct StreamCursor { int tile, a, kk; };
// The down kernel's work: the k blocks of all tiles in one row, dealt to the first n_ctas CTAs in equal runs.
struct StreamRun {
  int kb_s, kb_m, n_act, kb_tile, blocks, n_ctas;
  __device__ __forceinline__ StreamRun(const StreamArgs& p, int n_active, int bk) {
    kb_s = p.has_s ? (p.shared_w + bk - 1) / bk : 0;
    kb_m = (p.m + bk - 1) / bk;
    n_act = n_active;
    kb_tile = kb_s + n_act * kb_m;
    blocks = kb_tile * ((p.d + 127) / 128);
    n_ctas = min((int)gridDim.x, max(blocks / kStreamMinRun, 1));
  }
  __device__ __forceinline__ int lo(int cta) const { return cta >= n_ctas ? blocks : (int)((long long)cta * blocks / n_ctas); }
  __device__ __forceinline__ int cta_of(int block) const { return (int)(((long long)(block + 1) * n_ctas - 1) / blocks); }
  __device__ __forceinline__ StreamCursor cursor(int b) const {
    StreamCursor c;
    c.tile = b / kb_tile;
    const int kb = b - c.tile * kb_tile;
    if (kb < kb_s) { c.a = -1; c.kk = kb; } else { c.a = (kb - kb_s) / kb_m; c.kk = kb - kb_s - c.a * kb_m; }
    return c;
  }
  __device__ __forceinline__ int group_end(int tile_b0, int b) const {    // end of the group that block b of a tile belongs to
    const int kb = b - tile_b0;
    return tile_b0 + (kb < kb_s ? kb_s : kb_s + ((kb - kb_s) / kb_m + 1) * kb_m);
  }
  __device__ __forceinline__ void advance(StreamCursor& c) const {
    if (++c.kk == (c.a < 0 ? kb_s : kb_m)) {
      c.kk = 0;
      if (++c.a == n_act) { c.a = kb_s > 0 ? -1 : 0; ++c.tile; }
    }
  }
};

template <int NT, bool W8>
__global__ void __maxnreg__(96)
stream_up_kernel(const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_x, const StreamArgs p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* tail = smem_raw + (base - raw);                  // in front of the ring: the MMAs read up to 16 KB past a tile
  // full[8] empty[8] acc_full[2] acc_empty[2] table, TMEM slot, abort flag, active count; active list; gate tables
  const uint32_t full0 = base, empty0 = base + 64, accf0 = base + 128, acce0 = base + 144, tbl_bar = base + 160;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 168);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 172);
  int* n_active = reinterpret_cast<int*>(tail + 176);
  int* active = reinterpret_cast<int*>(tail + 192);             // [32]
  float* gate_tables = reinterpret_cast<float*>(tail + kStreamTail);    // [8 warps][NT]
  const uint32_t ring = base + (kStreamTail + 8 * NT * 4 + 1023) / 1024 * 1024;
  const int h = p.tile_rows, stages = p.stages;
  const uint32_t plane = h * 128, stage_bytes = 2 * plane + (W8 ? 2 : 1) * p.tok_rows * 128;
  constexpr int kBK = W8 ? 2 * kUmmaBK : kUmmaBK;              // k per stage: 128 bytes of a weight row
  constexpr int kAcc = (W8 ? 2 : 1) * NT;                       // columns of one accumulator
  constexpr int kBufs = 2 * 2 * kAcc > 256 ? 1 : 2;             // the down kernel's 256 columns have to fit as well
  constexpr int kTmemCols = kBufs * 2 * kAcc < 32 ? 32 : kBufs * 2 * kAcc;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int s = 0; s < 8; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf0 + 8 * b, 1); mbar_init(acce0 + 8 * b, 8); }
    mbar_init(tbl_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  if (warp == 0 && p.dense) stream_list_active(p, true, active, n_active);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int n_ctas = gridDim.x;
  const int k_blocks = (p.d + kBK - 1) / kBK;
  const int tiles_s = p.has_s ? (p.shared_w + h - 1) / h : 0, tiles_m = (p.m + h - 1) / h;
  // group of a tile: -1 the shared expert, else a routed expert; first neuron inside the group; its weight row
  struct Tile { int j, n0, width, w_row0; };
  auto tile_of = [&](int t) {
    Tile r;
    if (t < tiles_s) { r.j = -1; r.n0 = t * h; r.width = p.shared_w; r.w_row0 = 0; }
    else {
      const int a = (t - tiles_s) / tiles_m;
      r.j = active[a]; r.n0 = (t - tiles_s - a * tiles_m) * h; r.width = p.m;
      r.w_row0 = (p.has_s ? p.shared_w : 0) + r.j * p.m;
    }
    return r;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
    RingPos rp;
    bool ok = true, listed = p.dense != 0;
    int total = listed ? tiles_s + *n_active * tiles_m : tiles_s;
#pragma unroll 1
    for (int t = blockIdx.x; ok; t += n_ctas) {
      if (t >= total) {
        if (listed) break;
        grid_dep_wait();                                  // the router is done: list the active experts
        stream_list_active(p, false, active, n_active);
        if (lane == 0) mbar_arrive(tbl_bar);
        __syncwarp();
        listed = true;
        total = tiles_s + *n_active * tiles_m;
        if (t >= total) break;
      }
      const Tile tl = tile_of(t);
      const int row = tl.w_row0 + tl.n0;
#pragma unroll 1
      for (int kb = 0; kb < k_blocks; ++kb, rp.next(stages)) {
        if (!mbar_wait_warp(empty0 + 8 * rp.s, rp.ph ^ 1, abort_flag, p.err, kErrWaitEmpty)) { ok = false; break; }
        if (elect_one()) {
          const uint32_t fb = full0 + 8 * rp.s, sw = ring + rp.s * stage_bytes;
          mbar_expect_tx(fb, stage_bytes);
          tma_load_3d(sw, &tm_w, fb, kb * kBK, row, 0);              // gate rows, then the up rows behind them
          if (W8) tma_load_3d(sw + 2 * plane, &tm_x, fb, kb * kBK, 0, 0);        // hi rows, then the lo rows
          else tma_load_2d(sw + 2 * plane, &tm_x, fb, kb * kBK, 0);
        }
        __syncwarp();
      }
    }
    if (!ok) for (int i = 0; i < 200; ++i) __nanosleep(1000);             // let copies in flight land
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (whole warp, one lane issues)
    const uint32_t idesc = W8 ? umma_idesc_e4m3(2 * p.tok_rows) : umma_idesc(p.tok_rows);
    RingPos rp;
    uint32_t seg = 0;
    bool ok = true, listed = p.dense != 0;
    int total = listed ? tiles_s + *n_active * tiles_m : tiles_s;
#pragma unroll 1
    for (int t = blockIdx.x; ok; t += n_ctas, ++seg) {
      if (t >= total) {
        if (listed || !mbar_wait_warp(tbl_bar, 0, abort_flag, p.err, kErrWaitFull)) break;
        listed = true;
        total = tiles_s + *n_active * tiles_m;
        if (t >= total) break;
      }
      const uint32_t buf = seg % kBufs, use = seg / kBufs;
      if (!mbar_wait_warp(acce0 + 8 * buf, (use & 1) ^ 1, abort_flag, p.err, kErrWaitAccEmpty)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + buf * 2 * kAcc;
#pragma unroll 1
      for (int kb = 0; kb < k_blocks; ++kb, rp.next(stages)) {
        if (!mbar_wait_warp(full0 + 8 * rp.s, rp.ph, abort_flag, p.err, kErrWaitFull)) { ok = false; break; }
        tc_fence_after();
        const uint32_t sw = ring + rp.s * stage_bytes;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const uint32_t acc = (kb != 0 || k != 0) ? 1u : 0u;
            const uint64_t x_desc = umma_smem_desc(sw + 2 * plane + k * 32);
            if (W8) {
              umma_e4m3(d_tmem, umma_smem_desc(sw + k * 32), x_desc, idesc, acc);
              umma_e4m3(d_tmem + kAcc, umma_smem_desc(sw + plane + k * 32), x_desc, idesc, acc);
            } else {
              umma_bf16(d_tmem, umma_smem_desc(sw + k * 32), x_desc, idesc, acc);
              umma_bf16(d_tmem + kAcc, umma_smem_desc(sw + plane + k * 32), x_desc, idesc, acc);
            }
          }
          umma_commit(empty0 + 8 * rp.s);
        }
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(accf0 + 8 * buf);
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..9)
    const int quad = warp & 3, half = (warp - 2) >> 2;              // 8-column chunks half, half + 2, ...
    float* gate = gate_tables + (warp - 2) * NT;
    grid_dep_wait();                                  // the router's results are final: the down kernel may become
    grid_dep_trigger();                               // resident and list the active experts
    float ts_lo = 1.0f, ts_hi = 1.0f;                 // W8: this lane's token scales
    if (W8 && lane < p.n_rows) ts_lo = __ldcg(p.tok_scale + lane);
    if (W8 && lane + 32 < p.n_rows) ts_hi = __ldcg(p.tok_scale + lane + 32);
    bool ok = true, listed = p.dense != 0;
    int total = listed ? tiles_s + *n_active * tiles_m : tiles_s;
    uint32_t seg = 0;
#pragma unroll 1
    for (int t = blockIdx.x; ok; t += n_ctas, ++seg) {
      if (t >= total) {
        if (listed || !mbar_wait_warp(tbl_bar, 0, abort_flag, p.err, kErrWaitFull)) break;
        listed = true;
        total = tiles_s + *n_active * tiles_m;
        if (t >= total) break;
      }
      const Tile tl = tile_of(t);
      if (tl.j >= 0) {                                // this expert's gate per token
        __syncwarp();
#pragma unroll 1
        for (int c = lane; c < p.n_rows; c += 32) {
          float g = __int_as_float(kStreamUnselected);
#pragma unroll 1
          for (int k = 0; k < p.n_k; ++k)
            if (__ldcg(p.topk_idx + c * p.n_k + k) == tl.j) g = __ldcg(p.topk_gate + c * p.n_k + k);
          gate[c] = g;
        }
        __syncwarp();
      }
      const int r = quad * 32 + lane, nn = tl.n0 + r;
      const bool live = r < h && nn < tl.width;
      float sc_a = 1.0f, sc_u = 1.0f;                 // W8: scales of this thread's weight rows
      if (W8 && live) {
        sc_a = __ldg(p.scale_gu + tl.w_row0 + nn);
        sc_u = __ldg(p.scale_gu + p.rows_w + tl.w_row0 + nn);
      }
      bf16* dst = p.h + tl.w_row0 + nn;
      const uint32_t buf = seg % kBufs, use = seg / kBufs;
      if (!mbar_wait_warp(accf0 + 8 * buf, use & 1, abort_flag, p.err, kErrWaitAccFull)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + buf * 2 * kAcc + ((uint32_t)(quad * 32) << 16);
      const bool routed = tl.j >= 0;
#pragma unroll 1
      for (int c0 = 8 * half; c0 < p.n_rows; c0 += 16) {
        float a[8], u[8];
        tmem_ld8(taddr + c0, a);
        tmem_ld8(taddr + kAcc + c0, u);
        if constexpr (W8) {                           // (hi + lo / 16) x weight row scale x token scale
          float al[8], ul[8];
          tmem_ld8(taddr + p.tok_rows + c0, al);
          tmem_ld8(taddr + kAcc + p.tok_rows + c0, ul);
          tmem_ld_wait();
#pragma unroll
          for (int q = 0; q < 8; ++q) {
            const float ts = __shfl_sync(0xffffffffu, c0 < 32 ? ts_lo : ts_hi, (c0 + q) & 31);
            a[q] = fmaf(al[q], 0.0625f, a[q]) * (sc_a * ts);
            u[q] = fmaf(ul[q], 0.0625f, u[q]) * (sc_u * ts);
          }
        } else {
          tmem_ld_wait();
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          a[q] = swiglu_fast(a[q], u[q]);
          if (routed) {
            const float g = gate[c0 + q];
            a[q] = __float_as_int(g) == kStreamUnselected ? 0.0f : g * a[q];
          }
        }
        if (live) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            if (c0 + q < p.n_rows) dst[(size_t)(c0 + q) * p.ld_h] = __float2bfloat16_rn(a[q]);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(acce0 + 8 * buf);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

template <int NT, bool W8>
__global__ void __maxnreg__(104)
stream_down_kernel(const __grid_constant__ CUtensorMap tm_w_s, const __grid_constant__ CUtensorMap tm_w_r,
                   const __grid_constant__ CUtensorMap tm_h_s, const __grid_constant__ CUtensorMap tm_h_r,
                   const StreamArgs p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* tail = smem_raw + (base - raw);
  const uint32_t full0 = base, empty0 = base + 64, accf0 = base + 128, acce0 = base + 144;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(tail + 168);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tail + 172);
  int* n_active = reinterpret_cast<int*>(tail + 176);
  int* active = reinterpret_cast<int*>(tail + 192);             // [32]
  const uint32_t ring = base + (W8 ? 2048 : 1024);              // W8: [8 warps][32] token scales in between
  const int stages = p.stages;
  constexpr uint32_t kWBytes = 128 * 128;
  const uint32_t stage_bytes = kWBytes + (W8 ? 2 : 1) * p.tok_rows * 128;
  constexpr int kBK = W8 ? 2 * kUmmaBK : kUmmaBK;
  constexpr int kAcc = (W8 ? 2 : 1) * NT;
  constexpr int kTmemCols = 2 * kAcc < 32 ? 32 : 2 * kAcc;

  const int warp = warp_index(), lane = threadIdx.x & 31;
  if (threadIdx.x == 0) {
#pragma unroll 1
    for (int s = 0; s < 8; ++s) { mbar_init(full0 + 8 * s, 1); mbar_init(empty0 + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf0 + 8 * b, 1); mbar_init(acce0 + 8 * b, 8); }
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), kTmemCols);
    tmem_relinquish();
  }
  // the up kernel lets this one start only after the router is done: the counts are final
  if (warp == 0) stream_list_active(p, false, active, n_active);
  grid_dep_trigger();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  const int cta = blockIdx.x;
  const StreamRun run(p, *n_active, kBK);
  const int kb_tile = run.kb_tile, lo = run.lo(cta), hi = run.lo(cta + 1);

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
    auto load_weights = [&](int s, const StreamCursor& c) {
      const uint32_t fb = full0 + 8 * s, sw = ring + s * stage_bytes;
      if (c.a < 0) tma_load_3d(sw, &tm_w_s, fb, c.kk * kBK, c.tile * 128, 0);
      else tma_load_4d(sw, &tm_w_r, fb, c.kk * kBK, c.tile * 128, active[c.a], 0);
    };
    auto load_tokens = [&](int s, const StreamCursor& c) {
      const uint32_t fb = full0 + 8 * s, st = ring + s * stage_bytes + kWBytes;
      if (W8) {                                       // hi rows, then the lo rows
        if (c.a < 0) tma_load_3d(st, &tm_h_s, fb, c.kk * kBK, 0, 0);
        else tma_load_4d(st, &tm_h_r, fb, c.kk * kBK, active[c.a], 0, 0);
      } else {
        if (c.a < 0) tma_load_2d(st, &tm_h_s, fb, c.kk * kBK, 0);
        else tma_load_3d(st, &tm_h_r, fb, c.kk * kBK, active[c.a], 0);
      }
    };
    bool ok = true;
    const int ahead = min(stages, hi - lo);
    if (ahead > 0) {
      StreamCursor c = run.cursor(lo), c2 = c;
#pragma unroll 1
      for (int i = 0; i < ahead; ++i, run.advance(c)) {                       // the first ring of weights needs nothing
        if (elect_one()) { mbar_expect_tx(full0 + 8 * i, stage_bytes); load_weights(i, c); }
        __syncwarp();
      }
      grid_dep_wait();                                                    // Hd is complete
#pragma unroll 1
      for (int i = 0; i < ahead; ++i, run.advance(c2)) {
        if (elect_one()) load_tokens(i, c2);
        __syncwarp();
      }
      RingPos rp;
      rp.ph = 1;
#pragma unroll 1
      for (int b = lo + ahead; b < hi; ++b, run.advance(c), rp.next(stages)) {
        if (!mbar_wait_warp(empty0 + 8 * rp.s, rp.ph ^ 1, abort_flag, p.err, kErrWaitEmpty)) { ok = false; break; }
        if (elect_one()) {
          mbar_expect_tx(full0 + 8 * rp.s, stage_bytes);
          load_weights(rp.s, c);
          load_tokens(rp.s, c);
        }
        __syncwarp();
      }
    }
    if (!ok) for (int i = 0; i < 200; ++i) __nanosleep(1000);             // let copies in flight land
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (whole warp, one lane issues)
    const uint32_t idesc = W8 ? umma_idesc_e4m3(2 * p.tok_rows) : umma_idesc(p.tok_rows);
    RingPos rp;
    uint32_t seg = 0;
    bool ok = true;
#pragma unroll 1
    for (int b = lo; b < hi && ok; ++seg) {
      const int tile_b0 = b / kb_tile * kb_tile;
      int end = min(hi, tile_b0 + kb_tile);
      if (W8) end = min(end, run.group_end(tile_b0, b));          // scales differ from group to group: one accumulation each
      const uint32_t buf = seg & 1, use = seg >> 1;
      if (!mbar_wait_warp(acce0 + 8 * buf, (use & 1) ^ 1, abort_flag, p.err, kErrWaitAccEmpty)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + buf * kAcc;
      uint32_t acc = 0;
#pragma unroll 1
      for (; b < end; ++b, rp.next(stages)) {
        if (!mbar_wait_warp(full0 + 8 * rp.s, rp.ph, abort_flag, p.err, kErrWaitFull)) { ok = false; break; }
        tc_fence_after();
        const uint32_t sw = ring + rp.s * stage_bytes;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < 4; ++k)
            (W8 ? umma_e4m3 : umma_bf16)(d_tmem, umma_smem_desc(sw + k * 32), umma_smem_desc(sw + kWBytes + k * 32), idesc,
                                         k == 0 ? acc : 1u);
          umma_commit(empty0 + 8 * rp.s);
        }
        __syncwarp();
        acc = 1;
      }
      if (ok && elect_one()) umma_commit(accf0 + 8 * buf);
      __syncwarp();
    }
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..9)
    const int quad = warp & 3, half = (warp - 2) >> 2;              // 8-column chunks half, half + 2, ...
    const int slot_q = quad * 32 + lane;
    constexpr int kCh = NT / 16;                                    // this warp's chunks: columns 16 i + 8 half
    constexpr int kSum = W8 && NT == 64 ? 6 : 7;                    // contributions in flight: 4096 channels on 148 SMs have 6 or 7 (registers)
    float* tok_sc = reinterpret_cast<float*>(tail + 1024) + 32 * (warp - 2);
    grid_dep_wait();                                                // also orders this kernel's stores to `out`
    bool ok = true;
    uint32_t seg = 0;
#pragma unroll 1
    for (int b = lo; b < hi && ok;) {
      const int tile = b / kb_tile, tile_b0 = tile * kb_tile;
      const int end = min(hi, tile_b0 + kb_tile);
      const bool whole = b == tile_b0 && end == tile_b0 + kb_tile;
      const int ch = tile * 128 + slot_q;
      float v[kCh][8];
#pragma unroll
      for (int i = 0; i < kCh; ++i)
#pragma unroll
        for (int q = 0; q < 8; ++q) v[i][q] = 0.0f;
#pragma unroll 1
      for (; b < end; ++seg) {
        float sc = 1.0f;                                            // W8: scale of this thread's channel in the group
        if (W8) {
          const int kb = b - tile_b0;
          const int g = kb < run.kb_s ? 0 : 1 + active[(kb - run.kb_s) / run.kb_m];
          if (ch < p.d) sc = __ldg(p.scale_d + (size_t)g * p.d + ch);
          const int tok = 16 * (lane >> 3) + 8 * half + (lane & 7);  // the tokens' scales, in the order of v
          __syncwarp();
          if (tok < p.n_rows) tok_sc[lane] = __ldcg(p.tok_scale + g * kStreamMaxRows + tok);
          __syncwarp();
        }
        b = W8 ? min(end, run.group_end(tile_b0, b)) : end;
        const uint32_t buf = seg & 1, use = seg >> 1;
        if (!mbar_wait_warp(accf0 + 8 * buf, use & 1, abort_flag, p.err, kErrWaitAccFull)) { ok = false; break; }
        tc_fence_after();
        const uint32_t taddr = tmem_base + buf * kAcc + ((uint32_t)(quad * 32) << 16) + 8 * half;
#pragma unroll
        for (int i = 0; i < kCh; ++i)
          if (16 * i + 8 * half < p.n_rows) {
            float t[8];
            tmem_ld8(taddr + 16 * i, t);
            if constexpr (W8) {
              float l[8];
              tmem_ld8(taddr + p.tok_rows + 16 * i, l);
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 8; ++q) v[i][q] = fmaf(fmaf(l[q], 0.0625f, t[q]) * sc, tok_sc[8 * i + q], v[i][q]);
            } else {
              tmem_ld_wait();
#pragma unroll
              for (int q = 0; q < 8; ++q) v[i][q] = t[q];
            }
          }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(acce0 + 8 * buf);
      }
      if (!ok) break;
      auto store8 = [&](int c0, const float (&r)[8]) {
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          if (ch < p.d && c0 + q < p.n_rows) p.out[(size_t)(c0 + q) * p.d + ch] = __float2bfloat16_rn(r[q]);
        }
      };
      if (whole) {
#pragma unroll
        for (int i = 0; i < kCh; ++i)
          if (16 * i + 8 * half < p.n_rows) store8(16 * i + 8 * half, v[i]);
        continue;
      }
      int32_t* tk = p.ticket + (size_t)tile * 8 + (warp - 2);
      const int first = run.cta_of(tile_b0), nz = run.cta_of(tile_b0 + kb_tile - 1) - first + 1, own = cta - first;
      // slot of the tile's contributor z: the first one's is its CTA's second, the others' their first; [column / 4][128][4]
      auto slot = [&](int z) {
        return reinterpret_cast<float4*>(p.part) + (size_t)(2 * (first + z) + (z == 0 ? 1 : 0)) * (32 * NT) + slot_q;
      };
      float4* mine = slot(own) + 2 * half * 128;
#pragma unroll
      for (int i = 0; i < kCh; ++i)
        if (16 * i + 8 * half < p.n_rows) {
          __stcg(mine + (size_t)(4 * i) * 128, make_float4(v[i][0], v[i][1], v[i][2], v[i][3]));
          __stcg(mine + (size_t)(4 * i + 1) * 128, make_float4(v[i][4], v[i][5], v[i][6], v[i][7]));
        }
      __syncwarp();                                                 // the lanes' stores are ordered before lane 0's release
      int taken = 0;
      if (lane == 0) taken = atom_inc_acq_rel(tk);
      taken = __shfl_sync(0xffffffffu, taken, 0);
      if (taken != nz - 1) continue;
      __syncwarp();                                                 // lane 0's acquire for all: every contribution is in, add them in CTA order
#pragma unroll 1
      for (int c0 = 8 * half; c0 < p.n_rows; c0 += 16) {
        float r[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) r[q] = 0.0f;
#pragma unroll 1
        for (int z0 = 0; z0 < nz; z0 += kSum) {
          float4 t[kSum][2];
#pragma unroll
          for (int z = 0; z < kSum; ++z)
            if (z0 + z < nz) {
              const float4* sl = slot(z0 + z) + (size_t)(c0 / 4) * 128;
              t[z][0] = __ldcg(sl);
              t[z][1] = __ldcg(sl + 128);
            }
#pragma unroll
          for (int z = 0; z < kSum; ++z)
            if (z0 + z < nz) {
              r[0] += t[z][0].x; r[1] += t[z][0].y; r[2] += t[z][0].z; r[3] += t[z][0].w;
              r[4] += t[z][1].x; r[5] += t[z][1].y; r[6] += t[z][1].z; r[7] += t[z][1].w;
            }
        }
        store8(c0, r);
      }
      if (lane == 0) *tk = 0;                                       // ready for the next launch
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, kTmemCols);
  }
}

// ----------------------------------------------------------------------------- host
struct StreamPlan {
  bool built = false, fp8 = false;
  bf16* h = nullptr;                // Hd [kStreamMaxRows][d_ff]
  float* part = nullptr;
  int32_t* ticket = nullptr;
  CUtensorMap w_gu[16];             // gate/up rows, boxes of 64 k x 8 (i + 1) rows x 2 planes
  CUtensorMap h_s[4], h_r[4];       // Hd: shared columns; routed columns per expert; boxes of 16 (i + 1) rows
  CUtensorMap x[4];                 // x of this forward
  // FP8 weights (stream_plan_attach_fp8): codes of the gate/up rows, boxes of 128 k; E4M3 planes of x and of Hd
  CUtensorMap w_gu8[16], xq[4], hq_s[4], hq_r[4];
  uint8_t* hq = nullptr;            // [2][kStreamMaxRows][d_ff]
  float* hq_scale = nullptr;        // [1 + n_r][kStreamMaxRows]
  const float *x_scale = nullptr, *scale_gu = nullptr, *scale_d = nullptr;
};

inline size_t stream_part_floats(int max_rows) {       // 2 slots per CTA, 128 rows x token columns
  int nt = 16;
  while (nt < max_rows && nt < kStreamMaxRows) nt *= 2;
  return (size_t)2 * kStreamMaxGrid * 128 * nt;
}
inline size_t stream_tickets(int d) { return 8 * (size_t)((d + 127) / 128); }

// Ring sizes: the two kernels (and the router) share an SM: 228 KB, 1 KB of it per block.  tok: bytes of a stage's token rows.
// FP8 with 64 token rows (16 KB a stage) gives that up for tiles high enough to need one round (8B-shaped layer, 64
// rows: 66.8 -> 56.5 us).
inline int stream_up_stages(int h, int tok) {
  const int n = (tok >= 16384 ? 136 : 120) * 1024 / (h * 256 + tok);
  return n > 8 ? 8 : n;
}
inline int stream_up_smem(int h, int tok, int nt, int stages) {
  // a tile's MMAs read 128 rows per plane: the last stage's up plane may be read past the ring's end
  const int ring = stages * (h * 256 + tok), over = (stages - 1) * (h * 256 + tok) + h * 128 + 128 * 128;
  return 1024 + (kStreamTail + 32 * nt + 1023) / 1024 * 1024 + (ring > over ? ring : over);
}
inline int stream_down_stages(int tok) {
  const int n = 98 * 1024 / (16384 + tok);
  return n > 8 ? 8 : n;
}
inline int stream_down_smem(int tok, bool w8) { return 2048 + (w8 ? 1024 : 0) + stream_down_stages(tok) * (16384 + tok); }

template <int NT> inline cudaError_t stream_allow_smem() {
  cudaError_t e = allow_smem(stream_up_kernel<NT, false>, 227 * 1024);
  if (e == cudaSuccess) e = allow_smem(stream_down_kernel<NT, false>, 227 * 1024);
  if (e == cudaSuccess) e = allow_smem(stream_up_kernel<NT, true>, 227 * 1024);
  if (e == cudaSuccess) e = allow_smem(stream_down_kernel<NT, true>, 227 * 1024);
  return e;
}

// Shapes this path takes: plain layers whose k blocks can be numbered in 31 bits.  Their routed experts' W_down has to be finite
// as well: a token's sum runs over all active experts, with zeros in Hd for those it did not select, and 0 x Inf is NaN.
inline bool stream_shape_ok(const UmmaShape& s, int n_sms) {
  return s.plain && s.n_r <= kMaxRouted && n_sms <= kStreamMaxGrid && s.d_ff >= 128 &&
         (long long)((s.d + 127) / 128) * (s.d_ff / 64 + 40) < (1ll << 30);
}

inline bool stream_plan_create(UmmaPlan* P, StreamPlan* S) {
  const UmmaShape& s = P->shape;
  const size_t d = s.d, rows_w = (size_t)s.d_ff;
  bool ok = true;
  for (int i = 0; i < 16 && ok; ++i) {
    const cuuint64_t dims[3] = {d, rows_w, 2};
    const cuuint64_t str[2] = {d * 2, rows_w * d * 2};
    const cuuint32_t box[3] = {kUmmaBK, (cuuint32_t)(8 * (i + 1)), 2};
    ok = umma_encode(P, &S->w_gu[i], P->buf.w_gate_up, 3, dims, str, box, "gate/up weights (stream)");
  }
  for (int i = 0; i < 4 && ok; ++i) {
    const cuuint32_t rows = 16u * (i + 1);
    if (P->has_s) {
      const cuuint64_t dims[2] = {(cuuint64_t)s.shared_width, (cuuint64_t)kStreamMaxRows};
      const cuuint64_t str[1] = {rows_w * 2};
      const cuuint32_t box[2] = {kUmmaBK, rows};
      ok = umma_encode(P, &S->h_s[i], S->h, 2, dims, str, box, "Hd shared");
    }
    if (ok && P->has_r) {
      const cuuint64_t dims[3] = {(cuuint64_t)s.m, (cuuint64_t)s.n_r, (cuuint64_t)kStreamMaxRows};
      const cuuint64_t str[2] = {(cuuint64_t)s.m * 2, rows_w * 2};
      const cuuint32_t box[3] = {kUmmaBK, 1, rows};
      ok = umma_encode(P, &S->h_r[i], S->h + s.shared_width, 3, dims, str, box, "Hd routed");
    }
    if (!P->has_s) S->h_s[i] = S->h_r[i];
    if (!P->has_r) S->h_r[i] = S->h_s[i];
  }
  if (!ok) return false;
  cudaError_t e = stream_allow_smem<16>();
  if (e == cudaSuccess) e = stream_allow_smem<32>();
  if (e == cudaSuccess) e = stream_allow_smem<64>();
  if (e != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "cudaFuncSetAttribute (stream): %s", cudaGetErrorString(e));
    return false;
  }
  S->built = true;
  return true;
}

// FP8 codes and token planes of a quantised layer, all owned by the caller: w_gu8 [2][d_ff][d], xq [2][kStreamMaxRows][d],
// hq [2][kStreamMaxRows][d_ff], hq_scale [1 + n_r][kStreamMaxRows]; d, m and the shared width are multiples of 16.
inline bool stream_plan_attach_fp8(UmmaPlan* P, StreamPlan* S, const void* w_gu8, const uint8_t* xq, const float* x_scale,
                                   uint8_t* hq, float* hq_scale, const float* scale_gu, const float* scale_d) {
  const UmmaShape& s = P->shape;
  const cuuint64_t d = s.d, rows_w = s.d_ff, plane_rows = kStreamMaxRows;
  auto encode8 = [&](CUtensorMap* tm, const void* base, int rank, const cuuint64_t* dims, const cuuint64_t* str,
                     const cuuint32_t* box, const char* what) {
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    const CUresult r = P->encode(tm, CU_TENSOR_MAP_DATA_TYPE_UINT8, (cuuint32_t)rank, const_cast<void*>(base), dims, str,
                                 box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    if (r != CUDA_SUCCESS) {
      snprintf(P->error, sizeof(P->error), "cuTensorMapEncodeTiled(%s) failed with CUresult %d", what, (int)r);
      return false;
    }
    return true;
  };
  bool ok = true;
  for (int i = 0; i < 16 && ok; ++i) {
    const cuuint64_t dims[3] = {d, rows_w, 2}, str[2] = {d, rows_w * d};
    const cuuint32_t box[3] = {2 * kUmmaBK, (cuuint32_t)(8 * (i + 1)), 2};
    ok = encode8(&S->w_gu8[i], w_gu8, 3, dims, str, box, "FP8 gate/up weights (stream)");
  }
  for (int i = 0; i < 4 && ok; ++i) {
    const cuuint32_t rows = 16u * (i + 1);
    {
      const cuuint64_t dims[3] = {d, plane_rows, 2}, str[2] = {d, plane_rows * d};
      const cuuint32_t box[3] = {2 * kUmmaBK, rows, 2};
      ok = encode8(&S->xq[i], xq, 3, dims, str, box, "E4M3 planes of x (stream)");
    }
    if (ok && P->has_s) {
      const cuuint64_t dims[3] = {(cuuint64_t)s.shared_width, plane_rows, 2}, str[2] = {rows_w, plane_rows * rows_w};
      const cuuint32_t box[3] = {2 * kUmmaBK, rows, 2};
      ok = encode8(&S->hq_s[i], hq, 3, dims, str, box, "E4M3 planes of Hd shared");
    }
    if (ok && P->has_r) {
      const cuuint64_t dims[4] = {(cuuint64_t)s.m, (cuuint64_t)s.n_r, plane_rows, 2};
      const cuuint64_t str[3] = {(cuuint64_t)s.m, rows_w, plane_rows * rows_w};
      const cuuint32_t box[4] = {2 * kUmmaBK, 1, rows, 2};
      ok = encode8(&S->hq_r[i], hq + s.shared_width, 4, dims, str, box, "E4M3 planes of Hd routed");
    }
    if (!P->has_s) S->hq_s[i] = S->hq_r[i];
    if (!P->has_r) S->hq_r[i] = S->hq_s[i];
  }
  if (!ok) return false;
  S->hq = hq; S->hq_scale = hq_scale; S->x_scale = x_scale; S->scale_gu = scale_gu; S->scale_d = scale_d;
  S->fp8 = true;
  return true;
}

// Experts expected to be active, and whether to treat all as active: when the weights streamed in vain are expected to
// take less time than the part of the router's latency that is hidden in return (about 4 us, 24 MB of the stream).
inline double stream_expected_active(const UmmaShape& s, int n_rows) {
  if (s.n_r == 0 || s.n_k == 0) return 0.0;
  double miss = 1.0;
  for (int i = 0; i < n_rows && miss > 1e-6; ++i) miss *= 1.0 - (double)s.n_k / s.n_r;
  return s.n_r * (1.0 - miss);
}
// An upper estimate (one more round of tiles than planned costs more than slightly lower tiles).
inline int stream_likely_active(const UmmaShape& s, int n_rows, double active) {
  if (s.n_r == 0 || s.n_k == 0) return 0;
  const double p = active / s.n_r;
  int hi = (int)ceil(active + sqrt(s.n_r * p * (1.0 - p)));
  if (hi > s.n_r) hi = s.n_r;
  return (long long)hi > (long long)n_rows * s.n_k ? n_rows * s.n_k : hi;
}
inline bool stream_dense(const UmmaShape& s, double active, bool w8) {
  return (s.n_r - active) * s.m * (w8 ? 2.0 : 4.0) * s.d < 24e6;
}

// Neurons per tile: the height whose rounds over the SMs take the least time for the expected tiles.  A round is bound by
// its weight bytes, the token rows that go with each block (from L2, counted a third) and the MMAs of a block (at least the
// time of some 8 KB of the stream).
inline int stream_pick_rows(const UmmaShape& s, int active, int tok, int n_sms) {
  int best = 64;
  double best_cost = 1e30;
  for (int h = 128; h >= 16; h -= 8) {
    if (stream_up_stages(h, tok) < 3) continue;
    const int tiles = (s.shared_width + h - 1) / h + active * ((s.m + h - 1) / h);
    const int rounds = tiles > 0 ? (tiles + n_sms - 1) / n_sms : 1;
    const double bytes = h * 256.0 + tok / 3.0;
    const double cost = rounds * (bytes < 8192 ? 8192 : bytes);
    if (cost < best_cost * 0.999) { best_cost = cost; best = h; }
  }
  return best;
}

template <int NT, bool W8>
inline void stream_launch(const UmmaPlan* P, const StreamPlan* S, const CUtensorMap& wd_s, const CUtensorMap& wd_r, int bi,
                          StreamArgs a, cudaStream_t st, cudaEvent_t mid, bool dep, bool gate_up_only) {
  const int tok = (W8 ? 2 : 1) * a.tok_rows * 128, wi = a.tile_rows / 8 - 1;
  a.stages = stream_up_stages(a.tile_rows, tok);
  launch_kernel(dep, stream_up_kernel<NT, W8>, dim3(P->n_sms), dim3(kStreamThreads),
                stream_up_smem(a.tile_rows, tok, NT, a.stages), st, W8 ? S->w_gu8[wi] : S->w_gu[wi], W8 ? S->xq[bi] : S->x[bi], a);
  if (mid) cudaEventRecord(mid, st);
  if (gate_up_only) return;
  if (W8) {                                       // E4M3 planes of Hd
    const SplitGroups hd{S->h, S->hq, S->hq_scale, a.has_s ? a.shared_w : 0, a.m, a.ld_h, kStreamMaxRows};
    launch_kernel(dep, split_groups_e4m3_kernel, dim3(a.n_rows, 1 + a.n_r), dim3(kSplitGroupThreads), 0, st, hd);
    a.tok_scale = S->hq_scale;
  }
  a.stages = stream_down_stages(tok);
  launch_kernel(dep, stream_down_kernel<NT, W8>, dim3(P->n_sms), dim3(kStreamThreads), stream_down_smem(tok, W8), st, wd_s, wd_r,
                W8 ? S->hq_s[bi] : S->h_s[bi], W8 ? S->hq_r[bi] : S->h_r[bi], a);
}

// Both streamers for n_rows <= kStreamMaxRows rows of x; `h`: where the up kernel writes (Hd, or H of an all-shared
// layer when only the gate/up part is wanted).  FP8 layers: the planes of x have been written.  Returns the number of
// launches or -1.
inline int stream_forward(UmmaPlan* P, StreamPlan* S, const CUtensorMap& wd_s, const CUtensorMap& wd_r, const GroupRows* gr,
                          const void* x, int n_rows, bf16* out, bf16* h, int32_t* err_word, cudaStream_t st,
                          cudaEvent_t mid, bool dep, bool gate_up_only) {
  const UmmaShape& s = P->shape;
  const int bi = (n_rows + 15) / 16 - 1;
  const bool w8 = S->fp8;
  if (!w8 && !umma_encode_rows(P, &S->x[bi], x, (size_t)n_rows, (size_t)s.d, 16 * (bi + 1), "x (stream)")) return -1;
  const double active = P->has_r ? stream_expected_active(s, n_rows) : 0.0;
  StreamArgs a{};
  a.gr = gr; a.has_s = P->has_s; a.n_r = P->has_r ? s.n_r : 0; a.n_k = s.n_k;
  a.n_rows = n_rows; a.d = s.d; a.shared_w = s.shared_width; a.m = s.m;
  a.dense = !P->has_r || stream_dense(s, active, w8);
  a.tok_rows = 16 * (bi + 1);
  a.tile_rows = stream_pick_rows(s, a.dense && P->has_r ? s.n_r : stream_likely_active(s, n_rows, active),
                                 (w8 ? 2 : 1) * a.tok_rows * 128, P->n_sms);
  a.topk_idx = P->buf.topk_idx; a.topk_gate = P->buf.topk_gate;
  a.h = h; a.ld_h = s.d_ff; a.out = out;
  a.part = S->part; a.ticket = S->ticket; a.err = err_word;
  a.tok_scale = S->x_scale; a.scale_gu = S->scale_gu; a.scale_d = S->scale_d; a.rows_w = s.d_ff;
#define CMOE_STREAM(NT) (w8 ? stream_launch<NT, true> : stream_launch<NT, false>)(P, S, wd_s, wd_r, bi, a, st, mid, dep, gate_up_only)
  if (bi == 0) CMOE_STREAM(16);
  else if (bi == 1) CMOE_STREAM(32);
  else CMOE_STREAM(64);
#undef CMOE_STREAM
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "stream launch: %s", cudaGetErrorString(e));
    return -1;
  }
  return gate_up_only ? 1 : 2 + (w8 ? 1 : 0);
}

}  // namespace cmoe
