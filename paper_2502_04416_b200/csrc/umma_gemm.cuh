// Tensor-core kernels for sm_100a: tcgen05.mma with the accumulator in tensor memory
// (TMEM), operands staged in shared memory by TMA, one persistent CTA per SM,
// warp-specialised (TMA producer warp / MMA issuer / 4 epilogue warps), TMEM accumulator
// double-buffered so the epilogue of one tile overlaps the MMAs of the next.
//
//   MODE 1, gate/up GEMM: H[r, n] = Swish(x_r . Wg[n]) * (x_r . Wu[n])      (Eq. ori_ffn_method)
//       A tile  : 128 rows of x x 64 k.  Shared groups read consecutive outer rows by TMA.
//                 Routed groups gather their rows straight from x, so no permuted copy of
//                 x is ever written: four extra warps (one thread per tile row) issue
//                 16-byte cp.async copies into the 128-byte-swizzled layout the MMA expects
//                 and arrive on the stage's barrier when their copies land.  TMA tile::gather4
//                 does the same with one copy per 4 rows and is slower for every batch: 7B-shaped
//                 layer 200 / 256 rows 94.2 / 106.2 us against 78.2 / 78.1.
//       B tile  : bn gate rows + bn up rows of the group's neurons x 64 k (one 3-D TMA box)
//       D (TMEM): 128 lanes x 2*bn fp32 columns; epilogue fuses SiLU(gate)*up -> bf16 H
//   MODE 3, down GEMM of the shared experts of a plain layer with the combine in its epilogue (umma_folds_combine), after mode 2 for
//       the routed experts.
//   MODE 2, down GEMM: Y[r, c] = sum_n H[r, n] Wd[c, n]
//       A tile  : 128 rows of H x 64 k ;  B tile: 256 output channels of the group's W_down
//       block x 64 k ;  D: 128 x 256 fp32 ; epilogue rounds to bf16 Y.
// All operands are K-major with the 128-byte swizzle; rows or k beyond a tensor's extent
// are zero-filled by TMA, rows beyond a group's count are computed but never stored.
//
// Every mbarrier wait is bounded (about a second of SM clock); a wait that runs out sets
// the layer's device error word, raises a CTA-wide abort flag that the other waits poll,
// and the CTA falls through to the common teardown, which frees its TMEM.
#pragma once

#include <cuda.h>

#include <cstdio>

#include "common.cuh"

namespace cmoe {

constexpr int kUmmaBM = 128;          // rows per tile (UMMA M)
constexpr int kUmmaBK = 64;           // k per stage: 64 bf16 = one 128-byte swizzle row
constexpr int kUmmaStages = 4;
constexpr int kUmmaABytes = kUmmaBM * kUmmaBK * 2;       // 16 KB
constexpr int kUmmaBBytes = 256 * kUmmaBK * 2;           // 32 KB (up to 256 B rows)
constexpr int kUmmaStageBytes = kUmmaABytes + kUmmaBBytes;
constexpr int kUmmaMaxGroups = 1088;
constexpr int kUmmaThreads = 192;     // warp 0 TMA, warp 1 MMA, warps 2..5 epilogue
constexpr int kUmmaGatherThreads = 128;   // mode 1 only: warps 6..9, one thread per A-tile row
constexpr int kUmmaTmemCols = 512;    // two accumulator buffers of 256 columns
constexpr int kUmmaSmemBytes = 1024 /*alignment slack*/ + kUmmaStages * kUmmaStageBytes +
                               256 /*barriers*/ + (kUmmaMaxGroups + 1) * 4 + kUmmaMaxGroups * 8 /*group rows*/;
// A layer asks for its own groups only: a small router then fits on the SM beside the gate/up GEMM.
inline int umma_smem_bytes(int n_groups) { return kUmmaSmemBytes - (kUmmaMaxGroups - n_groups) * 12; }
constexpr long long kUmmaWaitCycles = 2000000000LL;   // ~1 s at SM clock

enum { kErrWaitFull = 1, kErrWaitEmpty = 2, kErrWaitAccFull = 3, kErrWaitAccEmpty = 4 };

// ----------------------------------------------------------------------------- PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// Bounded wait: false if the wait ran out (error word + abort flag set) or another wait
// of this CTA already gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                          int32_t* err_word, int code, long long limit = kUmmaWaitCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  for (;;) {
#pragma unroll 1
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort_flag) return false;
    if (clock64() - t0 > limit) {
      *abort_flag = 1;
      atomicCAS(err_word, 0, code);
      return false;
    }
  }
}
// The same for a whole warp: every lane gets the same answer, so the warp stays converged.
__device__ __forceinline__ bool mbar_wait_warp(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int32_t* err_word, int code) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity, abort_flag, err_word, code));
}
// One lane of a converged warp, always the same one.  tcgen05 and TMA instructions take their operands from
// uniform registers: issued under a branch on the lane number they cost 72-95 cycles each whatever their size
// (measured: back-to-back M = 128 MMAs), under elect.sync in a loop that the whole warp runs 39 cycles at
// N <= 32, 48 at N = 64, 64 at N = 128 and 128 at N = 256, the rate of the tensor core itself.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
// Warp index as a value the compiler knows to be uniform.
__device__ __forceinline__ int warp_index() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }
__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1) : "memory");
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1,
                                            int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2) : "memory");
}
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, uint32_t bar, int c0, int c1,
                                            int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"(tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
__device__ __forceinline__ void tmem_alloc(uint32_t smem_slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_slot), "r"(cols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// D[tmem] (+)= A[smem desc] * B[smem desc]^T, bf16 inputs, fp32 accumulate.
__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// D[tmem] (+)= A[smem desc] * B[smem desc]^T, E4M3 inputs (32 k values per step), fp32 accumulate.
__device__ __forceinline__ void umma_e4m3(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                          uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d_tmem), "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate) : "memory");
}
// mbarrier arrives once all tcgen05 operations issued so far by this thread have completed.
__device__ __forceinline__ void umma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// 16 consecutive fp32 columns of this thread's TMEM lane.
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
__device__ __forceinline__ void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor: K-major tile, 128-byte rows, 128-byte swizzle, 8-row
// groups 1024 bytes apart; `addr` is the 1024-byte-aligned tile base plus the k offset.
__device__ __forceinline__ uint64_t umma_smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)1 << 16;                 // leading-dimension offset (unused with swizzle)
  d |= (uint64_t)(1024 >> 4) << 32;       // stride between 8-row groups
  d |= (uint64_t)1 << 46;                 // descriptor version of sm_100
  d |= (uint64_t)2 << 61;                 // 128-byte swizzle
  return d;
}
// Instruction descriptor: bf16 x bf16 -> fp32, both operands K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t umma_idesc(int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kUmmaBM >> 4) << 24);
}

// One warp waits, with a limit of `limit` SM cycles, on an mbarrier that nobody arrives on, through the
// same mbar_wait the tensor-core kernels use: the wait gives up, the error word takes the code,
// the kernel returns normally.  No copy is in flight and no tensor memory is held.
__global__ void wait_timeout_probe_kernel(int32_t* err_word, long long limit) {
  __shared__ __align__(8) unsigned long long bar_mem;
  __shared__ int abort_flag;
  const uint32_t bar = smem_u32(&bar_mem);
  if (threadIdx.x == 0) {
    mbar_init(bar, 1);
    abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncwarp();
  if (threadIdx.x == 0) mbar_wait(bar, 0, &abort_flag, err_word, kErrWaitFull, limit);
  __syncwarp();
}

// Instruction descriptor of kind::f8f6f4: E4M3 x E4M3 (operand format code 0) -> fp32, both K-major, M = 128, N = n.
__device__ __forceinline__ uint32_t umma_idesc_e4m3(int n) {
  return (1u << 4) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(kUmmaBM >> 4) << 24);
}

// ----------------------------------------------------------------------------- kernel
struct UmmaArgs {
  const GroupStatic* gs;
  const GroupRows* gr;
  int n_groups, n_outer, n_r;
  int d;                 // model width: K of modes 1 and 3, N of mode 2
  int bn_s, bn_r;        // mode 1: neurons per tile for shared / routed groups
  bf16* out_s;           // mode 1: H_s ; mode 2: Y_s
  bf16* out_r;           // mode 1: H_r ; mode 2: Y_r
  int ld_out_s, ld_out_r;
  const int32_t* row_token;   // mode 1: outer row held by each routed row (gather source)
  int band_mt;                // row tiles per band of the tile order (see umma_decode)
  const bf16* x_rows_ptr;     // mode 1: the outer rows of x (source of the cp.async gather)
  int32_t* err;
  int shared_width;           // neurons of the shared experts
  int skip_groups;            // mode 2: this many groups ahead are left out (the shared experts, which mode 3 does)
  const bf16* y_r;            // mode 3: routed rows, their places and gates
  const int32_t* row_of;
  const float* topk_gate;
  int n_k;
  int early_rows;             // modes 1, 3: rows of group 0 where the host knows them (the shared experts of a plain layer), else 0
};

// tile_start[g + 1] holds the tiles of group g; turns them into the prefix sums, tile_start[0] = 0 (one warp).
__device__ __forceinline__ void warp_prefix(int32_t* tile_start, int n_groups, int lane) {
  const int each = (n_groups + 31) / 32, lo = lane * each, hi = min(lo + each, n_groups);
  int sum = 0;
  for (int g = lo; g < hi; ++g) sum += tile_start[g + 1];
  int incl = sum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int up = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += up;
  }
  int run = incl - sum;
  for (int g = lo; g < hi; ++g) { run += tile_start[g + 1]; tile_start[g + 1] = run; }
  if (lane == 0) tile_start[0] = 0;
}

struct TileCoord { int g, mt, nt, row0, count; };

template <int MODE>
__device__ __forceinline__ int umma_n_tiles(const UmmaArgs& p, int g) {
  const GroupStatic gs = p.gs[g];
  if (MODE == 1) {
    const int bn = gs.is_shared ? p.bn_s : p.bn_r;
    return (gs.width + bn - 1) / bn;
  }
  return gs.width > 0 ? (p.d + 255) / 256 : 0;
}

// Tile `local` of group g.
template <int MODE>
__device__ __forceinline__ TileCoord umma_tile_in(const UmmaArgs& p, int g, const GroupRows r, int n_tiles, int local) {
  // Order inside a group: bands of p.band_mt row tiles; inside a band the row tiles run fastest (CTAs
  // working side by side share a weight tile), then the n-tiles, then the next band.  A band's rows of A
  // (about 16 MB) stay in L2 while the n-tiles pass over them; without bands a large group's rows left L2
  // between two n-tiles and were read again for each (5.6 GB of DRAM reads instead of 0.45 GB in the gate/up
  // GEMM of the 16384-token workload), while letting the n-tiles run fastest everywhere was slower for the
  // groups that do fit (every CTA then streams a different weight tile).
  const int m_tiles = (r.count + kUmmaBM - 1) / kUmmaBM;
  const int band_mt = max(p.band_mt, 1);
  const int per_band = band_mt * n_tiles;
  const int band = local / per_band, in_band = local - band * per_band;
  const int cur_mt = min(band_mt, m_tiles - band * band_mt);
  TileCoord c;
  c.g = g; c.nt = in_band / cur_mt; c.mt = band * band_mt + in_band % cur_mt; c.row0 = r.row0; c.count = r.count;
  return c;
}

template <int MODE>
__device__ __forceinline__ TileCoord umma_decode(const UmmaArgs& p, const int32_t* tile_start, const GroupRows* rows,
                                                 int n_groups, int t) {
  int lo = 0, hi = n_groups;                 // last g with tile_start[g] <= t
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tile_start[mid] <= t) lo = mid; else hi = mid;
  }
  return umma_tile_in<MODE>(p, lo, rows[lo], umma_n_tiles<MODE>(p, lo), t - tile_start[lo]);
}

template <int MODE>
__global__ void __launch_bounds__(MODE == 2 ? kUmmaThreads : kUmmaThreads + 128, 1)
umma_grouped_kernel(const __grid_constant__ CUtensorMap tm_a_s, const __grid_constant__ CUtensorMap tm_a_r,
                    const __grid_constant__ CUtensorMap tm_b_s, const __grid_constant__ CUtensorMap tm_b_r,
                    const UmmaArgs p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);                       // generic pointer to the aligned base
  constexpr int kStages = kUmmaStages, kStageBytes = kUmmaStageBytes;
  const uint32_t bars = base + kStages * kStageBytes;   // barrier block
  uint8_t* bars_gen = gen + kStages * kStageBytes;
  // barrier block: full[8] empty[8] acc_full[2] acc_empty[2] (8 B each), tmem slot, abort flag
  const uint32_t full0 = bars, empty0 = bars + 64, accf0 = bars + 128, acce0 = bars + 144, tbl_bar = bars + 168;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars_gen + 160);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + 164);
  int32_t* tile_start = reinterpret_cast<int32_t*>(bars_gen + 256);
  GroupRows* rows = reinterpret_cast<GroupRows*>(tile_start + p.n_groups + 1);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const int n_groups = p.n_groups;

  if (threadIdx.x == 0) {
    // mode 1: besides the producer's expect_tx arrival, every gather thread arrives once per stage
    const uint32_t full_count = MODE == 1 ? 1 + kUmmaGatherThreads : 1;
    for (int s = 0; s < kStages; ++s) { mbar_init(full0 + 8 * s, full_count); mbar_init(empty0 + 8 * s, 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(accf0 + 8 * b, 1); mbar_init(acce0 + 8 * b, MODE == 3 ? 8 : 4); }
    mbar_init(tbl_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(tmem_slot), kUmmaTmemCols);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int k_blocks_fixed = (p.d + kUmmaBK - 1) / kUmmaBK;      // mode 1: K = d
  // Warp 2 counts the tiles of every group and publishes the table on a barrier; in mode 1 it waits for the router and the
  // permutation first, in mode 2 the preceding kernel has read the same rows already.  Tiles that need no table, those of the shared
  // experts of a plain layer (group 0, all rows of x), run at once, under the routing and this kernel's own start-up.
  // Mode 2 fetches the weights of its first stages under the end of the gate/up GEMM.  (With a wait at the top and a table that all
  // threads count and one sums, 3.7 us passed from the permutation's end to the first operands of a tile, 3.3 from the gate/up GEMM's:
  // 8B-shaped 300 / 2048 rows 102.0 / 231 -> 94.4 / 213 us, 7B-shaped 300 rows 79.2 -> 75.5, 13B-shaped 128.0 -> 113.2.)
  const int early_n = MODE == 3 ? (p.d + 255) / 256 : MODE == 1 && p.early_rows > 0 ? (p.shared_width + p.bn_s - 1) / p.bn_s : 0;
  const int early_tiles = (p.early_rows + kUmmaBM - 1) / kUmmaBM * early_n;
  if (MODE == 3) {
    if (warp == 2) { grid_dep_wait(); grid_dep_trigger(); }     // as an epilogue warp it waits all the same
  } else if (warp == 2) {
    for (int g = lane; g < n_groups; g += 32) tile_start[g + 1] = umma_n_tiles<MODE>(p, g);
    if (MODE == 1) { grid_dep_wait(); grid_dep_trigger(); }
    for (int g = lane; g < n_groups; g += 32) {
      const GroupRows gr = p.gr[g];
      rows[g] = gr;
      tile_start[g + 1] *= MODE == 2 && g < p.skip_groups ? 0 : (gr.count + kUmmaBM - 1) / kUmmaBM;
    }
    __syncwarp();
    warp_prefix(tile_start, n_groups, lane);
    __syncwarp();
    if (lane == 0) mbar_arrive(tbl_bar);
    if (MODE == 2) { grid_dep_wait(); grid_dep_trigger(); }     // what follows may count on the gate/up GEMM
  }
  bool seen = false;                             // this thread has waited for the table
  auto tile_at = [&](int t, TileCoord& c, GroupStatic& g, bool whole_warp, bool& ok) {   // false: no tile t, or a wait gave up
    if (MODE != 2 && t < early_tiles) {
      GroupRows all; all.row0 = 0; all.count = p.early_rows;
      c = umma_tile_in<MODE>(p, 0, all, early_n, t);
      g.w_row0 = 0; g.width = p.shared_width; g.wd_offset = 0; g.is_shared = 1; g.outer = 0;
      return true;
    }
    if (MODE == 3) return false;
    if (!seen) {
      ok = mbar_wait(tbl_bar, 0, abort_flag, p.err, kErrWaitFull);
      if (whole_warp) ok = __all_sync(0xffffffffu, ok);
      if (!ok) return false;
      if (MODE == 1) grid_dep_wait();
      seen = true;
    }
    if (t >= tile_start[n_groups]) return false;
    c = umma_decode<MODE>(p, tile_start, rows, n_groups, t);
    g = p.gs[c.g];
    return true;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (whole warp)
    uint32_t it = 0, n_ahead = 0;
    bool waited = false;
    bool ok = true;
    for (int t = blockIdx.x; ok; t += gridDim.x) {
      TileCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, true, ok)) break;
      const int row = c.row0 + c.mt * kUmmaBM;
      const bool by_threads = MODE == 1 && !g.is_shared;              // the gather warps fill A
      const CUtensorMap* ta = g.is_shared ? &tm_a_s : &tm_a_r;
      const CUtensorMap* tb = g.is_shared ? &tm_b_s : &tm_b_r;
      int k_blocks, b_bytes, b_row = 0, j = 0;
      if (MODE == 1) {
        const int bn = g.is_shared ? p.bn_s : p.bn_r;
        k_blocks = k_blocks_fixed;
        b_bytes = 2 * bn * kUmmaBK * 2;
        b_row = g.w_row0 + c.nt * bn;
      } else {
        k_blocks = (g.width + kUmmaBK - 1) / kUmmaBK;
        b_bytes = kUmmaBBytes;
        b_row = c.nt * 256;
        j = g.is_shared ? 0 : (c.g - p.n_outer) - g.outer * p.n_r;
      }
      auto load_b = [&](int kb, uint32_t sb, uint32_t fb) {
        if (MODE == 1) tma_load_3d(sb, tb, fb, kb * kUmmaBK, b_row, 0);
        else if (g.is_shared) tma_load_3d(sb, tb, fb, kb * kUmmaBK, b_row, g.outer);
        else tma_load_4d(sb, tb, fb, kb * kUmmaBK, b_row, j, g.outer);
      };
      if (MODE == 2 && it == 0 && !waited) {         // weights of the first stages ahead of the wait for the gate/up GEMM
        n_ahead = min(kStages, k_blocks);
        for (uint32_t i = 0; i < n_ahead; ++i) {
          if (elect_one()) {
            mbar_expect_tx(full0 + 8 * i, kUmmaABytes + b_bytes);
            load_b(i, base + i * kStageBytes + kUmmaABytes, full0 + 8 * i);
          }
          __syncwarp();
        }
        grid_dep_wait();
        waited = true;
      }
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const uint32_t s = it % kStages, n = it / kStages;
        if (!mbar_wait_warp(empty0 + 8 * s, (n & 1) ^ 1, abort_flag, p.err, kErrWaitEmpty)) { ok = false; break; }
        const uint32_t fb = full0 + 8 * s;
        const uint32_t sa = base + s * kStageBytes, sb = sa + kUmmaABytes;
        if (elect_one()) {
          if (MODE != 2 || it >= n_ahead) {
            mbar_expect_tx(fb, (by_threads ? 0 : kUmmaABytes) + b_bytes);
            load_b(kb, sb, fb);
          }
          if (!by_threads) tma_load_2d(sa, ta, fb, kb * kUmmaBK, row);
        }
        __syncwarp();
      }
    }
    if (!ok) for (int i = 0; i < 200; ++i) __nanosleep(1000);   // let copies in flight land
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (whole warp, one lane issues)
    uint32_t it = 0, tile_n = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok; t += gridDim.x, ++tile_n) {
      TileCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, true, ok)) break;
      int k_blocks, n_mma;
      if (MODE == 1) {
        k_blocks = k_blocks_fixed; n_mma = 2 * (g.is_shared ? p.bn_s : p.bn_r);
      } else {
        k_blocks = (g.width + kUmmaBK - 1) / kUmmaBK; n_mma = 256;
      }
      const uint32_t idesc = umma_idesc(n_mma);
      const uint32_t buf = tile_n & 1, use = tile_n >> 1;
      if (!mbar_wait_warp(acce0 + 8 * buf, (use & 1) ^ 1, abort_flag, p.err, kErrWaitAccEmpty)) { ok = false; break; }
      tc_fence_after();
      const uint32_t d_tmem = tmem_base + buf * 256;
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const uint32_t s = it % kStages, n = it / kStages;
        if (!mbar_wait_warp(full0 + 8 * s, n & 1, abort_flag, p.err, kErrWaitFull)) { ok = false; break; }
        if (MODE == 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // cp.async-written rows
        tc_fence_after();
        const uint32_t sa = base + s * kStageBytes, sb = sa + kUmmaABytes;
        if (elect_one()) {
#pragma unroll
          for (int k = 0; k < kUmmaBK / 16; ++k)
            umma_bf16(d_tmem, umma_smem_desc(sa + k * 32), umma_smem_desc(sb + k * 32), idesc,
                      (kb != 0 || k != 0) ? 1u : 0u);
          umma_commit(empty0 + 8 * s);         // stage reusable once these MMAs have read it
        }
        __syncwarp();
      }
      if (ok && elect_one()) umma_commit(accf0 + 8 * buf);  // accumulator complete
      __syncwarp();
    }
  } else if (MODE == 1 && warp >= 6) {
    // ------------------------------------------------------------ A-row gather (mode 1, warps 6..9)
    // For routed groups the 128 threads copy the tile's 128 rows x 128 bytes of
    // this k block from x: eight consecutive threads cover one row (coalesced 128-byte reads), 16
    // rows per pass, 8 passes; 16-byte chunk c of row r goes to the swizzled chunk c ^ (r & 7).
    // Otherwise the threads only arrive.
    const int gt = threadIdx.x - kUmmaThreads;
    const int ch = gt & 7, r_sub = gt >> 3;
    uint32_t it = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok; t += gridDim.x) {
      TileCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, false, ok)) break;
      const bool mine = !g.is_shared;
      const bf16* src_row[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        src_row[i] = nullptr;
        const int r = c.mt * kUmmaBM + i * 16 + r_sub;
        if (mine && r < c.count)                      // rows past the group are left as they are: nothing of them is stored
          src_row[i] = p.x_rows_ptr + (size_t)__ldcg(p.row_token + c.row0 + r) * p.d;
      }
      for (int kb = 0; kb < k_blocks_fixed; ++kb, ++it) {
        const uint32_t s = it % kStages, n = it / kStages;
        if (!mbar_wait(empty0 + 8 * s, (n & 1) ^ 1, abort_flag, p.err, kErrWaitEmpty)) { ok = false; break; }
        const uint32_t fb = full0 + 8 * s;
        if (mine) {
          const int k = kb * kUmmaBK + ch * 8;
          const uint32_t bytes = k < p.d ? 16u : 0u;                        // zero-fill past the end of the row
          const int k_src = k < p.d ? k : 0;
          const uint32_t sa = base + s * kStageBytes;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = i * 16 + r_sub;
            if (src_row[i])
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(sa + r * 128 + ((ch ^ (r & 7)) << 4)), "l"(src_row[i] + k_src), "r"(bytes)
                         : "memory");
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(fb) : "memory");
        } else {
          mbar_arrive(fb);
        }
      }
    }
    if (!ok) asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // ------------------------------------------------------------ epilogue (warps 2..5, mode 3: 2..9)
    const int quad = warp & 3;                 // TMEM lane quadrant this warp may read
    uint32_t tile_n = 0;
    bool ok = true;
    for (int t = blockIdx.x; ok; t += gridDim.x, ++tile_n) {
      TileCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, false, ok)) break;
      int pos[4];
      float gate[4];
      if (MODE == 3) {                             // this row's routing, under the multiplies
        const size_t tok = (size_t)(c.row0 + (c.mt * kUmmaBM + quad * 32 + lane));
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const bool on = j < p.n_k && (c.mt * kUmmaBM + quad * 32 + lane) < c.count;
          pos[j] = on ? __ldcg(p.row_of + tok * p.n_k + j) : 0;
          gate[j] = on ? __ldcg(p.topk_gate + tok * p.n_k + j) : 0.0f;
        }
        if (tile_n == 0) grid_dep_wait();          // the routed experts' rows are complete
      }
      const uint32_t buf = tile_n & 1, use = tile_n >> 1;
      if (!mbar_wait(accf0 + 8 * buf, use & 1, abort_flag, p.err, kErrWaitAccFull)) { ok = false; break; }
      tc_fence_after();
      const int row_in_group = c.mt * kUmmaBM + quad * 32 + lane;
      const bool row_ok = row_in_group < c.count;
      const uint32_t taddr = tmem_base + buf * 256 + ((uint32_t)(quad * 32) << 16);
      if (MODE == 1) {
        const int bn = g.is_shared ? p.bn_s : p.bn_r;
        const int ld = g.is_shared ? p.ld_out_s : p.ld_out_r;
        const int n0 = c.nt * bn;
        const int n_valid = min(bn, g.width - n0);
        bf16* dst = (g.is_shared ? p.out_s : p.out_r) + (size_t)(c.row0 + row_in_group) * ld + n0;
        const bool wide = ((ld | n0) & 15) == 0;          // 32-byte aligned row segments
        for (int c0 = 0; c0 < n_valid; c0 += 16) {
          float gt[16], up[16];
          tmem_ld16(taddr + c0, gt);
          tmem_ld16(taddr + bn + c0, up);
          tmem_ld_wait();
          if (row_ok) {
            float h16[16];
#pragma unroll
            for (int q = 0; q < 16; ++q) h16[q] = swiglu_fast(gt[q], up[q]);
            if (wide && c0 + 16 <= n_valid) {
              store16(dst + c0, h16);
            } else {
#pragma unroll
              for (int h = 0; h < 2; ++h) {
                if (c0 + h * 8 < n_valid) {
                  float v[8];
#pragma unroll
                  for (int q = 0; q < 8; ++q) v[q] = h16[h * 8 + q];
                  store8(dst + c0 + h * 8, v);
                }
              }
            }
          }
        }
      } else if (MODE == 3) {
        // out = Y_s + sum_j g_j Y_r[row_of_j], with the rounding and the order of combine_plain_bf16_kernel: the same bits.
        // 32 columns at a time: all loads of the routed rows before any arithmetic.
        const int n0 = c.nt * 256;
        const int n_valid = min(256, p.d - n0);                      // a multiple of 16
        const size_t tok = (size_t)(c.row0 + row_in_group);
        const bf16* yr[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) yr[j] = p.y_r + (size_t)pos[j] * p.d + n0;
        bf16* dst = p.out_s + tok * p.d + n0;
        const int c_end = min(n_valid, warp < 6 ? 128 : 256);         // warps 2..5 the left half, 6..9 the right
        for (int c0 = warp < 6 ? 0 : 128; c0 < c_end; c0 += 32) {
          const bool two = c0 + 16 < c_end;
          uint32_t w[4][16];
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (j < p.n_k && row_ok) {
              ld256_stream(yr[j] + c0, *reinterpret_cast<uint32_t(*)[8]>(&w[j][0]));
              if (two) ld256_stream(yr[j] + c0 + 16, *reinterpret_cast<uint32_t(*)[8]>(&w[j][8]));
            }
          float acc[32];
          tmem_ld16(taddr + c0, acc);
          if (two) tmem_ld16(taddr + c0 + 16, acc + 16);
          tmem_ld_wait();
          if (row_ok) {
#pragma unroll
            for (int q = 0; q < 32; ++q) {
              float y = __bfloat162float(__float2bfloat16_rn(acc[q]));
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (j < p.n_k) y = fmaf(gate[j], __uint_as_float((q & 1) ? (w[j][q >> 1] & 0xffff0000u) : (w[j][q >> 1] << 16)), y);
              acc[q] = y;
            }
            store16(dst + c0, acc);
            if (two) store16(dst + c0 + 16, acc + 16);
          }
        }
      } else {
        const int n0 = c.nt * 256;
        const int n_valid = min(256, p.d - n0);
        bf16* dst = (g.is_shared ? p.out_s : p.out_r) + (size_t)(c.row0 + row_in_group) * p.d + n0;
        const bool wide = (p.d & 15) == 0;
        for (int c0 = 0; c0 < n_valid; c0 += 16) {
          float acc[16];
          tmem_ld16(taddr + c0, acc);
          tmem_ld_wait();
          if (row_ok && wide && c0 + 16 <= n_valid) {
            store16(dst + c0, acc);
          } else if (row_ok) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              if (c0 + h * 8 < n_valid) {
                float v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = acc[h * 8 + q];
                store8(dst + c0 + h * 8, v);
              }
            }
          }
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
    tmem_dealloc(tmem_base, kUmmaTmemCols);
  }
}

// ----------------------------------------------------------------------------- host
struct UmmaShape {
  int d = 0, m = 0, shared_width = 0, d_ff = 0, n_outer = 1, n_r = 0, n_rp = 0, n_k = 0;
  bool plain = true;                 // no top-level router (a hierarchical layer may have one outer expert as well)
  size_t max_outer_rows = 0, max_routed_rows = 0;
};

struct UmmaBuffers {
  const void* w_gate_up = nullptr;   // [2][n_outer*d_ff][d]
  const void* w_down = nullptr;      // packed W_down
  const void* w_rep = nullptr;       // [n_outer][2*n_rp][d] padded representative rows
  const void* x_fixed = nullptr;     // hierarchical: the layer's own outer-row copy of x
  void *h_s = nullptr, *h_r = nullptr, *y_s = nullptr, *y_r = nullptr;
  const GroupStatic* gs_dev = nullptr;
  const float* topk_gate = nullptr;
  const int32_t* topk_idx = nullptr;
  const int32_t *row_token = nullptr, *row_of = nullptr;
};

typedef CUresult (*PFN_encodeTiled)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                    CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                    CUtensorMapFloatOOBfill);

struct UmmaPlan {
  bool built = false;
  char error[256] = "";
  UmmaShape shape;
  UmmaBuffers buf;
  int bn_s = 128, bn_r = 128, n_sms = 0, n_groups = 0;
  bool has_s = false, has_r = false;
  PFN_encodeTiled encode = nullptr;
  CUtensorMap x_rows;                      // x: 64 x 128 boxes of consecutive rows
  CUtensorMap b1_s, b1_r;                  // stacked gate+up rows, box heights bn_s / bn_r
  CUtensorMap a2_s, a2_r, b2_s, b2_r;      // H_s / H_r / shared W_down / routed W_down blocks
  CUtensorMap w_rep;                       // padded representative rows
};

// Neurons per gate/up tile: 128 (N = 256 MMAs, the fewest passes over the A rows) when that pads the width
// by at most 5 %, else the multiple of 8 in [96, 128] that wastes the least of the last tile.  (Measured on
// widths 864 / 1728 at 16384 tokens: 128 against 96, which pads nothing, is 12 % faster in the gate/up GEMM:
// seven instead of nine passes over the gathered rows outweigh 3.7 % of padded MMA work.  At 130 to 2000 rows the time
// of a k block hardly falls with the width (425 / 375 / 337 ns for 128 / 96 / 64), so narrower tiles that would even out
// the last round lose as well.)
inline int umma_pick_bn(int width) {
  if (width <= 0) return 128;
  if ((long long)((width + 127) / 128 * 128) * 100 <= (long long)width * 105) return 128;
  int best = 128, best_pad = (width + 127) / 128 * 128;
  for (int bn = 120; bn >= 96; bn -= 8) {
    const int pad = (width + bn - 1) / bn * bn;
    if (pad < best_pad) { best = bn; best_pad = pad; }
  }
  return best;
}

inline bool umma_encode(UmmaPlan* P, CUtensorMap* tm, const void* base, int rank, const cuuint64_t* dims,
                        const cuuint64_t* strides_bytes, const cuuint32_t* box, const char* what) {
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  for (int i = 0; i < rank; ++i)
    if (dims[i] == 0) { snprintf(P->error, sizeof(P->error), "tensor map %s: zero extent", what); return false; }
  const CUresult r = P->encode(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, (cuuint32_t)rank, const_cast<void*>(base),
                               dims, strides_bytes, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                               CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                               CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) {
    snprintf(P->error, sizeof(P->error), "cuTensorMapEncodeTiled(%s) failed with CUresult %d", what, (int)r);
    return false;
  }
  return true;
}

// [rows, cols] row-major bf16 matrix, box 64 columns x box_rows.
inline bool umma_encode_rows(UmmaPlan* P, CUtensorMap* tm, const void* base, size_t rows, size_t cols,
                             int box_rows, const char* what) {
  const cuuint64_t dims[2] = {cols, rows};
  const cuuint64_t str[1] = {cols * 2};
  const cuuint32_t box[2] = {kUmmaBK, (cuuint32_t)box_rows};
  return umma_encode(P, tm, base, 2, dims, str, box, what);
}

// Tensor maps of x for this forward: the caller's buffer for a plain layer (a host-side
// struct fill, no allocation), fixed at plan creation for a hierarchical layer.
inline bool umma_bind_x(UmmaPlan* P, const void* x_rows, int n_rows) {
  if (P->buf.x_fixed) return true;
  return umma_encode_rows(P, &P->x_rows, x_rows, (size_t)n_rows, (size_t)P->shape.d, kUmmaBM, "x");
}

// 0: plan built; 1: shape not taken by this path; -5: a driver call failed (P->error).
inline int umma_plan_create(UmmaPlan* P, const UmmaShape& s, const UmmaBuffers& buf, int n_groups) {
  P->built = false;
  P->has_s = s.shared_width > 0 && s.max_outer_rows > 0;
  P->has_r = s.n_r > 0 && s.n_k > 0 && s.max_routed_rows > 0;
  const bool has_s = P->has_s, has_r = P->has_r;
  if (!has_s && !has_r) return 1;
  if (s.d % 8 || s.m % 8 || s.shared_width % 8 || n_groups > kUmmaMaxGroups) return 1;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &q) != cudaSuccess || !fn ||
      q != cudaDriverEntryPointSuccess) {
    snprintf(P->error, sizeof(P->error), "cuTensorMapEncodeTiled entry point not found");
    return -5;
  }
  P->encode = reinterpret_cast<PFN_encodeTiled>(fn);
  P->shape = s;
  P->buf = buf;
  P->n_groups = n_groups;
  P->bn_s = umma_pick_bn(s.shared_width);
  P->bn_r = umma_pick_bn(s.m);
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&P->n_sms, cudaDevAttrMultiProcessorCount, dev);

  const size_t d = s.d, rows_w = (size_t)s.n_outer * s.d_ff;
  bool ok = true;
  // gate/up weights stacked, [2][rows_w][d]; box = 64 k x bn rows x 2 planes
  for (int shared = 0; shared < 2 && ok; ++shared) {
    const int bn = shared ? P->bn_s : P->bn_r;
    const cuuint64_t dims[3] = {d, rows_w, 2};
    const cuuint64_t str[2] = {d * 2, rows_w * d * 2};
    const cuuint32_t box[3] = {kUmmaBK, (cuuint32_t)bn, 2};
    ok = umma_encode(P, shared ? &P->b1_s : &P->b1_r, buf.w_gate_up, 3, dims, str, box, "gate/up weights");
  }
  if (ok && has_r) ok = umma_encode_rows(P, &P->a2_r, buf.h_r, s.max_routed_rows, s.m, kUmmaBM, "H routed");
  if (ok && has_s) ok = umma_encode_rows(P, &P->a2_s, buf.h_s, s.max_outer_rows, s.shared_width, kUmmaBM, "H shared");
  // W_down: shared block [d, W_s] of every outer expert; routed blocks [d, m] x N_r of every outer expert
  if (ok && has_s) {
    const cuuint64_t dims[3] = {(cuuint64_t)s.shared_width, d, (cuuint64_t)s.n_outer};
    const cuuint64_t str[2] = {(cuuint64_t)s.shared_width * 2, d * s.d_ff * 2};
    const cuuint32_t box[3] = {kUmmaBK, 256, 1};
    ok = umma_encode(P, &P->b2_s, buf.w_down, 3, dims, str, box, "shared W_down");
  }
  if (ok && has_r) {
    const cuuint64_t dims[4] = {(cuuint64_t)s.m, d, (cuuint64_t)s.n_r, (cuuint64_t)s.n_outer};
    const cuuint64_t str[3] = {(cuuint64_t)s.m * 2, d * s.m * 2, d * s.d_ff * 2};
    const cuuint32_t box[4] = {kUmmaBK, 256, 1, 1};
    ok = umma_encode(P, &P->b2_r, (const bf16*)buf.w_down + (size_t)s.shared_width * d, 4, dims, str, box,
                     "routed W_down");
  }
  if (ok && s.n_r > 0) {
    const cuuint64_t dims[3] = {d, (cuuint64_t)2 * s.n_rp, (cuuint64_t)s.n_outer};
    const cuuint64_t str[2] = {d * 2, (cuuint64_t)2 * s.n_rp * d * 2};
    const cuuint32_t box[3] = {kUmmaBK, (cuuint32_t)(2 * s.n_rp), 1};
    ok = umma_encode(P, &P->w_rep, buf.w_rep, 3, dims, str, box, "representative rows");
  }
  if (ok && buf.x_fixed)
    ok = umma_encode_rows(P, &P->x_rows, buf.x_fixed, s.max_outer_rows, d, kUmmaBM, "outer rows of x");
  if (!ok) return -5;
  // placeholders for absent operand classes (never dereferenced: such groups have no tiles)
  if (!has_r) { P->a2_r = P->a2_s; P->b2_r = P->b2_s; }
  if (!has_s) { P->a2_s = P->a2_r; P->b2_s = P->b2_r; }
  if (s.n_r == 0) P->w_rep = P->b1_s;
  cudaError_t e = cudaSuccess;
  if (e == cudaSuccess) e = cudaFuncSetAttribute(umma_grouped_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUmmaSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(umma_grouped_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUmmaSmemBytes);
  if (e == cudaSuccess) e = cudaFuncSetAttribute(umma_grouped_kernel<3>, cudaFuncAttributeMaxDynamicSharedMemorySize, kUmmaSmemBytes);
  if (e != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "cudaFuncSetAttribute: %s", cudaGetErrorString(e));
    return -5;
  }
  P->built = true;
  return 0;
}

inline void umma_plan_destroy(UmmaPlan* P) { P->built = false; }

// Row tiles per band of the tile order: about 16 MB of A rows (k_extent bf16 elements per row), an even count.
inline int umma_band_tiles(int k_extent) {
  const long long tile_bytes = (long long)kUmmaBM * k_extent * 2;
  long long n = (16ll << 20) / (tile_bytes > 0 ? tile_bytes : 1);
  n = n < 2 ? 2 : n;
  return (int)(n & ~1ll);
}

inline UmmaArgs umma_base_args(const UmmaPlan* P, const GroupRows* gr, int32_t* err_word) {
  const UmmaShape& s = P->shape;
  UmmaArgs a{};
  a.gs = P->buf.gs_dev; a.gr = gr; a.n_groups = P->n_groups; a.n_outer = s.n_outer; a.n_r = s.n_r;
  a.d = s.d; a.bn_s = P->bn_s; a.bn_r = P->bn_r; a.err = err_word;
  a.row_token = P->buf.row_token;
  a.shared_width = s.shared_width;
  a.row_of = P->buf.row_of; a.topk_gate = P->buf.topk_gate; a.n_k = s.n_k; a.y_r = (const bf16*)P->buf.y_r;
  a.x_rows_ptr = nullptr;
  return a;
}

// Whether the down GEMM of the shared experts runs after that of the routed ones and combines in its epilogue: Y_s is neither
// written nor read back, and the routed rows are read under its multiplies.  Bound by the epilogue's gathers (a thread reads
// 32-byte pieces of n_k rows), which a tile's multiplies must cover, and by the last round of tiles, which no routed tiles fill up any
// more: taken when the SMs' idle time in that round (425 ns per 64-wide k block) is at most a third of the combine's own time (3 us and
// the rows at 5.5 TB/s).  With / without, both forced: 8B-shaped 700 rows 106 / 101 us, 7B-shaped 300 rows 79.0 / 76.4, 13B-shaped 300 rows
// 105 / 99 (not taken), 8B-shaped 1400 and 7B-shaped 2500 rows even (not taken), 8B-shaped 1000 / 2048 / 8192 rows 131 / 221 / 716 against
// 143 / 229 / 738, 7B-shaped 4000 / 8000 rows 500 / 946 against 513 / 979, 13B-shaped 4096 / 16384 rows 615 / 2310 against 640 / 2397.
// Eight epilogue warps, each with half of the columns, keep twice the gathers of four in flight (8B-shaped 2048 rows 205.5 -> 198.7 us);
// fetching the routed rows of the next columns ahead as well (233 registers) was slower.
inline bool umma_folds_combine(const UmmaPlan* P, int R, int n_k, int d) {
  if (!P->has_s || !P->has_r || n_k < 1 || n_k > 4 || d % 16 != 0) return false;
  const int tiles = (R + kUmmaBM - 1) / kUmmaBM * ((d + 255) / 256), over = tiles % P->n_sms;
  const double idle = over ? (1.0 - (double)over / P->n_sms) * 0.425 * ((P->shape.shared_width + kUmmaBK - 1) / kUmmaBK) : 0.0;
  return 3.0 * idle <= 3.0 + (double)R * d * 2 * (n_k + 3) / 5.5e6;
}

// Enqueues the gate/up and the down GEMM over all groups.  Requires umma_bind_x for this forward.  which: bit 0 the
// gate/up GEMM, bit 1 the down GEMM.  early_rows: rows of the shared experts where the host knows them (plain layer).  Returns the number of kernels launched, or -1 (P->error).
inline int umma_forward(UmmaPlan* P, const GroupRows* gr, const void* x_rows, int32_t* err_word,
                        cudaStream_t st, cudaEvent_t mid, bool dep, int which, int early_rows,
                        bool skip_shared = false) {
  const UmmaShape& s = P->shape;
  UmmaArgs a = umma_base_args(P, gr, err_word);
  a.out_s = (bf16*)P->buf.h_s; a.out_r = (bf16*)P->buf.h_r; a.ld_out_s = s.shared_width; a.ld_out_r = s.m;
  a.x_rows_ptr = (const bf16*)x_rows;
  a.band_mt = umma_band_tiles(s.d);
  a.early_rows = early_rows;
  if (which & 1)
    launch_kernel(dep, umma_grouped_kernel<1>, dim3(P->n_sms), dim3(kUmmaThreads + kUmmaGatherThreads), umma_smem_bytes(P->n_groups),
                  st, P->x_rows, P->x_rows, P->b1_s, P->b1_r, a);
  if (mid && (which & 1)) cudaEventRecord(mid, st);
  a.out_s = (bf16*)P->buf.y_s; a.out_r = (bf16*)P->buf.y_r; a.ld_out_s = s.d; a.ld_out_r = s.d;
  a.band_mt = umma_band_tiles(s.shared_width > s.m ? s.shared_width : s.m);
  a.skip_groups = skip_shared ? s.n_outer : 0;
  if (which & 2)
    launch_kernel(dep, umma_grouped_kernel<2>, dim3(P->n_sms), dim3(kUmmaThreads), umma_smem_bytes(P->n_groups), st, P->a2_s,
                  P->a2_r, P->b2_s, P->b2_r, a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "tensor-core GEMM launch: %s", cudaGetErrorString(e));
    return -1;
  }
  return (which & 1) + ((which >> 1) & 1);
}

// Down GEMM of the shared experts with the combine, after the routed experts' (the other forms' down GEMM with skip_shared).
inline int umma_fold_forward(UmmaPlan* P, const GroupRows* gr, int n_rows, bf16* out, int32_t* err_word, cudaStream_t st, bool dep) {
  const UmmaShape& s = P->shape;
  UmmaArgs a = umma_base_args(P, gr, err_word);
  a.out_s = out; a.ld_out_s = s.d; a.early_rows = n_rows;
  a.band_mt = umma_band_tiles(s.shared_width);
  if (launch_kernel(dep, umma_grouped_kernel<3>, dim3(P->n_sms), dim3(kUmmaThreads + 128), umma_smem_bytes(P->n_groups), st, P->a2_s, P->a2_s,
                    P->b2_s, P->b2_s, a) != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "shared down GEMM launch failed");
    return -1;
  }
  return 1;
}

}  // namespace cmoe
