// Expert GEMMs on CTA pairs with the operands turned round: 256 weight rows on the M side of the MMA (128 per CTA) and up to 256
// tokens on the N side (half of them staged by each CTA, read by both).
//
// Bound: the tensor cores at the rate that the power limit allows (a round of 256 x 160 tiles on all pairs runs at 1.41 PFLOP/s even
// with every operand in L2), below ~1500 rows also the weights' way from DRAM.  Either way padded multiplies are lost, and with the
// tokens on N a group pads to a multiple of 32 columns instead of 128 or 256 rows: its tokens are cut into equal tiles of at most
// 256, so an expert with 143 rows costs 160 columns and one with 341 costs 352 (192 + 160).  Neurons pad to 128 per tile.
//
//   MODE 1, gate/up: the tile's 128 neurons are 64 per CTA, their gate and up rows interleaved by the TMA box (k, plane, neuron),
//           so that accumulator lanes 2i and 2i + 1 hold gate and up of a neuron: one shuffle brings them together, a second one
//           makes a 4-byte store of two neighbouring neurons of a token.
//   MODE 2, down:    128 output channels per CTA; one shuffle makes a 4-byte store of two channels.
// Roles, barriers and the gather of routed rows are those of umma2_gemm.cuh; eight epilogue warps per CTA, each with 32 of every 64
// columns (four: 6.4 us from a 256-column tile's last MMA to its last store, eight: 4.2).
//
// Chained forwards with single CTAs and token-major gate/up pairs alone / as umma_pick_forms chooses now (one side's runs differ by 0.3-3 %):
// hierarchical 2000 / 4096 tokens 928 / 1570 -> 878 / 1491 us, 8B-shaped 1000 rows 146.2 -> 142.7, 7B-shaped 400 / 512 / 1000 rows 101.9 / 105.3 /
// 161.3 -> 88.7 / 98.8 / 156.8, 13B-shaped 600 / 1000 rows 171.5 / 220.4 -> 151.8 / 205.4.
// Not taken: the k blocks of a tile started at another place per pair (even), the routed experts' first weights fetched into L2 under the
// shared experts' tiles (8B-shaped 1000 rows +0 to +6 us: it delays those tiles by what it saves later), shared and routed tiles on
// separate pairs at the same time (+3 to +20 us).
#pragma once

#include <cmath>

#include "umma2_gemm.cuh"
#include "umma_decode.cuh"

namespace cmoe {

constexpr int kUtThreads1 = kU2Threads1 + 128, kUtThreads2 = kUmmaThreads + 128;   // four more epilogue warps
constexpr int kUtMaxTok = 256;           // tokens per tile: N of the MMA
constexpr int kUtGrain = 32;             // N is a multiple of 32 on CTA pairs
constexpr int kUtBoxes = kUtMaxTok / kUtGrain;

// Maps of one token matrix: entry i has boxes of 16 (i + 1) rows, the half of a tile of 32 (i + 1) tokens.
struct TokenMaps { CUtensorMap m[kUtBoxes]; };

// A group's tokens in equal tiles.
struct TokenCut {
  int n, width;                          // tiles; tokens per tile but the last, a multiple of 32
  __host__ __device__ explicit TokenCut(int count) {
    n = (count + kUtMaxTok - 1) / kUtMaxTok;
    const int even = n > 0 ? (count + n - 1) / n : 0;
    width = (even + kUtGrain - 1) / kUtGrain * kUtGrain;
  }
  // columns of tile i
  __host__ __device__ int columns(int count, int i) const {
    const int left = count - i * width;
    return left >= width ? width : (left + kUtGrain - 1) / kUtGrain * kUtGrain;
  }
};

struct TurnedCoord { int g, tok0, cols, nt, row0, count; };   // first token inside the group, columns, weight tile

__device__ __forceinline__ TurnedCoord umma2t_tile_in(const UmmaArgs& p, int g, const GroupRows r, int n_tiles, int local) {
  // bands of token tiles, token tiles fastest inside a band, then weight tiles (see umma_tile_in)
  const TokenCut cut(r.count);
  const int band_t = max(p.band_mt >> 1, 1);
  const int per_band = band_t * n_tiles;
  const int band = local / per_band, in_band = local - band * per_band;
  const int cur = min(band_t, cut.n - band * band_t);
  TurnedCoord c;
  const int i = band * band_t + in_band % cur;
  c.g = g; c.nt = in_band / cur; c.tok0 = i * cut.width; c.cols = cut.columns(r.count, i); c.row0 = r.row0; c.count = r.count;
  return c;
}

template <int MODE>
__device__ __forceinline__ TurnedCoord umma2t_decode(const UmmaArgs& p, const int32_t* tile_start, const GroupRows* rows, int t) {
  int lo = 0, hi = p.n_groups;
  while (hi - lo > 1) {
    const int mid = (lo + hi) >> 1;
    if (tile_start[mid] <= t) lo = mid; else hi = mid;
  }
  return umma2t_tile_in(p, lo, rows[lo], umma_n_tiles<MODE>(p, lo), t - tile_start[lo]);
}

// v[q]: this lane's accumulators of 16 tokens, lane pairs hold two rows that belong together.  Returns the even and the odd row's
// values of 8 tokens, the even ones in even lanes and the odd ones in odd lanes.
__device__ __forceinline__ void pair_exchange(const float (&v)[16], bool odd, float (&even_row)[8], float (&odd_row)[8]) {
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float own = odd ? v[2 * q + 1] : v[2 * q];
    const float other = __shfl_xor_sync(0xffffffffu, odd ? v[2 * q] : v[2 * q + 1], 1);
    even_row[q] = odd ? other : own;
    odd_row[q] = odd ? own : other;
  }
}

// MODE 1 gate/up, MODE 2 down.
template <int MODE>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(MODE == 1 ? kUtThreads1 : kUtThreads2, 1)
umma2t_grouped_kernel(const __grid_constant__ CUtensorMap tm_w_s, const __grid_constant__ CUtensorMap tm_w_r,
                      const __grid_constant__ TokenMaps tm_t_s, const __grid_constant__ TokenMaps tm_t_r, const UmmaArgs p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  const uint32_t base = (raw + 1023u) & ~1023u;
  uint8_t* gen = smem_raw + (base - raw);
  const uint32_t bars = base + kU2Stages * kU2StageBytes;
  uint8_t* bars_gen = gen + kU2Stages * kU2StageBytes;
  const uint32_t full0 = bars, empty0 = bars + 64, accf0 = bars + 128, acce0 = bars + 144, tbl_bar = bars + 168, afull0 = bars + 192;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars_gen + 160);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(bars_gen + 164);
  int32_t* tile_start = reinterpret_cast<int32_t*>(bars_gen + 256);
  GroupRows* rows = reinterpret_cast<GroupRows*>(tile_start + p.n_groups + 1);

  const int warp = warp_index(), lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const bool leader = rank == 0;
  const int pair_id = blockIdx.x >> 1, n_pairs = gridDim.x >> 1;

  if (threadIdx.x == 0) {
    const uint32_t full_count = MODE == 1 ? 3 : 1;      // gate/up: plus one relay arrival per CTA
    for (int s = 0; s < kU2Stages; ++s) {
      mbar_init(full0 + 8 * s, full_count); mbar_init(empty0 + 8 * s, 1); mbar_init(afull0 + 8 * s, kUmmaGatherThreads);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(accf0 + 8 * b, 1); mbar_init(acce0 + 8 * b, 16); }
    mbar_init(tbl_bar, 1);
    *abort_flag = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  cluster_sync_all();                         // both CTAs' barriers exist before any remote use
  if (warp == 1) {
    tmem_alloc2(smem_u32(tmem_slot), kUmmaTmemCols);
    tmem_relinquish2();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  const int k_blocks_fixed = (p.d + kUmmaBK - 1) / kUmmaBK;
  // table and tiles that need none: as in umma_grouped_kernel
  const int early_n = MODE == 1 && p.early_rows > 0 ? (p.shared_width + p.bn_s - 1) / p.bn_s : 0;
  const int early_tiles = TokenCut(p.early_rows).n * early_n;
  if (warp == 2) {
    for (int g = lane; g < p.n_groups; g += 32) tile_start[g + 1] = umma_n_tiles<MODE>(p, g);
    if (MODE == 1) { grid_dep_wait(); grid_dep_trigger(); }
    for (int g = lane; g < p.n_groups; g += 32) {
      const GroupRows gr = p.gr[g];
      rows[g] = gr;
      tile_start[g + 1] *= MODE == 2 && g < p.skip_groups ? 0 : TokenCut(gr.count).n;
    }
    __syncwarp();
    warp_prefix(tile_start, p.n_groups, lane);
    __syncwarp();
    if (lane == 0) mbar_arrive(tbl_bar);
    if (MODE == 2) { grid_dep_wait(); grid_dep_trigger(); }     // what follows may count on the gate/up GEMM
  }
  bool seen = false;
  auto tile_at = [&](int t, TurnedCoord& c, GroupStatic& g, bool whole_warp, bool& ok) {
    if (MODE == 1 && t < early_tiles) {
      GroupRows all; all.row0 = 0; all.count = p.early_rows;
      c = umma2t_tile_in(p, 0, all, early_n, t);
      g.w_row0 = 0; g.width = p.shared_width; g.wd_offset = 0; g.is_shared = 1; g.outer = 0;
      return true;
    }
    if (!seen) {
      ok = mbar_wait(tbl_bar, 0, abort_flag, p.err, kErrWaitFull);
      if (whole_warp) ok = __all_sync(0xffffffffu, ok);
      if (!ok) return false;
      if (MODE == 1) grid_dep_wait();
      seen = true;
    }
    if (t >= tile_start[p.n_groups]) return false;
    c = umma2t_decode<MODE>(p, tile_start, rows, t);
    g = p.gs[c.g];
    return true;
  };

  if (warp == 0) {
    // ------------------------------------------------------------ TMA producer (whole warp, one lane issues)
    uint32_t it = 0, n_ahead = 0;
    bool waited = false;
    bool ok = true;
    for (int t = pair_id; ok; t += n_pairs) {
      TurnedCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, true, ok)) break;
      const int half = c.cols >> 1;                                        // token rows that this CTA stages
      const int tok_row = c.row0 + c.tok0 + (int)rank * half;
      const CUtensorMap* tw = g.is_shared ? &tm_w_s : &tm_w_r;
      const CUtensorMap* tt = &(g.is_shared ? tm_t_s : tm_t_r).m[c.cols / kUtGrain - 1];
      const bool by_threads = MODE == 1 && !g.is_shared;                   // the gather warps fetch the tokens
      int k_blocks, w_bytes, w_row, j = 0;
      if (MODE == 1) {
        const int bn = g.is_shared ? p.bn_s : p.bn_r;                      // neurons of the pair: bn / 2 per CTA, gate and up rows
        k_blocks = k_blocks_fixed;
        w_bytes = bn * kUmmaBK * 2;
        w_row = g.w_row0 + c.nt * bn + (int)rank * (bn >> 1);
      } else {
        k_blocks = (g.width + kUmmaBK - 1) / kUmmaBK;
        w_bytes = kU2ABytes;
        w_row = c.nt * 256 + (int)rank * 128;
        j = g.is_shared ? 0 : (c.g - p.n_outer) - g.outer * p.n_r;
      }
      const int stage_tx = 2 * (w_bytes + (by_threads ? 0 : half * kUmmaBK * 2));
      auto load_w = [&](int kb, uint32_t sw, uint32_t fb) {
        if (MODE == 1) tma2_load_3d(sw, tw, fb, kb * kUmmaBK, 0, w_row);   // gate and up rows of a neuron next to each other
        else if (g.is_shared) tma2_load_3d(sw, tw, fb, kb * kUmmaBK, w_row, g.outer);
        else tma2_load_4d(sw, tw, fb, kb * kUmmaBK, w_row, j, g.outer);
      };
      if (MODE == 2 && it == 0 && !waited) {
        n_ahead = min(kU2Stages, k_blocks);
        for (uint32_t i = 0; i < n_ahead; ++i) {
          if (elect_one()) {
            if (leader) mbar_expect_tx(full0 + 8 * i, stage_tx);
            load_w(i, base + i * kU2StageBytes, mapa_shared(full0 + 8 * i, 0));
          }
          __syncwarp();
        }
        grid_dep_wait();
        waited = true;
      }
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const uint32_t s = it % kU2Stages, n = it / kU2Stages;
        if (!mbar_wait_warp(empty0 + 8 * s, (n & 1) ^ 1, abort_flag, p.err, kErrWaitEmpty)) { ok = false; break; }
        const uint32_t fb_local = full0 + 8 * s;
        const uint32_t fb = mapa_shared(fb_local, 0);               // the leader's barrier
        const uint32_t sw = base + s * kU2StageBytes, st = sw + kU2ABytes;
        if (elect_one()) {
          if (MODE == 1 || it >= n_ahead) {
            if (leader) mbar_expect_tx(fb_local, stage_tx);
            load_w(kb, sw, fb);
          }
          if (!by_threads) tma2_load_2d(st, tt, fb, kb * kUmmaBK, tok_row);
        }
        __syncwarp();
      }
    }
    if (!ok) for (int i = 0; i < 200; ++i) __nanosleep(1000);
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (leader CTA only; whole warp, one lane issues)
    if (leader) {
      uint32_t it = 0, tile_n = 0;
      bool ok = true;
      for (int t = pair_id; ok; t += n_pairs, ++tile_n) {
        TurnedCoord c;
        GroupStatic g;
        if (!tile_at(t, c, g, true, ok)) break;
        const int k_blocks = MODE == 1 ? k_blocks_fixed : (g.width + kUmmaBK - 1) / kUmmaBK;
        const uint32_t idesc = umma2_idesc(c.cols);
        const uint32_t buf = tile_n & 1, use = tile_n >> 1;
        if (!mbar_wait_warp(acce0 + 8 * buf, (use & 1) ^ 1, abort_flag, p.err, kErrWaitAccEmpty)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_tmem = tmem_base + buf * 256;
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const uint32_t s = it % kU2Stages, n = it / kU2Stages;
          if (!mbar_wait_warp(full0 + 8 * s, n & 1, abort_flag, p.err, kErrWaitFull)) { ok = false; break; }
          if (MODE == 1) asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          tc_fence_after();
          const uint32_t sw = base + s * kU2StageBytes, st = sw + kU2ABytes;
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kUmmaBK / 16; ++k)
              umma2_bf16(d_tmem, umma_smem_desc(sw + k * 32), umma_smem_desc(st + k * 32), idesc, (kb | k) != 0 ? 1u : 0u);
            umma2_commit_both(empty0 + 8 * s);
          }
          __syncwarp();
        }
        if (ok && elect_one()) umma2_commit_both(accf0 + 8 * buf);
        __syncwarp();
      }
    }
  } else if (MODE == 1 && warp == 10) {
    // ------------------------------------------------------------ relay (gate/up, both CTAs): see umma2_grouped_kernel
    if (lane == 0) {
      uint32_t it = 0;
      bool ok = true;
      for (int t = pair_id; ok; t += n_pairs) {
        TurnedCoord c;
        GroupStatic g;
        if (!tile_at(t, c, g, false, ok)) break;
        for (int kb = 0; kb < k_blocks_fixed; ++kb, ++it) {
          const uint32_t s = it % kU2Stages, n = it / kU2Stages;
          if (!mbar_wait(afull0 + 8 * s, n & 1, abort_flag, p.err, kErrWaitFull)) { ok = false; break; }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
          mbar_arrive_remote(mapa_shared(full0 + 8 * s, 0));
        }
      }
    }
  } else if (MODE == 1 && warp >= 6 && warp < 10) {
    // ------------------------------------------------------------ token gather (gate/up, warps 6..9, both CTAs)
    // Eight consecutive threads cover one 128-byte row segment, 16 rows per pass, as many passes as half the tile has rows.
    const int gt = threadIdx.x - kUmmaThreads;
    const int ch = gt & 7, r_sub = gt >> 3;
    uint32_t it = 0;
    bool ok = true;
    for (int t = pair_id; ok; t += n_pairs) {
      TurnedCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, false, ok)) break;
      const bool mine = !g.is_shared;
      const int half = c.cols >> 1;
      const bf16* src_row[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        src_row[i] = nullptr;
        const int in_half = i * 16 + r_sub, r = c.tok0 + (int)rank * half + in_half;
        if (mine && in_half < half && r < c.count)    // columns past the group are left as they are: nothing of them is stored
          src_row[i] = p.x_rows_ptr + (size_t)__ldcg(p.row_token + c.row0 + r) * p.d;
      }
      for (int kb = 0; kb < k_blocks_fixed; ++kb, ++it) {
        const uint32_t s = it % kU2Stages, n = it / kU2Stages;
        if (!mbar_wait(empty0 + 8 * s, (n & 1) ^ 1, abort_flag, p.err, kErrWaitEmpty)) { ok = false; break; }
        const uint32_t ab = afull0 + 8 * s;
        if (mine) {
          const int k = kb * kUmmaBK + ch * 8;
          const uint32_t bytes = k < p.d ? 16u : 0u;                        // zero-fill past the end of the row
          const int k_src = k < p.d ? k : 0;
          const uint32_t st = base + s * kU2StageBytes + kU2ABytes;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int r = i * 16 + r_sub;
            if (src_row[i])
              asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                         ::"r"(st + r * 128 + ((ch ^ (r & 7)) << 4)), "l"(src_row[i] + k_src), "r"(bytes)
                         : "memory");
          }
          asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(ab) : "memory");
        } else {
          mbar_arrive(ab);
        }
      }
    }
    if (!ok) asm volatile("cp.async.wait_all;" ::: "memory");
  } else {
    // ------------------------------------------------------------ epilogue (eight warps, both CTAs: 2..5, then 11..14 or 6..9)
    const int quad = warp & 3, first = warp < 6 ? 0 : 32;             // columns first, first + 64, ..., 32 at a time
    uint32_t tile_n = 0;
    bool ok = true;
    for (int t = pair_id; ok; t += n_pairs, ++tile_n) {
      TurnedCoord c;
      GroupStatic g;
      if (!tile_at(t, c, g, false, ok)) break;
      const uint32_t buf = tile_n & 1, use = tile_n >> 1;
      const int left = c.count - c.tok0;                             // tokens of the group from this tile on
      const int n_tok = min(left, c.cols);
      if (!mbar_wait(accf0 + 8 * buf, use & 1, abort_flag, p.err, kErrWaitAccFull)) { ok = false; break; }
      tc_fence_after();
      const uint32_t taddr = tmem_base + buf * 256 + ((uint32_t)(quad * 32) << 16);
      bf16* out = g.is_shared ? p.out_s : p.out_r;
      if (MODE == 1) {
        // lanes 2i, 2i + 1: gate and up of neuron i of this warp's 16.  After two exchanges a lane holds two neighbouring neurons
        // of four of the 16 tokens: lanes 4i .. 4i + 3 tokens 4q + (0, 1, 2, 3).
        const int bn = g.is_shared ? p.bn_s : p.bn_r, ld = g.is_shared ? p.ld_out_s : p.ld_out_r;
        const int local = quad * 16 + ((lane >> 2) << 1);            // neurons local, local + 1 of the CTA's bn / 2
        const int n0 = c.nt * bn + (int)rank * (bn >> 1) + local;
        const bool live = local < (bn >> 1) && n0 < g.width;
        bf16* dst = out + (size_t)(c.row0 + c.tok0) * ld + n0;
        for (int c0 = first; c0 < n_tok; c0 += 64) {
          float v[2][16];
          tmem_ld16(taddr + c0, v[0]);
          tmem_ld16(taddr + c0 + 16, v[1]);             // past the tile's columns: other columns of the buffers, not stored
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float gt[8], up[8], h[8];
            pair_exchange(v[i], lane & 1, gt, up);
#pragma unroll
            for (int q = 0; q < 8; ++q) h[q] = swiglu_fast(gt[q], up[q]);
            const bool upper = lane & 2;
#pragma unroll
            for (int q = 0; q < 4; ++q) {                            // tokens 4q + (lane & 1) and 4q + 2 + (lane & 1)
              const float keep = upper ? h[2 * q + 1] : h[2 * q];
              const float got = __shfl_xor_sync(0xffffffffu, upper ? h[2 * q] : h[2 * q + 1], 2);
              const uint32_t two = pack_bf16x2(upper ? got : keep, upper ? keep : got);
              const int tok = c0 + 16 * i + 4 * q + (lane & 3);
              if (live && tok < n_tok) *reinterpret_cast<uint32_t*>(dst + (size_t)tok * ld) = two;
            }
          }
        }
      } else {
        const int ch = c.nt * 256 + (int)rank * 128 + quad * 32 + (lane & ~1);     // channels ch, ch + 1
        const bool live = ch < p.d;
        bf16* dst = out + (size_t)(c.row0 + c.tok0) * p.d + ch;
        for (int c0 = first; c0 < n_tok; c0 += 64) {
          float v[2][16];
          tmem_ld16(taddr + c0, v[0]);
          tmem_ld16(taddr + c0 + 16, v[1]);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float lo[8], hi[8];
            pair_exchange(v[i], lane & 1, lo, hi);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const int tok = c0 + 16 * i + 2 * q + (lane & 1);
              const uint32_t two = pack_bf16x2(lo[q], hi[q]);
              if (live && tok < n_tok) *reinterpret_cast<uint32_t*>(dst + (size_t)tok * p.d) = two;
            }
          }
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(mapa_shared(acce0 + 8 * buf, 0));
    }
  }
  tc_fence_before();
  cluster_sync_all();                         // the peer is done with this CTA's smem and TMEM use
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc2(tmem_base, kUmmaTmemCols);
  }
}

// ----------------------------------------------------------------------------- host
struct Umma2tPlan {
  bool built = false;
  int bn_s = 128, bn_r = 128;      // neurons per gate/up tile
  CUtensorMap w1_s, w1_r;          // gate/up rows, boxes of 64 k x (gate, up) x bn / 2 neurons
  TokenMaps x, h_s, h_r;           // x of this forward (plain layer: only the boxes that it uses)
};

// Neurons per gate/up tile: the least multiple of 16 that covers the width with as few tiles of 128.
inline int umma2t_bn(int width) {
  if (width <= 0) return 128;
  const int n = (width + 127) / 128;
  return ((width + n - 1) / n + 15) / 16 * 16;
}

inline bool umma2t_plan_create(UmmaPlan* P, Umma2tPlan* Q) {
  const UmmaShape& s = P->shape;
  const size_t d = s.d, rows_w = (size_t)s.n_outer * s.d_ff;
  bool ok = true;
  Q->bn_s = umma2t_bn(P->has_s ? s.shared_width : 0);
  Q->bn_r = umma2t_bn(P->has_r ? s.m : 0);
  for (int shared = 0; shared < 2 && ok; ++shared) {
    const cuuint64_t dims[3] = {d, 2, rows_w};
    const cuuint64_t str[2] = {rows_w * d * 2, d * 2};
    const cuuint32_t box[3] = {kUmmaBK, 2, (cuuint32_t)((shared ? Q->bn_s : Q->bn_r) / 2)};
    ok = umma_encode(P, shared ? &Q->w1_s : &Q->w1_r, P->buf.w_gate_up, 3, dims, str, box, "gate/up weights (turned)");
  }
  for (int i = 0; i < kUtBoxes && ok; ++i) {
    const int rows = 16 * (i + 1);
    if (P->has_s) ok = umma_encode_rows(P, &Q->h_s.m[i], P->buf.h_s, s.max_outer_rows, s.shared_width, rows, "H shared (turned)");
    if (ok && P->has_r) ok = umma_encode_rows(P, &Q->h_r.m[i], P->buf.h_r, s.max_routed_rows, s.m, rows, "H routed (turned)");
    if (ok && P->buf.x_fixed) ok = umma_encode_rows(P, &Q->x.m[i], P->buf.x_fixed, s.max_outer_rows, d, rows, "outer rows of x (turned)");
  }
  if (!ok) return false;
  if (!P->has_s) Q->h_s = Q->h_r;
  if (!P->has_r) Q->h_r = Q->h_s;
  cudaError_t e = cudaFuncSetAttribute(umma2t_grouped_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kU2SmemBytes);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(umma2t_grouped_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, kU2SmemBytes);
  if (e != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "cudaFuncSetAttribute (turned CTA pair): %s", cudaGetErrorString(e));
    return false;
  }
  Q->built = true;
  return true;
}

// As umma2_forward.  A plain layer's x: boxes for the widths that its shared experts' tiles have.
inline int umma2t_forward(UmmaPlan* P, Umma2tPlan* Q, int grid, DecodePlan* D, const GroupRows* gr, const void* x_rows, int n_rows,
                          int32_t* err_word, cudaStream_t st, cudaEvent_t mid, bool dep, int which, int early_rows,
                          bool skip_shared = false) {
  const UmmaShape& s = P->shape;
  UmmaArgs a = umma_base_args(P, gr, err_word);
  a.bn_s = Q->bn_s; a.bn_r = Q->bn_r;
  a.out_s = (bf16*)P->buf.h_s; a.out_r = (bf16*)P->buf.h_r; a.ld_out_s = s.shared_width; a.ld_out_r = s.m;
  a.x_rows_ptr = (const bf16*)x_rows;
  a.band_mt = umma_band_tiles(s.d);
  a.early_rows = early_rows;
  if (which & 1) {
    if (!P->buf.x_fixed) {
      const TokenCut cut(n_rows);
      for (int i = 0; i < cut.n; i += cut.n > 1 ? cut.n - 1 : 1) {          // the first and the last tile
        const int cols = cut.columns(n_rows, i);
        if (!umma_encode_rows(P, &Q->x.m[cols / kUtGrain - 1], x_rows, (size_t)n_rows, (size_t)s.d, cols / 2, "x (turned)")) return -1;
      }
    }
    launch_kernel(dep, umma2t_grouped_kernel<1>, dim3(grid), dim3(kUtThreads1), umma2_smem_bytes(P->n_groups), st,
                  Q->w1_s, Q->w1_r, Q->x, Q->x, a);
  }
  if (mid && (which & 1)) cudaEventRecord(mid, st);
  a.out_s = (bf16*)P->buf.y_s; a.out_r = (bf16*)P->buf.y_r; a.ld_out_s = s.d; a.ld_out_r = s.d;
  a.band_mt = umma_band_tiles(s.shared_width > s.m ? s.shared_width : s.m);
  a.skip_groups = skip_shared ? s.n_outer : 0;
  if (which & 2)
    launch_kernel(dep, umma2t_grouped_kernel<2>, dim3(grid), dim3(kUtThreads2), umma2_smem_bytes(P->n_groups), st, D->wd_s,
                  D->wd_r, Q->h_s, Q->h_r, a);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    snprintf(P->error, sizeof(P->error), "turned CTA-pair GEMM launch: %s", cudaGetErrorString(e));
    return -1;
  }
  return (which & 1) + ((which >> 1) & 1);
}

// ----------------------------------------------------------------------------- tile shapes
constexpr int kPairMinRows = 256;        // outer rows from which the expert GEMMs may run on CTA pairs
constexpr int kPairLargeRows = 2048;     // outer rows from which the part runs at its power limit for the whole forward

enum class GemmForm { kSingle, kPair, kTurned };     // umma_gemm.cuh, umma2_gemm.cuh, this file
struct GemmForms { GemmForm gate_up = GemmForm::kSingle, down = GemmForm::kSingle; };

// Expected number of `rows`-row tiles of a group whose rows are binomial with this mean and deviation.
inline double umma_expected_tiles(double mean, double dev, int rows) {
  double n = 0.0;
  for (int j = 0; j * rows < mean + 5.0 * dev + 1.0; ++j) {
    const double z = dev > 1e-3 ? (j * rows + 0.5 - mean) / dev : (j * rows + 0.5 > mean ? 9.0 : -9.0);
    n += 0.5 * erfc(z * 0.70710678);
  }
  return n;
}

// Busiest CTA (or pair) of n_slots when n_s tiles of cost c_s and then n_r tiles of cost c_r are dealt round-robin.  The load changes
// with the slot only where one of the two runs of tiles ends.
inline double umma_busiest(int n_s, double c_s, int n_r, double c_r, int n_slots) {
  const int ends_s = n_s % n_slots, ends_all = (n_s + n_r) % n_slots;
  double worst = 0.0;
  for (int i : {0, ends_s, ends_all}) {
    const int s = n_s / n_slots + (i < ends_s), all = (n_s + n_r) / n_slots + (i < ends_all);
    const double load = s * c_s + (all - s) * c_r;
    worst = load > worst ? load : worst;
  }
  return worst;
}

// Token columns that a group of `rows` rows takes in turned tiles.
inline int umma2t_columns(int rows) {
  const TokenCut cut(rows);
  return cut.n > 0 ? (cut.n - 1) * cut.width + cut.columns(rows, cut.n - 1) : 0;
}

// Which tiles the two GEMMs run on, for R outer rows and n_sel selections over n_routed groups (even load assumed).  All are
// persistent kernels whose tiles are dealt round-robin.
//   Below kPairLargeRows: a few rounds, so what counts for gate/up is the busiest SM, or the weights' way from DRAM (5.8 TB/s) where
// that takes longer.  Per 64-wide k block a 128 x 256 tile takes 425 ns on a single CTA (the operands' round trip through four
// stages), a token-major tile 350 on a pair, a turned tile of N tokens 120 + 0.95 N (240 at least); pairs have to win by 9 %.  The load is
// taken as expected and, with a third of the weight, with a fifth more routed tiles, for skewed routing.  The constants are those that choose
// best over 251 measured sizes (7B-, 8B- and 13B-shaped, hierarchical and 28 random shapes): 1.6 % above the fastest form (geometric mean, the
// runs themselves differ by about 1 %), 4.4 % with single CTAs and token-major pairs only.
//   From there on the part runs at its power limit and every padded multiply costs energy: the form with the fewest, single
// tiles counted 8 % dearer for the operands that both of a pair's CTAs would have shared (over 70 measured sizes from 2048 rows on the choice is 1.0 %
// above the best form, geometric mean; 1.3 % with 5 %, 1.9 % where pairs had to win by another 3 %: 8B-shaped 3200 / 14592 / 16384 rows
// 307 / 1314 / 1475 on pairs, 322 / 1448 / 1633 on single CTAs).
//   Down: turned tiles where an expert has more than 128 rows (a single tile's height) and K is more than seven k blocks (448 neurons even
// or 2 % slower, 496 neurons 4696 rows 445 against 484).
// Whole forwards, gate/up on single CTAs / token-major pairs / turned pairs, each with single and turned down tiles (alternating, us):
//   7B-shaped   300 rows  79 79 / 85 86 / 80 80      512  108 104 / 102 96 / 100 95     710  119 117 / 112 110 / 114 112
//              1000      161 160 / 157 157 / 153 154  1470 212 211 / 208 202 / 208 206   2047 285 271 / 275 268 / 283 268
//   13B-shaped  600      162 150 / 151 142 / 147 137  1000 217 210 / 230 231 / 222 217   4096 687 664 / 666 640 / 651 636
//   8B-shaped (448 neurons: turned tiles pad them by 14 %)
//               300       99 101 / 98 100 / 97 95    1000 150 151 / 141 142 / 140 139    1500 182 182 / 171 172 / 178 178
//              8192      783 771 / 730 732 / 745 750
//   hierarchical 700 tokens 569 564 / 599 622 / 595 589   2048 986 936 / 956 866 / 892 858   4096 1531 1509 / 1602 1626 / 1506 1478
// Down, turned / token-major on pairs (from kPairLargeRows on, where the turned tiles pad as much): 13B-shaped 16384 rows 2426 / 2380, 12288 even;
// 7B-shaped 8192 rows even; where they pad less, 7B-shaped 4096 rows (1376 columns against 1536) 497 / 505.
inline GemmForms umma_pick_forms(const UmmaPlan* P, int pair_grid, int R, int n_sel, int n_routed, int gemm_path) {
  GemmForms f;
  if (gemm_path == 2 || R < kPairMinRows) return f;
  const UmmaShape& s = P->shape;
  const double mean = P->has_r && n_routed > 0 ? (double)n_sel / n_routed : 0.0;
  const int rows_s = P->has_s ? (R + s.n_outer - 1) / s.n_outer : 0, rows_r = (int)ceil(mean);
  auto up = [](int v, int unit) { return (double)((v + unit - 1) / unit * unit); };
  auto work = [&](double cols_s, int unit_s, double cols_r, int unit_r) {       // neuron rows x token columns, padded
    return s.n_outer * cols_s * up(s.shared_width, unit_s) + n_routed * cols_r * up(s.m, unit_r);
  };
  const double pair = work(up(rows_s, 256), P->bn_s, up(rows_r, 256), P->bn_r);
  const double turned = work(umma2t_columns(rows_s), 128, umma2t_columns(rows_r), 128);
  // equal work: token-major pairs (shorter epilogue: 7B-shaped profiling chunk of 2048 rows 306 against 309 us)
  const GemmForm on_pairs = turned < 0.97 * pair ? GemmForm::kTurned : GemmForm::kPair;
  if (gemm_path == 3) {
    f.gate_up = on_pairs;
    f.down = GemmForm::kTurned;
    return f;
  }
  if (R >= kPairLargeRows) {
    if ((turned < pair ? turned : pair) < 1.08 * work(up(rows_s, 128), P->bn_s, up(rows_r, 128), P->bn_r)) f.gate_up = on_pairs;
  } else {
    const double dev = mean > 0 ? sqrt(mean * (1.0 - (mean < rows_s ? mean / rows_s : 1.0))) : 0.0;
    const double dev_s = s.n_outer > 1 ? sqrt((double)rows_s) : 0.0;
    const int w_s = P->has_s ? (s.shared_width + 127) / 128 : 0, w_r = P->has_r ? (s.m + 127) / 128 : 0;
    const double dram = (s.n_outer * w_s + n_routed * w_r) * 32768.0 / 5800.0;
    auto cost = [&](GemmForm form) {
      const int rows = form == GemmForm::kSingle ? kUmmaBM : 256;            // of a full tile
      auto tile = [&](double r) {                      // a tile of a group with r rows
        if (form != GemmForm::kTurned) return form == GemmForm::kSingle ? 425.0 : 350.0;
        const double t = 120.0 + 0.95 * TokenCut((int)ceil(r)).width;
        return t > 240.0 ? t : 240.0;
      };
      const bool turn = form == GemmForm::kTurned;
      const int per_s = turn || !P->has_s ? w_s : (s.shared_width + P->bn_s - 1) / P->bn_s;
      const int per_r = turn || !P->has_r ? w_r : (s.m + P->bn_r - 1) / P->bn_r;
      const int n_s = (int)(s.n_outer * umma_expected_tiles(rows_s, dev_s, rows) * per_s + 0.5);
      const double n_r = n_routed * umma_expected_tiles(mean, dev, rows) * per_r, c_s = tile(rows_s + dev_s / 2), c_r = tile(mean + dev / 2);
      double sum = 0.0;
      for (int skewed = 0; skewed < 2; ++skewed) {
        const double b = umma_busiest(n_s, c_s, (int)((skewed ? 1.2 : 1.0) * n_r + 0.5), c_r,
                                      form == GemmForm::kSingle ? P->n_sms : pair_grid / 2);
        sum += (b > dram ? b : dram) * (skewed ? 1.0 : 2.0) / 3.0;
      }
      return sum;
    };
    double best = cost(GemmForm::kSingle);
    for (GemmForm form : {GemmForm::kTurned, GemmForm::kPair}) {
      const double c = 1.09 * cost(form);
      if (c < best) { best = c; f.gate_up = form; }
    }
  }
  if (s.m > 448 && (mean > kUmmaBM || !P->has_r)) {
    // K x token columns, padded
    const double down_pair = (double)s.n_outer * s.shared_width * up(rows_s, 256) + (double)n_routed * s.m * up(rows_r, 256);
    const double down_turned = (double)s.n_outer * s.shared_width * umma2t_columns(rows_s) + (double)n_routed * s.m * umma2t_columns(rows_r);
    f.down = R >= kPairLargeRows && down_turned >= 0.97 * down_pair ? GemmForm::kPair : GemmForm::kTurned;
  }
  return f;
}

}  // namespace cmoe
