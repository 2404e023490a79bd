// Analytical router (Eq. router) and gate logic (Eq. final_gate); top-level
// router of a hierarchical layer (Section 4.4).  One warp owns two rows; the
// N_r <= 32 routed experts of a row live one per lane for the softmax and the
// warp-shuffle top-k.
#pragma once

#include "common.cuh"

namespace cmoe {

// Index of the outer expert whose row range [off[g], off[g+1]) holds row r.
__device__ __forceinline__ int find_outer(const int32_t* __restrict__ off, int n_outer, int r) {
  int g = 0;
#pragma unroll 4
  for (int i = 1; i < n_outer; ++i) g += (__ldcg(off + i) <= r) ? 1 : 0;
  return g;
}

// Warp-wide arg-max over (key, index): the larger key wins, equal keys go to the
// lower index.  Lanes that do not take part pass index >= 64.
__device__ __forceinline__ void warp_argmax(float& key, int& idx) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const float k2 = __shfl_xor_sync(0xffffffffu, key, o);
    const int i2 = __shfl_xor_sync(0xffffffffu, idx, o);
    if (k2 > key || (k2 == key && i2 < idx)) { key = k2; idx = i2; }
  }
}

// Gate logic for one row held across a warp: lane j < n_r carries the gate and up
// pre-activations (a, v) of routed expert j's representative neuron.
__device__ __forceinline__ void gate_row(int lane, int n_r, int n_k, float a, float v,
                                         const float* __restrict__ u, const float* __restrict__ b,
                                         int group_base, float* __restrict__ scores_row,
                                         float* __restrict__ keys_row, int32_t* __restrict__ idx_row,
                                         float* __restrict__ gates_row) {
  const bool live = lane < n_r;
  const float s = live ? silu_accurate(a) * v : -INFINITY;            // Eq. router
  const float s_max = warp_max(s);
  const float e = live ? expf(s - s_max) : 0.0f;
  const float s_prime = e / warp_sum(e);                               // Softmax over all N_r
  const float key = live ? s_prime + __ldcg(b + lane) : -INFINITY;
  if (live) { scores_row[lane] = s; keys_row[lane] = key; }
  const float gate = live ? 1.0f + s_prime * __ldcg(u + lane) : 0.0f;   // 1 + s'_i u_i
  const float rank_key = (key != key) ? -INFINITY : key;               // NaN ranks last
  bool taken = !live;
  for (int i = 0; i < n_k; ++i) {
    float best = taken ? -INFINITY : rank_key;
    int who = taken ? 64 + lane : lane;
    warp_argmax(best, who);
    const float g = __shfl_sync(0xffffffffu, gate, who & 31);
    if (lane == who) taken = true;
    if (lane == 0) { idx_row[i] = group_base + who; gates_row[i] = g; }
  }
}

// A float's bits mapped so that unsigned order is numeric order (-0 counts as +0).
__device__ __forceinline__ uint32_t ordered_bits(float v) {
  const uint32_t b = __float_as_uint(v + 0.0f);
  return (b & 0x80000000u) ? ~b : (b | 0x80000000u);
}

// gate_row for U rows at once, step by step so that the rows' chains of reductions overlap, with u and b already in
// registers and the arg-max by one warp-wide integer reduction and a ballot (the same order: larger key first, equal keys by
// index).  Lane i < n_k returns its selections in `sel`; rows that are not live are not stored.
template <int U>
__device__ __forceinline__ void gate_rows_redux(int lane, int n_r, int n_k, const float (&a)[U], const float (&v)[U], float u,
                                                float b, int group_base, const size_t (&row)[U], const bool (&row_live)[U],
                                                float* __restrict__ scores, float* __restrict__ keys,
                                                int32_t* __restrict__ idx, float* __restrict__ gates, int (&sel)[U]) {
  const bool live = lane < n_r;
  float s[U], m[U], e[U], sum[U], gate[U], my_gate[U];
  uint32_t bits[U];
#pragma unroll
  for (int q = 0; q < U; ++q) { s[q] = live ? silu_accurate(a[q]) * v[q] : -INFINITY; m[q] = s[q]; }   // Eq. router
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < U; ++q) m[q] = fmaxf(m[q], __shfl_xor_sync(0xffffffffu, m[q], o));
#pragma unroll
  for (int q = 0; q < U; ++q) { e[q] = live ? expf(s[q] - m[q]) : 0.0f; sum[q] = e[q]; }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int q = 0; q < U; ++q) sum[q] += __shfl_xor_sync(0xffffffffu, sum[q], o);
#pragma unroll
  for (int q = 0; q < U; ++q) {
    const float s_prime = e[q] / sum[q];                               // Softmax over all N_r
    const float key = live ? s_prime + b : -INFINITY;
    if (live && row_live[q]) { scores[row[q] * n_r + lane] = s[q]; keys[row[q] * n_r + lane] = key; }
    gate[q] = 1.0f + s_prime * u;                                      // 1 + s'_i u_i
    bits[q] = live ? ordered_bits((key != key) ? -INFINITY : key) : 0u;  // NaN ranks last; every live key is above 0
    my_gate[q] = 0.0f;
  }
#pragma unroll 1
  for (int i = 0; i < n_k; ++i) {
    uint32_t best[U];
    int who[U];
#pragma unroll
    for (int q = 0; q < U; ++q) best[q] = __reduce_max_sync(0xffffffffu, bits[q]);
#pragma unroll
    for (int q = 0; q < U; ++q) who[q] = __ffs(__ballot_sync(0xffffffffu, bits[q] == best[q])) - 1;
#pragma unroll
    for (int q = 0; q < U; ++q) {
      const float g = __shfl_sync(0xffffffffu, gate[q], who[q]);
      if (lane == who[q]) bits[q] = 0u;
      if (lane == i) { sel[q] = group_base + who[q]; my_gate[q] = g; }
    }
  }
  if (lane < n_k)
#pragma unroll
    for (int q = 0; q < U; ++q)
      if (row_live[q]) { idx[row[q] * n_k + lane] = sel[q]; gates[row[q] * n_k + lane] = my_gate[q]; }
}
__device__ __forceinline__ void gate_row_redux(int lane, int n_r, int n_k, float a, float v, float u, float b, int group_base,
                                               size_t row, float* __restrict__ scores, float* __restrict__ keys,
                                               int32_t* __restrict__ idx, float* __restrict__ gates, int& sel) {
  const float a1[1] = {a}, v1[1] = {v};
  const size_t r1[1] = {row};
  const bool l1[1] = {true};
  int s1[1] = {0};
  gate_rows_redux<1>(lane, n_r, n_k, a1, v1, u, b, group_base, r1, l1, scores, keys, idx, gates, s1);
  sel = s1[0];
}

// Top-level selection of one row (the outer_k largest logits, ties to the lower index; weights = softmax over the
// selected logits) by the same reduction: lane j < n_outer carries logit j.  Lane i < outer_k returns its selection.
__device__ __forceinline__ void outer_row_redux(int lane, int n_outer, int outer_k, float logit, float* __restrict__ logits_row,
                                                int32_t* __restrict__ idx_row, float* __restrict__ weight_row, int& sel) {
  const bool live = lane < n_outer;
  if (live) logits_row[lane] = logit;
  uint32_t bits = live ? ordered_bits((logit != logit) ? -INFINITY : logit) : 0u;
  float sel_logit = -INFINITY;
#pragma unroll 1
  for (int i = 0; i < outer_k; ++i) {
    const uint32_t best = __reduce_max_sync(0xffffffffu, bits);
    const int who = __ffs(__ballot_sync(0xffffffffu, bits == best)) - 1;
    const float l = __shfl_sync(0xffffffffu, logit, who);
    if (lane == who) bits = 0u;
    if (lane == i) { sel = who; sel_logit = l; }
  }
  const float mx = warp_max(lane < outer_k ? sel_logit : -INFINITY);
  const float e = lane < outer_k ? expf(sel_logit - mx) : 0.0f;
  const float weight = e / warp_sum(e);
  if (lane < outer_k) { idx_row[lane] = sel; weight_row[lane] = weight; }
}

// One row per warp, for batches that leave SMs idle otherwise (bound by latency).  The column sums meet by a reduce-scatter over the lanes (each step halves
// the columns a lane still carries): the pairs of lanes are those of warp_sum, so every sum has the same bits.
template <typename T, int NACC>
__global__ void __launch_bounds__(128)
router_row_kernel(const T* __restrict__ xo, int n_rows, int d, int n_r, int n_rp, int n_k,
                  const T* __restrict__ w_rep, const float* __restrict__ u, const float* __restrict__ b,
                  const int32_t* __restrict__ outer_off, int n_outer,
                  float* __restrict__ scores, float* __restrict__ keys,
                  int32_t* __restrict__ topk_idx, float* __restrict__ topk_gate) {
  grid_dep_wait();
  grid_dep_trigger();
  const int lane = threadIdx.x & 31;
  const int row = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (row >= n_rows) return;
  const int go = outer_off ? find_outer(outer_off, n_outer, row) : 0;
  const int n2 = 2 * n_rp;
  const T* xr = xo + (size_t)row * d;
  const T* w = w_rep + (size_t)go * n2 * d;
  const float u_pre = lane < n_r ? __ldcg(u + go * n_r + lane) : 0.0f, b_pre = lane < n_r ? __ldcg(b + go * n_r + lane) : 0.0f;
  float acc[NACC];
#pragma unroll
  for (int j = 0; j < NACC; ++j) acc[j] = 0.0f;
#pragma unroll 1
  for (int k = lane * 8; k < d; k += 256) {
    float xa[8];
    load8(xr + k, xa);
#pragma unroll
    for (int j = 0; j < NACC; ++j)
      if (j < n2) {
        float wa[8];
        load8(w + (size_t)j * d + k, wa);
#pragma unroll
        for (int q = 0; q < 8; ++q) acc[j] = fmaf(wa[q], xa[q], acc[j]);
      }
  }
  // after the steps with a column to give away, lane l carries column l * NACC / 32 (NACC = 64: two columns, j and j + 32)
  constexpr int kSets = NACC > 32 ? NACC / 32 : 1, kCols = NACC / kSets;
  float col[kSets];
#pragma unroll
  for (int s = 0; s < kSets; ++s) {
    float* v = acc + s * kCols;
    int n = kCols;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      if (n > 1) {
        n >>= 1;
        const bool up = lane & o;
#pragma unroll
        for (int j = 0; j < kCols / 2; ++j)
          if (j < n) {
            const float give = up ? v[j] : v[j + n], keep = up ? v[j + n] : v[j];
            v[j] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
      } else {
        v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
      }
    }
    col[s] = v[0];
  }
  constexpr int kPer = 32 / kCols;                // lanes that carry the same column
  const int cv = n_rp + lane;                     // column of expert `lane`'s up sum
  const float a = __shfl_sync(0xffffffffu, col[0], (lane * kPer) & 31);
  float v = __shfl_sync(0xffffffffu, col[0], (cv * kPer) & 31);
  if (kSets > 1) {
    const float v1 = __shfl_sync(0xffffffffu, col[kSets - 1], cv & 31);
    if (cv >= 32) v = v1;
  }
  int sel = 0;
  gate_row_redux(lane, n_r, n_k, a, v, u_pre, b_pre, go * n_r, (size_t)row, scores, keys, topk_idx, topk_gate, sel);
}

template <typename T, int NACC>
__global__ void __launch_bounds__(256)
router_kernel(const T* __restrict__ xo, int n_rows, int d, int n_r, int n_rp, int n_k,
              const T* __restrict__ w_rep, const float* __restrict__ u, const float* __restrict__ b,
              const int32_t* __restrict__ outer_off, int n_outer,
              float* __restrict__ scores, float* __restrict__ keys,
              int32_t* __restrict__ topk_idx, float* __restrict__ topk_gate) {
  grid_dep_wait();
  grid_dep_trigger();
  const int lane = threadIdx.x & 31;
  const int warp = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const int r0 = warp * 2;
  if (r0 >= n_rows) return;
  const bool has1 = r0 + 1 < n_rows;
  const int r1 = has1 ? r0 + 1 : r0;
  const int g0 = outer_off ? find_outer(outer_off, n_outer, r0) : 0;
  const int g1 = outer_off ? find_outer(outer_off, n_outer, r1) : 0;
  const int n2 = 2 * n_rp;      // W^R block: n_rp gate rows (zero-padded), then n_rp up rows
  const T* x0 = xo + (size_t)r0 * d;
  const T* x1 = xo + (size_t)r1 * d;
  const T* w0 = w_rep + (size_t)g0 * n2 * d;
  const T* w1 = w_rep + (size_t)g1 * n2 * d;
  const bool same = g0 == g1;

  float acc0[NACC], acc1[NACC];
#pragma unroll
  for (int j = 0; j < NACC; ++j) { acc0[j] = 0.0f; acc1[j] = 0.0f; }

  for (int k = lane * 8; k < d; k += 256) {
    float xa[8], xb[8];
    load8(x0 + k, xa);
    load8(x1 + k, xb);
#pragma unroll
    for (int j = 0; j < NACC; ++j) {
      if (j < n2) {
        float wa[8];
        load8(w0 + (size_t)j * d + k, wa);
        float t0 = acc0[j];
#pragma unroll
        for (int q = 0; q < 8; ++q) t0 = fmaf(wa[q], xa[q], t0);
        acc0[j] = t0;
        if (!same) load8(w1 + (size_t)j * d + k, wa);
        float t1 = acc1[j];
#pragma unroll
        for (int q = 0; q < 8; ++q) t1 = fmaf(wa[q], xb[q], t1);
        acc1[j] = t1;
      }
    }
  }

  float a0 = 0.f, v0 = 0.f, a1 = 0.f, v1 = 0.f;
#pragma unroll
  for (int j = 0; j < NACC; ++j) {
    if (j < n2) {
      const float t0 = warp_sum(acc0[j]);
      const float t1 = warp_sum(acc1[j]);
      if (lane == j) { a0 = t0; a1 = t1; }
      if (lane == j - n_rp) { v0 = t0; v1 = t1; }
    }
  }
  gate_row(lane, n_r, n_k, a0, v0, u + g0 * n_r, b + g0 * n_r, g0 * n_r,
           scores + (size_t)r0 * n_r, keys + (size_t)r0 * n_r,
           topk_idx + (size_t)r0 * n_k, topk_gate + (size_t)r0 * n_k);
  if (has1)
    gate_row(lane, n_r, n_k, a1, v1, u + g1 * n_r, b + g1 * n_r, g1 * n_r,
             scores + (size_t)r1 * n_r, keys + (size_t)r1 * n_r,
             topk_idx + (size_t)r1 * n_k, topk_gate + (size_t)r1 * n_k);
}

// Top-level router of an existing MoE layer: logits = W_r x, the outer_k largest
// logits (ties: lower index), weights = softmax over the selected logits.
template <typename T>
__global__ void __launch_bounds__(256)
outer_router_kernel(const T* __restrict__ x, int n_tokens, int d, int n_outer, int outer_k,
                    const T* __restrict__ w_router, float* __restrict__ logits,
                    int32_t* __restrict__ outer_idx, float* __restrict__ outer_w) {
  const int lane = threadIdx.x & 31;
  const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (t >= n_tokens) return;
  float acc[kMaxOuter];
#pragma unroll
  for (int j = 0; j < kMaxOuter; ++j) acc[j] = 0.0f;
  const T* xr = x + (size_t)t * d;
  for (int k = lane * 8; k < d; k += 256) {
    float xa[8];
    load8(xr + k, xa);
#pragma unroll
    for (int j = 0; j < kMaxOuter; ++j) {
      if (j < n_outer) {
        float wa[8];
        load8(w_router + (size_t)j * d + k, wa);
        float s = acc[j];
#pragma unroll
        for (int q = 0; q < 8; ++q) s = fmaf(wa[q], xa[q], s);
        acc[j] = s;
      }
    }
  }
  float logit = -INFINITY;
#pragma unroll
  for (int j = 0; j < kMaxOuter; ++j) {
    if (j < n_outer) {
      const float s = warp_sum(acc[j]);
      if (lane == j) logit = s;
    }
  }
  const bool live = lane < n_outer;
  if (live) logits[(size_t)t * n_outer + lane] = logit;
  const float rank_key = (logit != logit) ? -INFINITY : logit;
  bool taken = !live;
  float sel_logit = -INFINITY;   // lane i < outer_k keeps the i-th selected logit
  int sel_who = 0;
  for (int i = 0; i < outer_k; ++i) {
    float best = taken ? -INFINITY : rank_key;
    int who = taken ? 64 + lane : lane;
    warp_argmax(best, who);
    const float l = __shfl_sync(0xffffffffu, logit, who & 31);
    if (lane == who) taken = true;
    if (lane == i) { sel_logit = l; sel_who = who; }
  }
  const float mx = warp_max(lane < outer_k ? sel_logit : -INFINITY);
  const float e = lane < outer_k ? expf(sel_logit - mx) : 0.0f;
  const float w = e / warp_sum(e);
  if (lane < outer_k) {
    outer_idx[(size_t)t * outer_k + lane] = sel_who;
    outer_w[(size_t)t * outer_k + lane] = w;
  }
}

}  // namespace cmoe
