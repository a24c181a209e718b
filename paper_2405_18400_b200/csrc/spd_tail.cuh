// Pieces of the method's tail that both kernels of the library run: per-block top-k of the logits with
// softmax statistics, KeepTopK over the blocks' partial lists (Algorithm 1), the first timestep's
// assignment (Eq. 1) and the drafts' weights (Eq. 4).  Each runs on one warp.
#pragma once
#include <cuda_runtime.h>
#include <math_constants.h>

#include "spd_params.h"

namespace spd {

// ---------------------------------------------------------------- LM head: block-level top-k and softmax statistics
// Ranking order everywhere: larger value first, then smaller index.
__device__ __forceinline__ bool ranks_before(float v, int i, float w, int j) { return v > w || (v == w && i < j); }

// Floats as words of the same order; 0 is below all of them, NaN the next, -0 and +0 are one value.
__device__ __forceinline__ uint32_t order_key(float v) {
  const uint32_t u = __float_as_uint(v + 0.f);
  return v != v ? 1u : ((u & 0x80000000u) ? ~u : (u | 0x80000000u));
}
__device__ __forceinline__ float order_value(uint32_t key) { return __uint_as_float((key & 0x80000000u) ? (key & 0x7fffffffu) : ~key); }

// The warp's best candidate (i < 0: a lane without one), to all lanes.  Two reductions of words: with five rounds of two shuffles and
// the comparison a call took 0.2 us, and a timestep's tail makes 3 k of them while all blocks wait.
__device__ __forceinline__ void warp_best(float &v, int &i) {
  const uint32_t mine = i >= 0 ? order_key(v) : 0u, best = __reduce_max_sync(0xffffffffu, mine);
  i = (int)__reduce_min_sync(0xffffffffu, mine == best && i >= 0 ? (uint32_t)i : 0xffffffffu);
  if (best) v = order_value(best);
}

// One warp: the k best logits among rows [r0, r1) and (max, sum exp) of z / tau over them, into list `slot` of the
// partial lists (the decode and prefill kernels: warp 0 of each block, slot = the block), best first.  A lane asks for eight
// rows at a time, and keeps them for all rounds when that is all there is (up to 256 rows: a block's share of the LM head).
// A NaN ranks as -inf does (fmaxf passes over it): compared as it is, one in a lane's first row would hide the lane's other rows.
constexpr int kTopkFlight = 8;
static __device__ void block_topk(const KParams &p, int r0, int r1, int slot) {
  const int lane = threadIdx.x & 31;
  const bool once = r1 - r0 <= 32 * kTopkFlight;
  float z[kTopkFlight];
  auto fetch = [&](int r) {
#pragma unroll
    for (int e = 0; e < kTopkFlight; ++e) z[e] = r + 32 * e < r1 ? p.logits[r + 32 * e] : 0.f;
  };
  fetch(r0 + lane);
  float pv = 0.f;
  int pi = -1;
  uint32_t taken = 0u;  // of the lane's rows in registers
  float mx = -CUDART_INF_F;
  for (int j = 0; j < p.k; ++j) {
    float bv = 0.f;
    int bi = -1;
    if (once) {
#pragma unroll
      for (int e = 0; e < kTopkFlight; ++e) {
        const int id = r0 + lane + 32 * e;
        const float v = fmaxf(z[e], -CUDART_INF_F);
        if (id < r1 && !(taken >> e & 1u) && (bi < 0 || v > bv)) { bv = v; bi = id; }
      }
    } else {
      for (int r = r0 + lane; r < r1; r += 32 * kTopkFlight) {
        fetch(r);
#pragma unroll
        for (int e = 0; e < kTopkFlight; ++e) {
          const int id = r + 32 * e;
          const float v = fmaxf(z[e], -CUDART_INF_F);
          // (rows already taken, the previous winner among them, are passed over)
          if (id < r1 && (j == 0 || ranks_before(pv, pi, v, id)) && (bi < 0 || ranks_before(v, id, bv, bi))) { bv = v; bi = id; }
        }
      }
    }
    warp_best(bv, bi);
    if (once && bi >= 0 && ((bi - r0) & 31) == lane) taken |= 1u << ((bi - r0) >> 5);
    if (lane == 0) {
      p.pk_val[(size_t)slot * p.k + j] = bi >= 0 ? bv : -CUDART_INF_F;
      p.pk_id[(size_t)slot * p.k + j] = bi;
    }
    pv = bv;
    pi = bi;
    if (j == 0) mx = bi >= 0 ? bv * p.inv_tau : -CUDART_INF_F;
    if (bi < 0) {  // fewer rows than k: the rest stay empty
      for (int jj = j + 1; jj < p.k; ++jj)
        if (lane == 0) {
          p.pk_val[(size_t)slot * p.k + jj] = -CUDART_INF_F;
          p.pk_id[(size_t)slot * p.k + jj] = -1;
        }
      break;
    }
  }
  float s = 0.f;
  for (int r = r0 + lane; r < r1; r += 32 * kTopkFlight) {
    if (!once) fetch(r);
#pragma unroll
    for (int e = 0; e < kTopkFlight; ++e)
      if (r + 32 * e < r1) s += __expf(z[e] * p.inv_tau - mx);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) p.pk_ms[slot] = make_float2(mx, s);
}

// KeepTopK over the whole vocabulary from the n_lists (<= kMaxLists) partial lists (Algorithm 1), with log-probabilities
// under temperature tau.  Warp 0.  The lists are in rank order, so a lane keeps the heads of its lists in registers and a
// round is a vote over the heads and one load, of the winning list's next entry: the warp stands alone between two grid
// barriers here, and a trip to L2 per candidate and round (148 lists: 14 of them for k = 3, 37 for k = 8) was most of a
// timestep's tail (with the other two places where loads stood in a row, block_topk and the input's embedding: tiny model, 150 steps
// in one launch, 11.4 -> 8.6 ms; 7B shape, k = 8, 2.76 -> 2.64 ms per timestep).
static __device__ void tail_keep_topk(const KParams &p, int n_lists) {
  const int lane = threadIdx.x & 31;
  constexpr int kMine = kMaxLists / 32;
  State *st = p.st;
  float2 ms[kMine];
  float hv[kMine];
  int hid[kMine], next[kMine];
#pragma unroll
  for (int i = 0; i < kMine; ++i) {
    const int g = lane + 32 * i;
    const bool in = g < n_lists;
    ms[i] = in ? __ldcg(&p.pk_ms[g]) : make_float2(-CUDART_INF_F, 0.f);
    hv[i] = in ? __ldcg(&p.pk_val[(size_t)g * p.k]) : 0.f;
    hid[i] = in ? __ldcg(&p.pk_id[(size_t)g * p.k]) : -1;
    next[i] = 1;
  }
  float M = -CUDART_INF_F;
#pragma unroll
  for (int i = 0; i < kMine; ++i) M = fmaxf(M, ms[i].x);
  M = order_value(__reduce_max_sync(0xffffffffu, order_key(M)));
  float S = 0.f;
#pragma unroll
  for (int i = 0; i < kMine; ++i)
    if (lane + 32 * i < n_lists && ms[i].x > -CUDART_INF_F) S = fmaf(ms[i].y, __expf(ms[i].x - M), S);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) S += __shfl_xor_sync(0xffffffffu, S, o);
  const float lse = M + __logf(S);
  for (int j = 0; j < p.k; ++j) {
    float bv = 0.f;
    int bi = -1;
#pragma unroll
    for (int i = 0; i < kMine; ++i)
      if (hid[i] >= 0 && (bi < 0 || ranks_before(hv[i], hid[i], bv, bi))) { bv = hv[i]; bi = hid[i]; }
    warp_best(bv, bi);
    if (lane == 0) {
      // non-finite logits can leave a round without a winner: keep the token id valid
      st->cand_tok[j] = bi < 0 ? 0 : bi;
      st->cand_lp[j] = bv * p.inv_tau - lse;
    }
#pragma unroll
    for (int i = 0; i < kMine; ++i)
      if (bi >= 0 && hid[i] == bi) {  // this list's head was taken (an id is in one list only)
        const size_t at = (size_t)(lane + 32 * i) * p.k + next[i];
        const bool more = next[i] < p.k;
        hid[i] = more ? __ldcg(&p.pk_id[at]) : -1;
        hv[i] = more ? __ldcg(&p.pk_val[at]) : 0.f;
        ++next[i];
      }
  }
  __syncwarp();
}

// gamma_i = p_i / sum_j p_j (Eq. 4), from the drafts' log-probabilities; the step is then complete: the
// history windows have grown by one token.  One warp.
__device__ __forceinline__ void tail_gamma(const KParams &p, int lane) {
  State *st = p.st;
  const int k = p.k;
  const float lp = lane < k ? st->logP[lane] : -CUDART_INF_F;
  float mx = lp;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  const float e = lane < k ? expf(lp - mx) : 0.f;
  float den = e;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) den += __shfl_xor_sync(0xffffffffu, den, o);
  if (lane < k) st->gamma[lane] = e / den;
  if (lane == 0) {
    st->win_len = min(st->win_len + 1, kWin);
    st->n_gen += 1;
  }
}

// First timestep (Eq. 1): draft i takes the i-th kept token and its log-probability; no n-gram term.  Thread
// i < k of one warp.
__device__ __forceinline__ void tail_first(const KParams &p, int i, int step) {
  State *st = p.st;
  const int k = p.k;
  if (i < k) {
    const int tok = st->cand_tok[i];
    st->logP_in[i] = 0.f;
    int w[kWin];
#pragma unroll
    for (int j = 0; j < kWin; ++j) w[j] = st->win[i][j];
#pragma unroll
    for (int j = 0; j < kWin; ++j) st->win_in[i][j] = w[j];
#pragma unroll
    for (int j = 0; j + 1 < kWin; ++j) st->win[i][j] = w[j + 1];
    st->win[i][kWin - 1] = tok;
    st->logP[i] = st->cand_lp[i];
    st->sel[i] = i;
    p.hist_tok[(size_t)step * k + i] = tok;
    p.hist_par[(size_t)step * k + i] = i;
  }
}

}  // namespace spd
