// Nucleus sampling over the LM-head output (Section 2: the smallest set of most probable tokens whose
// probability mass reaches p; one token is drawn from it in proportion to its probability), for splicing
// Superposed Decoding onto nucleus-sampled prefixes (Section 4.5).  Runs on one block, all consumer threads.
//
// Tokens are ordered by logit, descending, equal logits by ascending id.  With e_i = exp(z_i / T - max) the
// nucleus is the shortest head of that order whose sum reaches p * sum_i e_i, and the draw u in [0, 1) picks
// the first token whose running sum exceeds u * (mass of the nucleus).  All sums are taken in 64-bit fixed
// point (e_i * 2^40, rounded down), so they are exact, independent of the order of summation, and every
// comparison is an integer comparison.  A nucleus of few tokens close to the best (ns_near) takes one pass over the logits.  Else both
// thresholds are located by a radix search over the logits' order-preserving 32-bit keys: six passes (6,6,6,6,6,2 bits), each a
// histogram of mass and count per digit among the logits that share the digits fixed so far, scanned from the top digit down.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "spd_params.h"
#include "spd_ptx.cuh"

namespace spd {

constexpr int kNsBins = 64;
constexpr int kNsBatch = 8;  // logits a thread loads before it looks at them

struct NsShared {
  // per warp and digit: mass as two 20-bit halves (32-bit shared-memory atomics are native, 64-bit ones are
  // not; a warp adds at most 2016 values below 2^20 to a cell) and count
  unsigned int hi[kConsumerWarps][kNsBins], lo[kConsumerWarps][kNsBins];
  unsigned int cnts[kConsumerWarps][kNsBins];
  unsigned long long park[3];   // values carried from the first search to the second
  unsigned long long tot[kNsBins];
  unsigned int ctot[kNsBins];
  // search state and results (thread 0 writes, everyone reads after a barrier)
  unsigned long long above;     // mass of the logits above the digits fixed so far
  unsigned long long total;     // mass of all logits
  unsigned long long target;    // the running sum to reach
  unsigned long long tie_mass;  // mass of the logits equal to the located one
  unsigned int tie_cnt;
  unsigned int prefix;          // digits fixed so far
  float zmax;
  int warp_cnt[kConsumerWarps];
  int token;
};
static_assert(sizeof(NsShared) <= 20480, "nucleus scratch must fit the block's scratch area");

__device__ __forceinline__ uint32_t ns_key(float z) {
  const uint32_t u = __float_as_uint(z + 0.f);  // -0 and +0 are one value
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
// e = exp(z / T - max) in 2^-40 units, rounded down, as two 20-bit halves (e * 2^20 and the remainder * 2^20 are
// exact in float32, so the halves are exact)
__device__ __forceinline__ void ns_mass(float z, float inv_t, float m, unsigned int &hi, unsigned int &lo) {
  const float e20 = __expf(fmaf(z, inv_t, -m)) * 1048576.f;
  const float fh = floorf(e20);
  hi = (unsigned int)fh;
  lo = (unsigned int)((e20 - fh) * 1048576.f);
}

// Locates the first token (in the order above) whose running sum reaches s.target (>= 1): leaves its key in
// s.prefix, the mass above it in s.above, and mass and count of the logits equal to it in s.tie_*.  With
// `fraction` > 0 the target is first set to ceil(fraction * total mass).  If rounding left the target above
// the total, the last token is located.
static __device__ void ns_search(NsShared &s, const float *logits, int V, float inv_t, float m, float fraction) {
  const int tid = threadIdx.x, warp = tid >> 5;
  int decided = 0;
  for (int pass = 0; pass < 6; ++pass) {
    const int width = pass < 5 ? 6 : 2, shift = 32 - decided - width;
    for (int i = tid; i < kConsumerWarps * kNsBins; i += kConsumerThreads) {
      (&s.hi[0][0])[i] = 0u;
      (&s.lo[0][0])[i] = 0u;
      (&s.cnts[0][0])[i] = 0u;
    }
    named_sync(1, kConsumerThreads);
    const uint32_t prefix = s.prefix;
    int cur = -1;  // a run of logits with one digit is summed in registers: at most 63 values of at most 2^20
    unsigned int cur_hi = 0u, cur_lo = 0u, cur_c = 0u;
    for (int r0 = tid; r0 < V; r0 += kNsBatch * kConsumerThreads) {
      float zb[kNsBatch];  // a batch of loads in flight: the logits come from L2
#pragma unroll
      for (int e = 0; e < kNsBatch; ++e) {
        const int r = r0 + e * kConsumerThreads;
        zb[e] = r < V ? __ldcg(logits + r) : 0.f;
      }
#pragma unroll
      for (int e = 0; e < kNsBatch; ++e) {
        if (r0 + e * kConsumerThreads >= V) break;
        const float z = zb[e];
        const uint32_t key = ns_key(z);
        if (decided == 0 || (key >> (32 - decided)) == prefix) {
          const int d = (int)((key >> shift) & ((1u << width) - 1u));
          if (d != cur) {
            if (cur >= 0) {
              atomicAdd(&s.hi[warp][cur], cur_hi + (cur_lo >> 20));
              atomicAdd(&s.lo[warp][cur], cur_lo & 0xfffffu);
              atomicAdd(&s.cnts[warp][cur], cur_c);
            }
            cur = d;
            cur_hi = cur_lo = cur_c = 0u;
          }
          unsigned int h, l;
          ns_mass(z, inv_t, m, h, l);
          cur_hi += h;
          cur_lo += l;
          cur_c += 1u;
        }
      }
    }
    if (cur >= 0) {
      atomicAdd(&s.hi[warp][cur], cur_hi + (cur_lo >> 20));
      atomicAdd(&s.lo[warp][cur], cur_lo & 0xfffffu);
      atomicAdd(&s.cnts[warp][cur], cur_c);
    }
    named_sync(1, kConsumerThreads);
    if (tid < kNsBins) {
      unsigned long long q = 0ull;
      unsigned int c = 0u;
      for (int w = 0; w < kConsumerWarps; ++w) {
        q += ((unsigned long long)s.hi[w][tid] << 20) + s.lo[w][tid];
        c += s.cnts[w][tid];
      }
      s.tot[tid] = q;
      s.ctot[tid] = c;
    }
    named_sync(1, kConsumerThreads);
    if (tid == 0) {
      if (pass == 0) {
        unsigned long long all = 0ull;
        for (int d = 0; d < kNsBins; ++d) all += s.tot[d];
        s.total = all;
        if (fraction > 0.f) {
          unsigned long long t = __double2ull_ru((double)fraction * (double)all);
          s.target = t < 1ull ? 1ull : (t > all ? all : t);
        }
      }
      unsigned long long cum = s.above, last_tot = 0ull;
      int g = -1, last = -1;
      for (int d = (1 << width) - 1; d >= 0; --d) {
        if (s.ctot[d] == 0u) continue;
        if (cum + s.tot[d] >= s.target) {
          g = d;
          break;
        }
        cum += s.tot[d];
        last = d;
        last_tot = s.tot[d];
      }
      if (g < 0) {  // the target lies above the total: the last token in the order
        g = last < 0 ? 0 : last;
        cum -= last_tot;
      }
      s.above = cum;
      s.prefix = (decided == 0 ? 0u : (s.prefix << width)) | (uint32_t)g;
      s.tie_mass = s.tot[g];
      s.tie_cnt = s.ctot[g];
    }
    named_sync(1, kConsumerThreads);
    decided += width;
  }
}

// The draw when few tokens lie near the best.  Those at distances x = max - z / T below 8 are listed and fall into 32 bins a quarter
// wide (in the order of the logits, for the distance is one rounding of a monotone function); what lies further off only adds to the
// total.  When the list holds them all and the nucleus ends among them, the two tokens sought are found by the running sums of their
// own bin: the same sums of the same whole numbers as in the search.  False: not such a case (a flat distribution, a nucleus of
// hundreds of tokens, no mass at all), nothing decided; known as soon as the list is full.
// One pass over the logits instead of fourteen, with four trips to L2 in it: 10 tokens drawn from 32000 logits at temperature 0.2,
// 7B shape, 25.60 -> 24.17 ms, 0.143 ms a draw.
constexpr int kNearBins = 32, kNearList = kConsumerThreads, kNearFlight = 16;
struct NsNear {
  unsigned int hi[kNearBins], lo[kNearBins];
  unsigned long long tot[kNearBins], before[kNearBins];  // per bin: its mass, the mass of the bins before it
  unsigned long long ord[kNearList], mass[kNearList];    // per listed token: place in the order (larger first), mass
  unsigned char bin[kNearList];
  unsigned long long far[kConsumerWarps];                // mass behind the bins, per warp
  unsigned long long target, nucleus;
  int listed, cut_bin, hit_bin, token;
};
static_assert(sizeof(NsNear) <= 20480, "nucleus scratch must fit the block's scratch area");

static __device__ bool ns_near(NsNear &s, const float *logits, int V, float inv_t, float m, float top_p, float u, int &token) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < kNearBins) s.hi[tid] = s.lo[tid] = 0u;
  if (tid == 0) {
    s.listed = 0;
    s.cut_bin = s.hit_bin = -1;
    s.token = 0;
  }
  named_sync(1, kConsumerThreads);
  unsigned int far_hi = 0u, far_lo = 0u;  // at most 128 values (V is below 65536), halves below 2^20
  for (int base = 0; base < V; base += kNearFlight * kConsumerThreads) {
    // One lane looks whether the list is full and all follow it: other warps add to it meanwhile, and lanes that each looked for
    // themselves could part in front of the votes below, which wait for the whole warp.  (Warps may leave in different rounds.)
    int listed = 0;
    if (lane == 0) listed = *reinterpret_cast<volatile int *>(&s.listed);
    if (__shfl_sync(0xffffffffu, listed, 0) > kNearList) break;
    float zb[kNearFlight];
#pragma unroll
    for (int e = 0; e < kNearFlight; ++e) {
      const int r = base + e * kConsumerThreads + tid;
      zb[e] = r < V ? __ldcg(logits + r) : -CUDART_INF_F;
    }
    __syncwarp();
#pragma unroll
    for (int e = 0; e < kNearFlight; ++e) {
      const float x = -fmaf(zb[e], inv_t, -m);
      const bool near = x < 8.f;
      unsigned int h = 0u, l = 0u;
      if (x < 30.f) ns_mass(zb[e], inv_t, m, h, l);  // (e^-30 is below 2^-40: no mass)
      const unsigned int votes = __ballot_sync(0xffffffffu, near);
      if (votes) {
        int at = 0;
        if (lane == 0) at = atomicAdd(&s.listed, __popc(votes));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(votes & ((1u << lane) - 1u));
        if (near && at < kNearList) {
          const int b = max((int)(x * 4.f), 0);
          atomicAdd(&s.hi[b], h);  // at most kNearList values of 2^20 in all
          atomicAdd(&s.lo[b], l);
          s.ord[at] = (unsigned long long)ns_key(zb[e]) << 32 | (0xffffffffu - (unsigned int)(base + e * kConsumerThreads + tid));
          s.mass[at] = ((unsigned long long)h << 20) + l;
          s.bin[at] = (unsigned char)b;
        }
      }
      if (!near) {
        far_hi += h;
        far_lo += l;
      }
    }
  }
  unsigned long long far = ((unsigned long long)far_hi << 20) + far_lo;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) far += __shfl_xor_sync(0xffffffffu, far, o);
  if (lane == 0) s.far[warp] = far;
  named_sync(1, kConsumerThreads);
  if (tid == 0 && s.listed <= kNearList) {
    unsigned long long all = 0ull;
    for (int b = 0; b < kNearBins; ++b) {
      s.before[b] = all;
      all += s.tot[b] = ((unsigned long long)s.hi[b] << 20) + s.lo[b];
    }
    for (int w = 0; w < kConsumerWarps; ++w) all += s.far[w];
    unsigned long long t = __double2ull_ru((double)top_p * (double)all);
    t = t < 1ull ? 1ull : (t > all ? all : t);
    s.target = t;
    for (int b = 0; b < kNearBins && s.cut_bin < 0; ++b)
      if (all > 0ull && s.before[b] + s.tot[b] >= t) s.cut_bin = b;
  }
  named_sync(1, kConsumerThreads);
  if (s.cut_bin < 0) return false;
  const int n = s.listed;
  const bool mine = tid < n;
  const unsigned long long ord = mine ? s.ord[tid] : 0ull, mass = mine ? s.mass[tid] : 0ull;
  const int bin = mine ? s.bin[tid] : -1;
  // the running sum in front of the thread's token, for the tokens of one bin
  auto sum_before = [&]() {
    unsigned long long a = s.before[bin];
    for (int j = 0; j < n; ++j)
      if (s.bin[j] == bin && s.ord[j] > ord) a += s.mass[j];
    return a;
  };
  if (bin == s.cut_bin) {
    const unsigned long long a = sum_before();
    if (a < s.target && a + mass >= s.target) s.nucleus = a + mass;  // the nucleus' last token
  }
  named_sync(1, kConsumerThreads);
  const unsigned long long all = s.nucleus;
  unsigned long long t = __double2ull_rd((double)u * (double)all);
  if (t >= all) t = all - 1ull;
  if (tid < kNearBins && s.before[tid] <= t && t < s.before[tid] + s.tot[tid]) s.hit_bin = tid;
  named_sync(1, kConsumerThreads);
  if (mine && bin == s.hit_bin) {
    const unsigned long long a = sum_before();
    if (a <= t && t < a + mass) s.token = (int)(0xffffffffu - (unsigned int)ord);
  }
  named_sync(1, kConsumerThreads);
  token = s.token;
  named_sync(1, kConsumerThreads);
  return true;
}

// Draws one token from the nucleus of softmax(logits / T) with the uniform number u in [0, 1).  Every
// consumer thread of the block calls it; all get the token.
// heads: the largest logit of each of n_heads parts of the vocabulary, stride apart (null: looked for here).
static __device__ __noinline__ int ns_sample(const float *logits, int V, float inv_t, float top_p, float u, uint8_t *scratch, const float *heads,
                                             int n_heads, int stride) {
  NsShared &s = *reinterpret_cast<NsShared *>(scratch);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  named_sync(1, kConsumerThreads);
  // largest logit
  float zm = -3.402823466e38f, head = -CUDART_INF_F;
  if (heads) {
    if (tid < n_heads) head = __ldcg(heads + (size_t)tid * stride);
    zm = fmaxf(zm, head);
  } else {
    for (int r0 = tid; r0 < V; r0 += kNsBatch * kConsumerThreads) {
#pragma unroll
      for (int e = 0; e < kNsBatch; ++e) {
        const int r = r0 + e * kConsumerThreads;
        if (r < V) zm = fmaxf(zm, __ldcg(logits + r));
      }
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) zm = fmaxf(zm, __shfl_xor_sync(0xffffffffu, zm, o));
  float *wmax = reinterpret_cast<float *>(&s.tot[0]);
  if (lane == 0) wmax[warp] = zm;
  named_sync(1, kConsumerThreads);
  if (tid == 0) {
    float z = wmax[0];
    for (int w = 1; w < kConsumerWarps; ++w) z = fmaxf(z, wmax[w]);
    s.zmax = z;
    s.above = 0ull;
    s.prefix = 0u;
    s.target = 1ull;
  }
  named_sync(1, kConsumerThreads);
  const float m = s.zmax * inv_t;
  // Not tried when fifteen in sixteen of the parts' largest logits are that near: with 148 parts of 216 some 400 tokens are then (an
  // attempt in vain costs a draw 8 us).  Vocabularies of 2000, 32000 and 50000, temperatures 0.05 to 2: 0.33 to 0.98 of the time of a
  // search with its own pass for the maximum, at the flat end 0.92 to 0.98.
  const unsigned int near_votes = __ballot_sync(0xffffffffu, -fmaf(head, inv_t, -m) < 8.f);
  if (lane == 0) s.warp_cnt[warp] = __popc(near_votes);
  named_sync(1, kConsumerThreads);
  int heads_near = 0;
  for (int w = 0; w < kConsumerWarps; ++w) heads_near += s.warp_cnt[w];
  if (16 * heads_near <= 15 * n_heads) {
    named_sync(1, kConsumerThreads);  // (maximum and counts have been read: the scratch is laid out anew)
    int token;
    if (ns_near(*reinterpret_cast<NsNear *>(scratch), logits, V, inv_t, m, top_p, u, token)) return token;
    named_sync(1, kConsumerThreads);
    if (tid == 0) {
      s.above = 0ull;
      s.prefix = 0u;
      s.target = 1ull;
    }
    named_sync(1, kConsumerThreads);
  }
  // where the nucleus ends
  ns_search(s, logits, V, inv_t, m, top_p);
  if (tid == 0) {
    const uint32_t cut_key = s.prefix;
    const unsigned long long q = s.tie_cnt ? s.tie_mass / s.tie_cnt : 0ull;  // equal logits have equal mass
    unsigned long long take = s.tie_cnt;  // how many of the equal logits at the cut belong to the nucleus
    if (q > 0ull) {
      const unsigned long long need = s.target > s.above ? s.target - s.above : 1ull;
      take = (need + q - 1ull) / q;
      if (take > s.tie_cnt) take = s.tie_cnt;
      if (take < 1ull) take = 1ull;
    }
    const unsigned long long mass = s.above + take * q;
    unsigned long long t = mass ? __double2ull_rd((double)u * (double)mass) : 0ull;
    if (mass && t >= mass) t = mass - 1ull;
    // second search: first token whose running sum exceeds t
    s.park[0] = t;
    s.park[1] = take;
    s.park[2] = (unsigned long long)cut_key;
    s.above = 0ull;
    s.prefix = 0u;
    s.target = t + 1ull;
  }
  named_sync(1, kConsumerThreads);
  const unsigned long long t = s.park[0], take = s.park[1];
  const uint32_t cut_key = (uint32_t)s.park[2];
  ns_search(s, logits, V, inv_t, m, 0.f);
  // which of the logits equal to the located one: the j-th by ascending id
  const uint32_t hit_key = s.prefix;
  unsigned long long j = 0ull;
  {
    const unsigned long long q = s.tie_cnt ? s.tie_mass / s.tie_cnt : 0ull;
    if (q > 0ull && t >= s.above) j = (t - s.above) / q;
    if (j >= s.tie_cnt) j = s.tie_cnt ? s.tie_cnt - 1ull : 0ull;
    if (hit_key == cut_key && j >= take) j = take - 1ull;
  }
  const int seg = (V + kConsumerThreads - 1) / kConsumerThreads;
  const int lo = tid * seg, hi = min(V, lo + seg);
  int mine = 0;
  for (int r0 = lo; r0 < hi; r0 += kNsBatch) {
#pragma unroll
    for (int e = 0; e < kNsBatch; ++e)
      if (r0 + e < hi) mine += ns_key(__ldcg(logits + r0 + e)) == hit_key ? 1 : 0;
  }
  int incl = mine;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) s.warp_cnt[warp] = incl;
  if (tid == 0) s.token = 0;
  named_sync(1, kConsumerThreads);
  int before = incl - mine;
  for (int w = 0; w < warp; ++w) before += s.warp_cnt[w];
  if (mine > 0 && (unsigned long long)before <= j && j < (unsigned long long)(before + mine)) {
    int left = (int)(j - (unsigned long long)before);
    for (int r = lo; r < hi; ++r)
      if (ns_key(__ldcg(logits + r)) == hit_key && left-- == 0) s.token = r;
  }
  named_sync(1, kConsumerThreads);
  const int tok = s.token;
  named_sync(1, kConsumerThreads);
  return tok;
}

}  // namespace spd
