// Batched Superposed Decoding: one timestep of up to 128 requests per pass over the weights (the paper's closing
// remark: batching is complementary to the method, since each request still needs one pass for its k drafts).
//
// A request is a context of its own (prefix, KV cache, draft state); the requests of a batch share the weights and
// the n-gram tables.  Their superposed inputs (Eq. 3) are the token rows of the tensor-core products
// (spd_tc_product_kernel in spd_prefill_tc.cu: the 256 weight rows of a tile are the wide tcgen05.mma operand, the
// requests' activations, as three exact bf16 terms, the narrow one, TMEM accumulators, stages dealt among pairs of blocks),
// so the weights are streamed once per timestep whatever the number of requests.  Between the products run
// element-wise kernels spread over requests and columns: the superposed embedding, the rotary embedding and the
// append to the request's own cache at its own position, attention over that cache (a block per request and head),
// residual add and SwiGLU; RMSNorm's 1 / rms is applied behind the product that follows it.  After the LM head (one
// more product, a row of logits per request) a block per request runs the method's tail on the request's own draft
// state: KeepTopK, Eq. 5-7 with the n-gram probes, Eq. 2, Eq. 4.  The row-wise kernels serve the jobs of the long-prefix path
// as well, whose norm for long jobs and whose last launch are here too.
#include <cuda_runtime.h>
#include <math_constants.h>

#include "spd_params.h"
#include "spd_prefill_tc.h"
#include "spd_ptx.cuh"
#include "spd_tail.cuh"
#include "spd_score.cuh"

namespace spd {

// v = hi + mid + lo exactly: each term takes the leading 8 significant bits of what is left, by truncation.
__device__ __forceinline__ void bt_split3(float v, uint32_t &hi, uint32_t &mid, uint32_t &lo) {
  hi = __float_as_uint(v) >> 16;
  const float r1 = v - __uint_as_float(hi << 16);
  mid = __float_as_uint(r1) >> 16;
  lo = __float_as_uint(r1 - __uint_as_float(mid << 16)) >> 16;
}
__device__ __forceinline__ void bt_put3(uint16_t *X, size_t term_stride, size_t at, float v) {
  uint32_t hi, mid, lo;
  bt_split3(v, hi, mid, lo);
  X[at] = (uint16_t)hi;
  X[at + term_stride] = (uint16_t)mid;
  X[at + 2 * term_stride] = (uint16_t)lo;
}
// Four neighbouring columns (at and term_stride multiples of 4).
__device__ __forceinline__ void bt_put3x4(uint16_t *X, size_t term_stride, size_t at, const float4 &v) {
  uint32_t h[4], m[4], l[4];
  bt_split3(v.x, h[0], m[0], l[0]);
  bt_split3(v.y, h[1], m[1], l[1]);
  bt_split3(v.z, h[2], m[2], l[2]);
  bt_split3(v.w, h[3], m[3], l[3]);
  *reinterpret_cast<uint2 *>(X + at) = make_uint2(h[0] | (h[1] << 16), h[2] | (h[3] << 16));
  *reinterpret_cast<uint2 *>(X + at + term_stride) = make_uint2(m[0] | (m[1] << 16), m[2] | (m[3] << 16));
  *reinterpret_cast<uint2 *>(X + at + 2 * term_stride) = make_uint2(l[0] | (l[1] << 16), l[2] | (l[3] << 16));
}
// Four neighbouring bf16 values (8-byte aligned).
__device__ __forceinline__ float4 bt_load4(const __nv_bfloat16 *p) {
  const uint2 w = *reinterpret_cast<const uint2 *>(p);
  return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16), __uint_as_float(w.y & 0xffff0000u));
}
__device__ __forceinline__ float4 bt_mul(const float4 &a, const float4 &b) { return make_float4(a.x * b.x, a.y * b.y, a.z * b.z, a.w * b.w); }

// The row-wise work between the products, of a batch's requests or a short job's tokens, is spread over rows and columns: a
// block takes kBtCols columns of one token row, a thread four neighbouring ones (16-byte loads; with two columns a
// thread and 2-byte stores of the terms the SwiGLU of 100 tokens, 7B shape, took 14 us, now 8).  RMSNorm's factor 1 / rms(h)
// is common to a row's columns and moves behind the product (as in the single-request kernel): the kernels that write a
// residual row h store h * gain as the next product's terms and the sum of squares of their columns (ss[row][chunk]);
// the kernels that read that product multiply its rows by rsqrt(sum of the row's chunks / d + eps).
constexpr int kBtCols = 512;
constexpr int kBtThreads = kBtCols / 4;
constexpr int kBtMaxChunks = 32;  // d_model <= 16384
static_assert(8 + 3 * kMaxK <= kBtResultWords, "a request's row of results holds the head and three lists of k");

// The gains of the thread's columns: weights, asked for before dep_wait.
__device__ __forceinline__ float4 bt_gain(const __nv_bfloat16 *gain, int c, int d) { return c < d ? bt_load4(gain + c) : make_float4(0.f, 0.f, 0.f, 0.f); }

// A chunk of a residual row: stored, its terms times the gain, its sum of squares.  All threads of the block.
__device__ __forceinline__ void bt_store_row(float *h, const float4 &gain, uint16_t *X, size_t term_stride, int row, int d, int c,
                                             const float4 &v, float *ss) {
  __shared__ float scratch[kBtThreads / 32];
  float sq = 0.f;
  if (c < d) {
    const size_t at = (size_t)row * d + c;
    *reinterpret_cast<float4 *>(h + at) = v;
    sq = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, v.w * v.w)));
    bt_put3x4(X, term_stride, at, bt_mul(v, gain));
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = sq;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.f;
#pragma unroll
    for (int w = 0; w < kBtThreads / 32; ++w) s += scratch[w];
    ss[row * kBtMaxChunks + blockIdx.y] = s;
  }
}

// 1 / rms of a row from its chunks' sums of squares (ss null: the product's terms were whole RMSNorms).  The first eight are asked for
// when the object is made, the product's sums by the caller behind that, and all are waited for together; they are added in order.
struct RowScale {
  static constexpr int kFirst = 8;
  const float *ss;
  int nch;
  float a[kFirst];
  __device__ __forceinline__ RowScale(const float *rows, int row, int d) : ss(rows ? rows + row * kBtMaxChunks : nullptr), nch((d + kBtCols - 1) / kBtCols) {
    if (ss) {  // (a select per load left the rotary kernel's blocks, and the attention's behind them, less evenly placed: 1024 columns, 200 tokens 1 %)
#pragma unroll
      for (int u = 0; u < kFirst; ++u) a[u] = u < nch ? ss[u] : 0.f;
    }
  }
  __device__ __forceinline__ float value(int d, float eps) const {
    if (!ss) return 1.f;
    float s = 0.f;
#pragma unroll
    for (int u = 0; u < kFirst; ++u) s += a[u];
    for (int c = kFirst; c < nch; ++c) s += ss[c];
    return rsqrtf(s / (float)d + eps);
  }
};

// Position of the request's input in timestep `step` of the call: the device copy of a request's parameters keeps the first one's in
// pos0.  (From the draft state, which the timestep before writes, it was two trips to L2 behind the kernels' wait.)
__device__ __forceinline__ int bt_pos(const KParams &p, int step) { return p.pos0 + step; }

// grid (requests, column chunks): the superposed input of Eq. 3, h = sum_i gamma_i E[last token of draft i], stored as
// the request's residual row; h * gain of the first layer's norm as three bf16 terms; the chunk's sum of squares.
// begin: the first timestep of a call, which clears the requests' error words (a memset per request took the stream 0.1 ms for 64).
__global__ void __launch_bounds__(kBtThreads) spd_batch_input_kernel(const KParams *kps, float *h, const __nv_bfloat16 *gain, uint16_t *X,
                                                                     size_t term_stride, int d, float *ss, int begin) {
  dep_launch();
  const int c = blockIdx.y * kBtCols + threadIdx.x * 4;
  const float4 gq = bt_gain(gain, c, d);
  dep_wait();
  const KParams &p = kps[blockIdx.x];
  const State *st = p.st;
  if (begin && blockIdx.y == 0 && threadIdx.x == 0) {
    p.st->bar = p.st->stop = p.st->abort_flag = 0u;
    p.st->err = p.st->err_info = 0;
  }
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < d)
    for (int i = 0; i < p.k; ++i) {
      const float g = st->gamma[i];
      const float4 e = bt_load4(p.tok_emb + (size_t)st->win[i][kWin - 1] * d + c);
      acc.x = fmaf(g, e.x, acc.x);
      acc.y = fmaf(g, e.y, acc.y);
      acc.z = fmaf(g, e.z, acc.z);
      acc.w = fmaf(g, e.w, acc.w);
    }
  bt_store_row(h, gq, X, term_stride, blockIdx.x, d, c, acc, ss);
}

// grid (tokens, column chunks): a job's residual rows start as its tokens' embeddings.
__global__ void __launch_bounds__(kBtThreads) spd_job_input_kernel(const int32_t *ids, const __nv_bfloat16 *tok_emb, float *h,
                                                                   const __nv_bfloat16 *gain, uint16_t *X, size_t term_stride, int d, float *ss) {
  dep_launch();
  const int c = blockIdx.y * kBtCols + threadIdx.x * 4;
  const float4 gq = bt_gain(gain, c, d);
  dep_wait();
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < d) v = bt_load4(tok_emb + (size_t)ids[blockIdx.x] * d + c);
  bt_store_row(h, gq, X, term_stride, blockIdx.x, d, c, v, ss);
}

// grid (rows, column chunks): residual add h += y, h * gain of the next norm as terms, the chunk's sum of squares.
template <int kFlight>
__global__ void __launch_bounds__(kBtThreads) spd_batch_resid_kernel(float *h, const __grid_constant__ Product y, const __nv_bfloat16 *gain,
                                                                     uint16_t *X, size_t term_stride, int d, float *ss) {
  dep_launch();
  const int c = blockIdx.y * kBtCols + threadIdx.x * 4;
  const float4 gq = bt_gain(gain, c, d);
  dep_wait();
  float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
  if (c < d) {
    v = *reinterpret_cast<const float4 *>(h + (size_t)blockIdx.x * d + c);
    const float4 a = product_sum4<kFlight>(y, blockIdx.x, c);
    v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
  }
  bt_store_row(h, gq, X, term_stride, blockIdx.x, d, c, v, ss);
}

// Long jobs (more than 128 tokens): a token row per block, the whole RMSNorm before the product.  With hundreds of rows
// the chip is full either way; the norm stays in front of the product there so that the tensor cores see the same operands,
// and truncate the same way, as they always have for these lengths (a bf16 cache turns a difference in the sixth digit into
// another rounding of one value in a hundred).  The row waits in shared memory between the sum of squares, taken a column
// per thread, and the terms, four columns per thread (8-byte stores).
template <int kFlight>
__global__ void __launch_bounds__(256) spd_job_norm_kernel(float *h, const __grid_constant__ Product y, const int32_t *ids, const __nv_bfloat16 *emb,
                                                           const __nv_bfloat16 *gain, uint16_t *X, size_t term_stride, int d, float eps) {
  dep_launch();
  dep_wait();
  extern __shared__ __align__(16) float jn_row[];  // [d]
  __shared__ float scratch[8];
  const int t = blockIdx.x;
  float *hr = h + (size_t)t * d;
  for (int c = threadIdx.x * 4; c < d; c += 1024) {
    float4 v;
    if (ids) v = bt_load4(emb + (size_t)ids[t] * d + c);
    else {
      v = *reinterpret_cast<const float4 *>(hr + c);
      const float4 a = product_sum4<kFlight>(y, t, c);
      v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
    }
    *reinterpret_cast<float4 *>(hr + c) = v;
    *reinterpret_cast<float4 *>(jn_row + c) = v;
  }
  __syncthreads();
  float ss = 0.f;
  for (int c = threadIdx.x; c < d; c += 256) ss = fmaf(jn_row[c], jn_row[c], ss);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffffffu, ss, o);
  if ((threadIdx.x & 31) == 0) scratch[threadIdx.x >> 5] = ss;
  __syncthreads();
  float sum = 0.f;
#pragma unroll
  for (int w = 0; w < 8; ++w) sum += scratch[w];
  const float rs = rsqrtf(sum / (float)d + eps);
  for (int c = threadIdx.x * 4; c < d; c += 1024) {
    const float4 v = *reinterpret_cast<const float4 *>(jn_row + c);
    bt_put3x4(X, term_stride, (size_t)t * d + c, bt_mul(make_float4(v.x * rs, v.y * rs, v.z * rs, v.w * rs), bt_load4(gain + c)));
  }
}

// Columns c .. c+3 of one token row: the QKV product's row [q | k | v] times 1 / rms, rotary embedding of q and k
// (adjacent pairs) at position pos, q to Q, k and v into the cache.
__device__ __forceinline__ float4 bt_rotate(const float4 &x, const float4 &cs) {  // cs = (cos, sin) of the two pairs
  return make_float4(__fmaf_rn(x.x, cs.x, -__fmul_rn(x.y, cs.y)), __fmaf_rn(x.x, cs.y, __fmul_rn(x.y, cs.x)),
                     __fmaf_rn(x.z, cs.z, -__fmul_rn(x.w, cs.w)), __fmaf_rn(x.z, cs.w, __fmul_rn(x.w, cs.z)));
}
__device__ __forceinline__ void bt_store_kv(void *cache, int kv_bf16, size_t at, const float4 &v) {
  if (kv_bf16) {
    const __nv_bfloat162 a = __halves2bfloat162(__float2bfloat16_rn(v.x), __float2bfloat16_rn(v.y));
    const __nv_bfloat162 b = __halves2bfloat162(__float2bfloat16_rn(v.z), __float2bfloat16_rn(v.w));
    *reinterpret_cast<uint2 *>(static_cast<__nv_bfloat16 *>(cache) + at) =
        make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
  } else {
    *reinterpret_cast<float4 *>(static_cast<float *>(cache) + at) = v;
  }
}
__device__ __forceinline__ float4 bt_angles(const float2 *rope, int hd, int pos, int c) {
  return *reinterpret_cast<const float4 *>(rope + (size_t)pos * (hd / 2) + (c % hd) / 2);
}
template <int kFlight>
__device__ __forceinline__ void bt_rope_cache(const Product &y, const float *ss, float eps, float *Q, void *kcache, void *vcache, const float4 &cs, int max_pos,
                                              int kv_bf16, int d, int layer, int t, int pos, int c) {
  const RowScale scale(kFlight ? ss : nullptr, t, d);  // (rows that cut no tiles have their norms in front of the product)
  const float4 q = product_sum4<kFlight>(y, t, c), k = product_sum4<kFlight>(y, t, d + c), v = product_sum4<kFlight>(y, t, 2 * d + c);
  const float rs = scale.value(d, eps);
  const size_t at = ((size_t)layer * max_pos + pos) * d + c;
  *reinterpret_cast<float4 *>(Q + (size_t)t * d + c) = bt_rotate(make_float4(q.x * rs, q.y * rs, q.z * rs, q.w * rs), cs);
  bt_store_kv(kcache, kv_bf16, at, bt_rotate(make_float4(k.x * rs, k.y * rs, k.z * rs, k.w * rs), cs));
  bt_store_kv(vcache, kv_bf16, at, make_float4(v.x * rs, v.y * rs, v.z * rs, v.w * rs));
}

// grid (requests, column chunks): each request at its own position, into its own cache.
template <int kFlight>
__global__ void __launch_bounds__(kBtThreads) spd_batch_rope_cache_kernel(const __grid_constant__ Product y, const float *ss, float eps, float *Q,
                                                                          const KParams *kps, int d, int hd, int layer, int step) {
  // what does not hang on the product: the request's parameters (as old as the call), its position's angles
  const KParams &p = kps[blockIdx.x];
  const int c = blockIdx.y * kBtCols + threadIdx.x * 4, pos = bt_pos(p, step), max_pos = p.max_pos, kv_bf16 = p.kv_bf16;
  void *kcache = p.kcache, *vcache = p.vcache;
  const float4 cs = c < d ? bt_angles(p.rope, hd, pos, c) : make_float4(0.f, 0.f, 0.f, 0.f);
  dep_wait();
  dep_launch();
  if (c >= d) return;
  bt_rope_cache<kFlight>(y, ss, eps, Q, kcache, vcache, cs, max_pos, kv_bf16, d, layer, blockIdx.x, pos, c);
}

// The same for a job of prefix tokens of one request (token t at position pos0 + t, one cache).
template <int kFlight>
__global__ void __launch_bounds__(kBtThreads) spd_job_rope_cache_kernel(const __grid_constant__ Product y, const float *ss, float eps, float *Q,
                                                                        void *kcache, void *vcache, const float2 *rope, int max_pos, int kv_bf16,
                                                                        int d, int hd, int layer, int pos0) {
  const int c = blockIdx.y * kBtCols + threadIdx.x * 4, pos = pos0 + blockIdx.x;
  const float4 cs = c < d ? bt_angles(rope, hd, pos, c) : make_float4(0.f, 0.f, 0.f, 0.f);  // (a table as old as the context)
  dep_wait();
  dep_launch();
  if (c >= d) return;
  bt_rope_cache<kFlight>(y, ss, eps, Q, kcache, vcache, cs, max_pos, kv_bf16, d, layer, blockIdx.x, pos, c);
}

// grid (rows, chunks of the FFN): u = SiLU(gate) * up from the gate / up product's row times 1 / rms
// (Y row = [gate_0, up_0, gate_1, up_1, ...]), as three bf16 terms.
__device__ __forceinline__ float bt_swiglu(float gate, float up, float rs) {
  const float g = gate * rs, u = up * rs;
  return g / (1.f + __expf(-g)) * u;
}
template <int kFlight>
__global__ void __launch_bounds__(kBtThreads) spd_batch_swiglu_kernel(const __grid_constant__ Product y, const float *ss, float eps, int d, uint16_t *X,
                                                                      size_t term_stride, int f) {
  dep_launch();
  dep_wait();
  const int t = blockIdx.x, j = blockIdx.y * kBtCols + threadIdx.x * 4;
  if (j >= f) return;
  // (rows that cut no tiles have their norms in front of the product)
  // The scale is waited for in front of the sums.  Asked for together with them it takes two more registers, and an attention of just
  // over the 740 blocks that are resident together then ends later: 16 layers of the 7B shape, float32 cache, behind 400 positions, 24 /
  // 26 requests 2.94 / 3.02 ms instead of 2.78 / 2.84 (16 requests 2.31 instead of 2.43; neither way is the better one elsewhere).
  const float rs = RowScale(kFlight ? ss : nullptr, t, d).value(d, eps);
  const float4 a = product_sum4<kFlight>(y, t, 2 * j), b = product_sum4<kFlight>(y, t, 2 * j + 4);
  bt_put3x4(X, term_stride, (size_t)t * f + j,
            make_float4(bt_swiglu(a.x, a.y, rs), bt_swiglu(a.z, a.w, rs), bt_swiglu(b.x, b.y, rs), bt_swiglu(b.z, b.w, rs)));
}

// One (request, head) per block of eight warps: softmax attention of the request's query over its own cache.  Bound by
// the cache rows' latency and bytes, so a position is read with one 16-byte load per lane and cache: HD * sizeof(E) / 16
// lanes hold a position (16 for bf16 of head size 128, two positions per warp side by side), and four positions per
// group of lanes are in flight before the first is used; they enter the running softmax together (one rescale per round).
// A round of the block is 32 (float32, head size 128) to 128 positions (bf16, 64).  The groups' states are merged in
// shared memory in a fixed order; output as three bf16 terms.  7B shape, bf16 cache, whole timestep of 8 / 64 requests
// behind 150 positions each: 4.58 / 7.99 ms (a warp per position, one in flight, element-wise loads), now 3.51 / 6.14 ms; with the
// request's position known before the wait, no trip to L2 for it, and the rows asked into L2 while the rotary kernel runs, three
// timesteps of 8 / 64 requests behind 15 to 90 positions (float32 cache) 9.47 / 16.28 -> 9.31 / 15.58 ms.
// The blocks that are resident together ask for half of L2, their first rows.  All rows at once, where that is more than L2 holds, push
// one another out before they are read.  8 layers of the 7B shape, ms per timestep, none / bounded / all: float32, 32 requests behind
// 500 positions 1.66 / 1.63 / 1.89, behind 2000 3.75 / 3.76 / 5.11, 16 behind 1000 1.66 / 1.55 / 1.73, 1 behind 2000 1.40 / 1.28 / 1.27;
// bf16, 32 behind 2000 2.54 / 2.46 / 2.93.  (32 to 96 MB, for all blocks or for the first to come only: alike.)
constexpr int kBaWarps = 8, kBaFlight = 4, kBaPerSm = 5, kBaAhead = 64 << 20;

template <typename E>
__device__ __forceinline__ void ba_unpack(const uint4 &v, float (&x)[16 / sizeof(E)]) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int e = 0; e < 4; ++e) {
    if constexpr (sizeof(E) == 2) {
      x[2 * e] = __uint_as_float(w[e] << 16);
      x[2 * e + 1] = __uint_as_float(w[e] & 0xffff0000u);
    } else {
      x[e] = __uint_as_float(w[e]);
    }
  }
}

template <int HD, typename E>
__device__ void ba_head(const float *q_row, const E *kc, const E *vc, int d, int T, uint16_t *X, size_t term_stride, size_t x_at, float *s_acc,
                        float *s_m, float *s_l) {
  constexpr int EPL = 16 / (int)sizeof(E);           // elements per lane
  constexpr int LP = HD / EPL;                       // lanes per position
  constexpr int GW = 32 / LP, G = GW * kBaWarps;     // groups of lanes per warp, per block
  const int lane = threadIdx.x & 31, group = (threadIdx.x >> 5) * GW + lane / LP, at = (lane % LP) * EPL;
  const float scale = 1.f / sqrtf((float)HD);
  float q[EPL], acc[EPL];
#pragma unroll
  for (int e = 0; e < EPL; e += 4) {
    const float4 v = *reinterpret_cast<const float4 *>(q_row + at + e);
    q[e] = v.x; q[e + 1] = v.y; q[e + 2] = v.z; q[e + 3] = v.w;
  }
#pragma unroll
  for (int e = 0; e < EPL; ++e) acc[e] = 0.f;
  float m = -CUDART_INF_F, l = 0.f;
  for (int tb = 0; tb < T; tb += G * kBaFlight) {  // all lanes of a warp go round together (the shuffles)
    uint4 kq[kBaFlight], vq[kBaFlight];
#pragma unroll
    for (int u = 0; u < kBaFlight; ++u) kq[u] = *reinterpret_cast<const uint4 *>(kc + (size_t)min(tb + u * G + group, T - 1) * d + at);
#pragma unroll
    for (int u = 0; u < kBaFlight; ++u) vq[u] = *reinterpret_cast<const uint4 *>(vc + (size_t)min(tb + u * G + group, T - 1) * d + at);
    float sc[kBaFlight], mn = m;
    bool any = false;
#pragma unroll
    for (int u = 0; u < kBaFlight; ++u) {
      float kx[EPL], dot = 0.f;
      ba_unpack<E>(kq[u], kx);
#pragma unroll
      for (int e = 0; e < EPL; ++e) dot = fmaf(q[e], kx[e], dot);
#pragma unroll
      for (int o = LP / 2; o > 0; o >>= 1) dot += __shfl_xor_sync(0xffffffffu, dot, o);
      sc[u] = tb + u * G + group < T ? dot * scale : -CUDART_INF_F;
      mn = fmaxf(mn, sc[u]);
      any |= sc[u] != -CUDART_INF_F;
    }
    if (any) {  // else no position of this round belongs to the group (a NaN score, which fmaxf passes over, has to reach the sums)
      const float c = __expf(m - mn);
      l *= c;
#pragma unroll
      for (int e = 0; e < EPL; ++e) acc[e] *= c;
#pragma unroll
      for (int u = 0; u < kBaFlight; ++u) {
        const float pw = __expf(sc[u] - mn);  // 0 past the last position
        float vx[EPL];
        ba_unpack<E>(vq[u], vx);
        l += pw;
#pragma unroll
        for (int e = 0; e < EPL; ++e) acc[e] = fmaf(pw, vx[e], acc[e]);
      }
      m = mn;
    }
  }
#pragma unroll
  for (int e = 0; e < EPL; ++e) s_acc[group * HD + at + e] = acc[e];
  if (lane % LP == 0) {
    s_m[group] = m;
    s_l[group] = l;
  }
  __syncthreads();
  if (threadIdx.x < HD) {
    float M = -CUDART_INF_F;
#pragma unroll
    for (int g = 0; g < G; ++g) M = fmaxf(M, s_m[g]);
    float L = 0.f, A = 0.f;
#pragma unroll 8
    for (int g = 0; g < G; ++g) {
      const float wgt = s_m[g] == -CUDART_INF_F ? 0.f : __expf(s_m[g] - M);
      L = fmaf(s_l[g], wgt, L);
      A = fmaf(s_acc[g * HD + threadIdx.x], wgt, A);
    }
    bt_put3(X, term_stride, x_at + threadIdx.x, A / L);
  }
}

// ahead: bytes of keys, and of values, that a block may ask for before its wait.
template <int HD>
__global__ void __launch_bounds__(kBaWarps * 32) spd_batch_attn_kernel(const float *Q, const KParams *kps, uint16_t *X, size_t term_stride, int d,
                                                                       int layer, int step, int ahead) {
  dep_launch();
  constexpr int kGroups = kBaWarps * 32 / (HD / 8);  // bf16: the larger number of groups
  __shared__ float s_acc[kGroups * HD], s_m[kGroups], s_l[kGroups];
  const KParams &p = kps[blockIdx.x];
  const int T = bt_pos(p, step) + 1, kv_bf16 = p.kv_bf16;
  const void *kcache = p.kcache, *vcache = p.vcache;
  const size_t x_at = (size_t)blockIdx.x * d + blockIdx.y * HD, base = (size_t)layer * p.max_pos * d + blockIdx.y * HD;
  // The first cached rows are on their way to L2 while the kernel before this one still runs (a hint: they are read behind the wait).
  {
    const int esz = kv_bf16 ? 2 : 4, shift = (HD == 128 ? 1 : 0) + (kv_bf16 ? 0 : 1);  // a row is 2^shift lines of 128 bytes
    const int rows = min(T - 1, ahead >> (7 + shift));
    for (int i = threadIdx.x; i < rows << shift; i += kBaWarps * 32) {
      const size_t off = (base + (size_t)(i >> shift) * d) * esz + (size_t)(i & ((1 << shift) - 1)) * 128;
      asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const uint8_t *>(kcache) + off));
      asm volatile("prefetch.global.L2 [%0];" ::"l"(static_cast<const uint8_t *>(vcache) + off));
    }
  }
  dep_wait();
  if (kv_bf16)
    ba_head<HD>(Q + x_at, static_cast<const __nv_bfloat16 *>(kcache) + base, static_cast<const __nv_bfloat16 *>(vcache) + base, d, T, X,
                term_stride, x_at, s_acc, s_m, s_l);
  else
    ba_head<HD>(Q + x_at, static_cast<const float *>(kcache) + base, static_cast<const float *>(vcache) + base, d, T, X, term_stride, x_at,
                s_acc, s_m, s_l);
}

// One request per block (512 threads): the request's row of logits (the LM head's partial products added, times
// 1 / rms of the final norm) goes to its own buffer; every warp ranks a sixteenth of the vocabulary, warp 0 merges
// the sixteen lists (KeepTopK with log-probabilities under temperature tau, Algorithm 1); then Eq. 5-7, Eq. 2 and
// Eq. 4 on the request's own draft state, as block 0 of the single-request kernel does.
__global__ void __launch_bounds__(kConsumerThreads) spd_batch_tail_kernel(const KParams *kps, const __grid_constant__ Product y, const float *ss,
                                                                          float eps, int V, int32_t *results) {
  dep_wait();
  dep_launch();
  extern __shared__ __align__(16) uint8_t bt_smem[];
  __shared__ int s_dead, s_quit;
  const KParams &p = kps[blockIdx.x];
  const float rs = RowScale(ss, blockIdx.x, p.d).value(p.d, eps);
  const float *row = y.y + (size_t)blockIdx.x * V;
  // a warp takes row tiles of the product (256 logits, alike in their parts) in turn
  for (int rt = threadIdx.x >> 5; rt * 256 < V; rt += kConsumerWarps) {
    const TileParts tp = product_parts(y, blockIdx.x, rt);
    float z[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int c = rt * 256 + e * 32 + (threadIdx.x & 31);
      z[e] = c < V ? row[c] : 0.f;
    }
    for (int q = tp.first; q < tp.last; ++q)
#pragma unroll
      for (int e = 0; e < 8; ++e) z[e] += y.parts[q * tp.step + tp.at + e * 32 + (threadIdx.x & 31)];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const int c = rt * 256 + e * 32 + (threadIdx.x & 31);
      if (c < V) p.logits[c] = z[e] * rs;
    }
  }
  if (threadIdx.x == 0) s_dead = s_quit = 0;
  __syncthreads();
  {
    const int warp = threadIdx.x >> 5;
    const int r0 = (int)((long long)V * warp / kConsumerWarps), r1 = (int)((long long)V * (warp + 1) / kConsumerWarps);
    block_topk(p, r0, r1, warp);  // this warp's list: slot `warp` of the request's own partial lists
  }
  __threadfence_block();
  __syncthreads();
  if (threadIdx.x < 32) tail_keep_topk(p, kConsumerWarps);
  __syncthreads();
  Blk b;
  b.p = &p;
  b.part = reinterpret_cast<float *>(bt_smem);
  b.dead = &s_dead;
  b.quit = &s_quit;
  b.bar_target = 0;
  b.c_stage = b.c_phase = 0;
  const int step = p.st->n_gen;
  tail_score_select(b, false, step);
  // The request's row of the batch's results, which the host fetches with one copy for all requests: the state's
  // first words (stop, abort flag, error, error info, window length, tokens generated), then the k new tokens, their
  // parents and gamma.
  __syncthreads();
  if (threadIdx.x < kBtResultWords) {
    const State *st = p.st;
    const int i = threadIdx.x;
    int32_t v = 0;
    if (i == 0) v = (int32_t)st->stop;
    else if (i == 1) v = (int32_t)st->abort_flag;
    else if (i == 2) v = st->err;
    else if (i == 3) v = st->err_info;
    else if (i == 4) v = st->win_len;
    else if (i == 5) v = st->n_gen;
    else if (i >= 8 && i < 8 + p.k) v = p.hist_tok[(size_t)step * p.k + (i - 8)];
    else if (i >= 8 + kMaxK && i < 8 + kMaxK + p.k) v = p.hist_par[(size_t)step * p.k + (i - 8 - kMaxK)];
    else if (i >= 8 + 2 * kMaxK && i < 8 + 2 * kMaxK + p.k) v = __float_as_int(st->gamma[i - 8 - 2 * kMaxK]);
    results[(size_t)blockIdx.x * kBtResultWords + i] = v;
  }
}

// The end of a prefix on the long-prefix path: the last product's partial sums and the residual row of the prefix's last
// token, the final norm, that row's logits, KeepTopK and the first timestep (Eq. 1), one launch.  One token row against
// [V][d] weights is a stream of the weights (262 MB at 7B shape, 40 us at the copy bandwidth), so a block per SM takes a
// contiguous range of the vocabulary and a warp four of its rows at a time (4 rows x 16 bytes per lane in flight, each
// eight activations read from shared memory serve four rows), float32 multiplies; every block computes the norm itself
// from L2.  The block that arrives last merges the blocks' top-k lists and takes the step.
constexpr int kHeadRows = 4;
__global__ void __launch_bounds__(kConsumerThreads) spd_job_head_kernel(const __grid_constant__ KParams p, const float *h,
                                                                        const __grid_constant__ Product y) {
  extern __shared__ __align__(16) float jh_x[];  // [d]: residual row times the final norm's gain
  __shared__ float s_sum[kConsumerWarps];
  __shared__ int s_last;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int r0 = (int)((long long)p.V * blockIdx.x / gridDim.x), r1 = (int)((long long)p.V * (blockIdx.x + 1) / gridDim.x);
  // the warp's first rows on their way to L2 while the product before this kernel still runs
  for (int e = lane; e < kHeadRows * p.d / 64; e += 32) {
    const int r = r0 + warp * kHeadRows + e / (p.d / 64);
    if (r < r1) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.lm_head + (size_t)r * p.d + (e % (p.d / 64)) * 64));
  }
  for (int c = threadIdx.x * 64; c < p.d; c += kConsumerThreads * 64) asm volatile("prefetch.global.L2 [%0];" ::"l"(p.final_norm + c));
  dep_wait();
  float sq = 0.f;
  for (int c = threadIdx.x * 4; c < p.d; c += kConsumerThreads * 4) {
    float4 v = *reinterpret_cast<const float4 *>(h + c);
    const float4 a = product_sum4<kPartFlight>(y, 0, c);
    v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
    sq = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, sq))));
    *reinterpret_cast<float4 *>(jh_x + c) = bt_mul(v, bt_load4(p.final_norm + c));
    if (blockIdx.x == 0) *reinterpret_cast<float4 *>(p.h + c) = v;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
  if (lane == 0) s_sum[warp] = sq;
  __syncthreads();
  float ss = 0.f;
#pragma unroll
  for (int w = 0; w < kConsumerWarps; ++w) ss += s_sum[w];
  const float rs = rsqrtf(ss / (float)p.d + p.eps);
  for (int r = r0 + warp * kHeadRows; r < r1; r += kConsumerWarps * kHeadRows) {
    float acc[kHeadRows];
    const __nv_bfloat16 *w[kHeadRows];
#pragma unroll
    for (int i = 0; i < kHeadRows; ++i) {
      acc[i] = 0.f;
      w[i] = p.lm_head + (size_t)min(r + i, r1 - 1) * p.d;  // past the range: its last row again, not stored
    }
#pragma unroll 2
    for (int c = lane * 8; c < p.d; c += 256) {
      uint4 v[kHeadRows];
#pragma unroll
      for (int i = 0; i < kHeadRows; ++i) v[i] = __ldcs(reinterpret_cast<const uint4 *>(w[i] + c));
      const float4 xa = *reinterpret_cast<const float4 *>(jh_x + c), xb = *reinterpret_cast<const float4 *>(jh_x + c + 4);
#pragma unroll
      for (int i = 0; i < kHeadRows; ++i) {
        acc[i] = fmaf(__uint_as_float(v[i].x << 16), xa.x, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].x & 0xffff0000u), xa.y, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].y << 16), xa.z, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].y & 0xffff0000u), xa.w, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].z << 16), xb.x, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].z & 0xffff0000u), xb.y, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].w << 16), xb.z, acc[i]);
        acc[i] = fmaf(__uint_as_float(v[i].w & 0xffff0000u), xb.w, acc[i]);
      }
    }
#pragma unroll
    for (int i = 0; i < kHeadRows; ++i) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], o);
      if (lane == 0 && r + i < r1) p.logits[r + i] = acc[i] * rs;
    }
  }
  __syncthreads();
  if (warp != 0) return;
  block_topk(p, r0, r1, blockIdx.x);
  if (lane == 0) {
    __threadfence();
    s_last = atomicAdd(&p.st->bar, 1u) == gridDim.x - 1;  // zeroed by the host at the start of the call
    __threadfence();
  }
  __syncwarp();
  if (!s_last) return;
  tail_keep_topk(p, gridDim.x);
  tail_first(p, lane, 0);
  __syncwarp();
  tail_gamma(p, lane);
}

}  // namespace spd

namespace {
constexpr size_t kBatchTailSmem = 20480;
}

// Enqueues one batched timestep of n requests (kps: their parameters in device memory, in row order) on stream s.
// job: the buffers of the context that lends its long-prefix workspace; y_logits: [128][V] floats.  *launches receives
// the number of kernels enqueued.
// step: timesteps of the call before this one.
extern "C" cudaError_t spd_internal_batch_step(const spd::TcJob *job, const spd::KParams *kps, int n, int step, int V, const __nv_bfloat16 *final_norm,
                                               float *y_logits, int32_t *results, cudaStream_t s, int *launches) {
  const spd::TcJob &j = *job;
  const int d = j.d, f = j.f;
  const size_t ts_d = (size_t)j.x_term_rows * d, ts_f = (size_t)j.x_term_rows * f;
  const int nch = (d + spd::kBtCols - 1) / spd::kBtCols, nch_f = (f + spd::kBtCols - 1) / spd::kBtCols;
  const dim3 threads(spd::kBtThreads);
  const bool few = n <= spd::kFewRows;
  const int blocks = n * j.H, resident = spd::kBaPerSm * j.sm_count, ahead = spd::kBaAhead / 2 / (blocks < resident ? blocks : resident);
  int count = 0;
  cudaError_t e = cudaSuccess;
  spd::Product pr;  // where the last product's sums are
  auto done = [&](cudaError_t r) {  // a kernel enqueued
    e = r;
    ++count;
  };
  auto product = [&](int wide, int which, int N) {
    if (e == cudaSuccess) done(spd_internal_product(job, n, wide, which, j.y, N, &pr, s));
  };
  auto resid = [&](const __nv_bfloat16 *gain) {
    if (e == cudaSuccess)
      done(spd::launch_dep(few ? spd::spd_batch_resid_kernel<spd::kPartFlight> : spd::spd_batch_resid_kernel<1>, dim3(n, nch), threads, 0, s, j.h, pr, gain,
                           j.x, ts_d, d, j.ss));
  };
  done(spd::launch_dep(spd::spd_batch_input_kernel, dim3(n, nch), threads, 0, s, kps, j.h, j.layers[0].attn_norm, j.x, ts_d, d, j.ss, step == 0));
  for (int l = 0; l < j.L && e == cudaSuccess; ++l) {
    product(0, 4 * l, 3 * d);
    if (e == cudaSuccess)
      done(spd::launch_dep(few ? spd::spd_batch_rope_cache_kernel<spd::kPartFlight> : spd::spd_batch_rope_cache_kernel<1>, dim3(n, nch), threads, 0, s, pr, j.ss,
                           j.eps, j.q, kps, d, j.hd, l, step));
    if (e == cudaSuccess)
      done(j.hd == 128 ? spd::launch_dep(spd::spd_batch_attn_kernel<128>, dim3(n, j.H), dim3(spd::kBaWarps * 32), 0, s, j.q, kps, j.x, ts_d, d, l, step, ahead)
                       : spd::launch_dep(spd::spd_batch_attn_kernel<64>, dim3(n, j.H), dim3(spd::kBaWarps * 32), 0, s, j.q, kps, j.x, ts_d, d, l, step, ahead));
    product(0, 4 * l + 1, d);
    resid(j.layers[l].ffn_norm);
    product(0, 4 * l + 2, 2 * f);
    if (e == cudaSuccess)
      done(spd::launch_dep(few ? spd::spd_batch_swiglu_kernel<spd::kPartFlight> : spd::spd_batch_swiglu_kernel<1>, dim3(n, nch_f), threads, 0, s, pr, j.ss,
                           j.eps, d, j.x, ts_f, f));
    product(1, 4 * l + 3, d);
    resid(l + 1 < j.L ? j.layers[l + 1].attn_norm : final_norm);
  }
  spd::TcJob head = j;
  head.parts = j.head_parts;
  if (e == cudaSuccess) done(spd_internal_product(&head, n, 0, 4 * j.L, y_logits, V, &pr, s));
  if (e == cudaSuccess)
    done(spd::launch_dep(spd::spd_batch_tail_kernel, dim3(n), dim3(spd::kConsumerThreads), kBatchTailSmem, s, kps, pr, j.ss, j.eps, V, results));
  if (launches) *launches = count;
  return e;
}

// The row-wise kernels of a job of prefix tokens of one request (the long-prefix path), token t at position job.pos0 + t.
extern "C" cudaError_t spd_internal_job_resid(const spd::TcJob *job, const spd::Product *y, const __nv_bfloat16 *gain, cudaStream_t s) {
  const spd::TcJob &j = *job;
  const dim3 grid(j.n_tok, (j.d + spd::kBtCols - 1) / spd::kBtCols);
  const size_t ts = (size_t)j.x_term_rows * j.d;
  if (!y) return spd::launch_dep(spd::spd_job_input_kernel, grid, dim3(spd::kBtThreads), 0, s, j.ids, j.tok_emb, j.h, gain, j.x, ts, j.d, j.ss);
  return spd::launch_dep(j.n_tok <= spd::kFewRows ? spd::spd_batch_resid_kernel<spd::kPartFlight> : spd::spd_batch_resid_kernel<1>, grid,
                         dim3(spd::kBtThreads), 0, s, j.h, *y, gain, j.x, ts, j.d, j.ss);
}
extern "C" cudaError_t spd_internal_job_norm(const spd::TcJob *job, const spd::Product *y, const __nv_bfloat16 *gain, cudaStream_t s) {
  const spd::TcJob &j = *job;
  const spd::Product none = {};
  return spd::launch_dep(spd::cuts_tiles(j.n_tok) ? spd::spd_job_norm_kernel<1> : spd::spd_job_norm_kernel<0>, dim3(j.n_tok), dim3(256),
                         (size_t)j.d * 4, s, j.h, y ? *y : none, y ? nullptr : j.ids, j.tok_emb, gain, j.x, (size_t)j.x_term_rows * j.d, j.d, j.eps);
}
extern "C" cudaError_t spd_internal_job_rope_cache(const spd::TcJob *job, const spd::Product *y, int normed, int layer, cudaStream_t s) {
  const spd::TcJob &j = *job;
  return spd::launch_dep(j.n_tok <= spd::kFewRows ? spd::spd_job_rope_cache_kernel<spd::kPartFlight>
                         : spd::cuts_tiles(j.n_tok) ? spd::spd_job_rope_cache_kernel<1> : spd::spd_job_rope_cache_kernel<0>,
                         dim3(j.n_tok, (j.d + spd::kBtCols - 1) / spd::kBtCols), dim3(spd::kBtThreads), 0, s, *y,
                         normed ? nullptr : j.ss, j.eps, j.q, j.kcache, j.vcache, j.rope, j.max_pos, j.kv_bf16, j.d, j.hd, layer, j.pos0);
}
extern "C" cudaError_t spd_internal_job_swiglu(const spd::TcJob *job, const spd::Product *y, int normed, cudaStream_t s) {
  const spd::TcJob &j = *job;
  return spd::launch_dep(j.n_tok <= spd::kFewRows ? spd::spd_batch_swiglu_kernel<spd::kPartFlight>
                         : spd::cuts_tiles(j.n_tok) ? spd::spd_batch_swiglu_kernel<1> : spd::spd_batch_swiglu_kernel<0>,
                         dim3(j.n_tok, (j.f + spd::kBtCols - 1) / spd::kBtCols), dim3(spd::kBtThreads), 0, s, *y,
                         normed ? nullptr : j.ss, j.eps, j.d, j.x, (size_t)j.x_term_rows * j.f, j.f);
}

extern "C" cudaError_t spd_internal_job_head(const spd::KParams *p, const float *h, const spd::Product *y, int sm_count, cudaStream_t s) {
  return spd::launch_dep(spd::spd_job_head_kernel, dim3(sm_count), dim3(spd::kConsumerThreads), (size_t)p->d * 4, s, *p, h, *y);
}

// Kernel attributes of the current device: a row of up to 16384 float32 values in shared memory.
extern "C" cudaError_t spd_internal_job_prepare(void) {
  cudaError_t e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&spd::spd_job_norm_kernel<0>), cudaFuncAttributeMaxDynamicSharedMemorySize, 65536);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(reinterpret_cast<const void *>(&spd::spd_job_norm_kernel<1>), cudaFuncAttributeMaxDynamicSharedMemorySize, 65536);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(reinterpret_cast<const void *>(&spd::spd_job_head_kernel), cudaFuncAttributeMaxDynamicSharedMemorySize, 65536);
}
