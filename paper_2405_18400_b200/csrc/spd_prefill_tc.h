// Host-side description of one long-prefix prefill job (see spd_prefill_tc.cu).
#pragma once
#include "spd_params.h"

namespace spd {

// Requests of a batch at most; jobs of up to so many tokens apply 1 / rms behind the product; the most tokens of a context's
// jobs are a multiple of it.
constexpr int kTcTile = 128;
constexpr int kTcMaxTokens = 512; // tokens one job takes at most
// Runs of more tokens than this take the path with every model, shorter ones with large models: beyond, the 16-token kernel needs
// two launches (27 tokens, 7B shape: 9.2 ms, the job 3.5; 17 tokens, 8 layers of 1.6 MB: the job 0.32 where one launch takes 0.38).
constexpr int kTcMinPrefix = 16;

// A product Y = X W^T as it is dealt out among pairs of blocks, and where its sums are (spd_tc_product_kernel).  Tiles of
// 256 weight rows x tile_tok token rows, token tiles fastest; a tile has nk stages of 64 columns; the stages of all tiles,
// one after the other, are cut into `pairs` equal runs.  Of a tile that is cut, the part with its first column is in y
// [token][N], each later part in the buffer [tile_tok][256] of its pair.
constexpr int kTcMaxPairs = 80;  // pairs of blocks used at most (74 on 148 SMs)
constexpr int kTcMaxTileTok = 256;
struct Product {
  const float *y, *parts;
  int32_t N, nk, tile_tok, tok_tiles, total, pairs, shape;  // shape: 16, 32, 64, 128 or 256, the kernel's instance
  int32_t align;  // a cut lies a multiple of so many stages behind its tile's first (rounded down)
  int32_t seg;    // stages whose sums an accumulator takes before they move to registers
  int32_t small_first;  // one instruction per term: a stage's small terms before the large one
};

// Whether products of so many token rows may cut tiles.
inline bool cuts_tiles(int n_tok) { return n_tok <= kTcMaxTileTok; }

inline Product plan_product(int n_tok, int N, int C, int sm_count, const float *y, const float *parts) {
  Product pr;
  pr.y = y;
  pr.parts = parts;
  pr.N = N;
  pr.nk = (C + 63) / 64;
  // Up to 64 token rows the three terms share an instruction; up to 256 rows are one tile; more rows make enough tiles of
  // up to 128 (all alike) to fill the pairs without cutting one: then every sum is one pair's.  From 65 rows on a tile's rows
  // are rounded up to 16, which is what an instruction's N allows (to 32: 100 tokens, 7B shape, 5.5 ms instead of 5.1; 400
  // tokens as one job 18.6 instead of 17.0).  Between 129 and 256 rows tiles are cut at multiples of eight stages.
  const bool whole = !cuts_tiles(n_tok);
  pr.shape = n_tok <= 16 ? 16 : (n_tok <= 32 ? 32 : (n_tok <= 64 ? 64 : (n_tok <= 128 || whole ? 128 : 256)));
  pr.tok_tiles = whole ? (n_tok + 127) / 128 : 1;
  pr.tile_tok = pr.shape <= 64 ? pr.shape : ((n_tok + pr.tok_tiles - 1) / pr.tok_tiles + 15) / 16 * 16;
  pr.total = (N + 255) / 256 * pr.tok_tiles * pr.nk;
  pr.align = whole ? pr.nk : (pr.shape == 256 ? 8 : 1);
  // The accumulators add with truncation, so the error grows with the additions between two moves to registers: 4 per stage
  // and accumulator where every term has its own (up to 64 rows), 12 where the terms share one (small ones first: 4 at the
  // sum's own size).  4 stages cost nothing (2: 1 % at 15 tokens, 3 % at 64; 1: 2 % and 10 %).  Where the terms share one, C / 512
  // stages at most, as many additions as the 3 C / 128 that a warp of the 16-token kernel chains; two at least beyond 128 rows,
  // where the epilogue of one stage takes longer than its instructions (8 layers of 256 columns, 200 tokens: one stage 0.85 ms,
  // two 0.77; error of the first timestep 4.0e-7 and 5.9e-7, the 16-token kernel's path 1.9e-6).  Uncut tiles of wide matrices
  // take up to 8 stages, the terms in order: a bf16 cache behind a long prefix then holds the bits that it always has.  (Four
  // there, and two up to 384 rows, cost 1 % of the time and come closer to 64 bits: 300 tokens, 7B shape, first timestep's
  // logits, relative 2-norm, 6.8e-6 instead of 3.1e-5.  But 28 of 60 requests then chose another draft within nine timesteps behind
  // 100 to 1900 tokens.)
  const int least_seg = n_tok > 128 ? 2 : 1, most_seg = whole ? 8 : 4, wide = C / 512;
  pr.seg = pr.shape <= 64 ? 4 : (wide < least_seg ? least_seg : (wide < most_seg ? wide : most_seg));
  pr.small_first = pr.seg < 8;
  // a pair takes a whole tile, two steps of the cuts (16 stages) or four stages at least (small matrices: fewer parts to add)
  const int least = whole ? pr.nk : (pr.align > 1 ? 2 * pr.align : 4);
  const int most = sm_count / 2 < kTcMaxPairs ? sm_count / 2 : kTcMaxPairs, worth = pr.total / least;
  pr.pairs = most < worth ? most : worth;
  if (pr.pairs < 1) pr.pairs = 1;
  return pr;
}

#ifdef __CUDACC__
// First stage of a pair's run.
__device__ __forceinline__ int product_cut(const Product &pr, int pair) {
  const int raw = (int)((unsigned)pr.total * (unsigned)pair / (unsigned)pr.pairs);
  return raw - raw % pr.nk % pr.align;
}
// The last pair whose cut, before the rounding, is not behind a stage.
__device__ __forceinline__ int product_pair(const Product &pr, int stage) {
  return (int)(((unsigned)(stage + 1) * (unsigned)pr.pairs - 1u) / (unsigned)pr.total);
}
// The later parts of row tile `rt`'s sums for token t: parts [first, last) and the offset of row 0 of the tile in part 0.
struct TileParts {
  int first, last;
  size_t at, step;
};
__device__ __forceinline__ TileParts product_parts(const Product &pr, int t, int rt) {
  const int tt = t / pr.tile_tok, u = (rt * pr.tok_tiles + tt) * pr.nk;
  TileParts tp;
  tp.first = product_pair(pr, u + min(pr.align, pr.nk) - 1) + 1;  // (cuts that were rounded down to the tile's first stage)
  tp.last = product_pair(pr, u + pr.nk - 1) + 1;
  tp.step = (size_t)pr.tile_tok * 256;
  tp.at = (size_t)(t - tt * pr.tile_tok) * 256;
  return tp;
}
// Y[t][r .. r+3]; r and N multiples of 4.  kFlight parts are asked for together; they are added in order whatever it is.
// Few token rows (up to kFewRows), 6: the row-wise kernels between two products are little more than a chain of trips to L2, and
// a loop that adds as it loads makes one trip per part (7B shape: five later parts of a tile in the attention-output and
// down products).  With the gains and rotary angles asked for before dep_wait, 8 requests 3.13 -> 3.03 ms per timestep, 27 tokens
// 3.29 -> 3.22 ms.
// More rows, 1: six parts take 56 to 72 registers instead of 42 to 54, so fewer blocks fit an SM, and the attention's blocks,
// which come onto the SMs as these leave, lie less evenly.  One / six: 4096 columns, 8 layers, 15 tokens 0.859 / 0.842 ms, 27
// 0.878 / 0.869, 64 1.012 / 1.043; 3072 columns, 4 layers, 128 tokens 0.500 / 0.558.
// Rows whose products cut no tiles, 0: no parts, 28 to 32 registers.  None / one / six: 1024 columns, heads of 64, 8 layers,
// 700 tokens 1.72 / 1.76 / 1.82 ms, 1500 3.09 / 3.27 / 3.38; 4096 columns, 8 layers, 512 tokens 4.39 / 4.44 / 4.42.
constexpr int kFewRows = 32, kPartFlight = 6;
template <int kFlight>
__device__ __forceinline__ float4 product_sum4(const Product &pr, int t, int r) {
  float4 v = *reinterpret_cast<const float4 *>(pr.y + (size_t)t * pr.N + r);
  if constexpr (kFlight > 0) {
    const TileParts tp = product_parts(pr, t, r >> 8);
    const float *part = pr.parts + tp.at + (r & 255);
    for (int p = tp.first; p < tp.last; p += kFlight) {
      float4 w[kFlight];
#pragma unroll
      for (int u = 0; u < kFlight; ++u)
        if (p + u < tp.last) w[u] = *reinterpret_cast<const float4 *>(part + (p + u) * tp.step);
#pragma unroll
      for (int u = 0; u < kFlight; ++u)
        if (p + u < tp.last) { v.x += w[u].x; v.y += w[u].y; v.z += w[u].z; v.w += w[u].w; }
    }
  }
  return v;
}
#endif

struct TcJob {
  int32_t L, d, H, hd, f, max_pos, kv_bf16;
  float eps;
  const LayerW *layers;              // HOST copy of the layer table [L]
  const __nv_bfloat16 *tok_emb;
  const uint8_t *w_tmaps;            // device: tensor maps of the layers' matrices, four per layer, then the LM head's
  const uint8_t *x_tmaps;            // device: tensor maps of the term buffer seen as [3 * x_term_rows][d] and [..][f], in boxes of 8, 16, 32
                                     // and 64 rows (two each)
  void *kcache, *vcache;
  const float2 *rope;
  float *h, *y, *q;                  // [x_term_rows][d], [x_term_rows][max(3d, 2f)], [x_term_rows][d]
  float *parts;                      // [pairs][rows of a tile][256]: parts of a product's cut tiles
  float *head_parts;                 // the same for the LM head's product of a batch, whose output overlaps `parts`
  uint16_t *x;                       // [3][x_term_rows][max(d, f)] bf16 terms
  int32_t x_term_rows;
  const int32_t *ids;                // device: the job's token ids
  int32_t pos0, n_tok;               // first position; tokens (<= x_term_rows)
  State *st;
  int32_t sm_count;                  // SMs of the device
  float *ss;                         // [128][32]: sums of squares of the residual rows per 512-column chunk
};

// Words of a request's row in a batched timestep's results (written by the tail kernel, fetched by the host in one copy).
constexpr int kBtResultWords = 64;

// Programmatic dependent launch.  dep_wait: returns once the kernel before this one in the stream has completed and
// its writes are visible (at once when the launch did not ask for the overlap).  dep_launch: the kernel after this
// one may be brought onto the SMs, where it runs up to its own dep_wait, as soon as every block of this kernel has
// said so or has ended.
#ifdef __CUDACC__
__device__ __forceinline__ void dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
#endif

// Launch with programmatic stream serialization: the kernel may be brought onto the SMs once every block of the one
// before it in the stream has said so (dep_launch) or has ended, and waits there (dep_wait) until that one has completed.
// Every block passes dep_wait before it ends, so a kernel that has completed stands for all before it and the kernels of a
// chain may be set up several deep; before its dep_wait a block touches only weights, what is as old as the call (a batch's request
// parameters, rotary tables), its own shared and tensor memory, and L2 by prefetches.
// No kernel waits for one that cannot start: a block comes onto an SM only when all blocks of the kernel before it have.
// All kernels say so first thing, so that the next product's first weight copies are under way while the one before
// drains (8 / 64 requests 3.29 / 4.38 -> 3.19 / 4.30 ms per 7B timestep), but for the rotary embedding: the attention's
// blocks would be placed while the product still holds most SMs, unevenly (3.49 -> 3.51 ms when it was tried).
template <typename... P, typename... A>
inline cudaError_t launch_dep(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

}  // namespace spd

extern "C" cudaError_t spd_internal_tc_prepare(void);
extern "C" cudaError_t spd_internal_job_prepare(void);
extern "C" cudaError_t spd_internal_tc_stall(const spd::TcJob *job, int few, cudaStream_t stream);
extern "C" cudaError_t spd_internal_tc_prefill(const spd::TcJob *job, const spd::KParams *head, cudaStream_t stream, int *launches);
// A product of n_tok token rows with matrix `which` of the weights' tensor maps; `wide`: the terms have d_ffn columns.
extern "C" cudaError_t spd_internal_product(const spd::TcJob *job, int n_tok, int wide, int which, float *Y, int N, spd::Product *out, cudaStream_t s);
// Row-wise kernels of a job (spd_batch.cu).
// y null: the rows start as the embeddings of the job's tokens.  normed: the product's terms were whole RMSNorms (spd_internal_job_norm).
extern "C" cudaError_t spd_internal_job_resid(const spd::TcJob *job, const spd::Product *y, const __nv_bfloat16 *gain, cudaStream_t s);
extern "C" cudaError_t spd_internal_job_norm(const spd::TcJob *job, const spd::Product *y, const __nv_bfloat16 *gain, cudaStream_t s);
extern "C" cudaError_t spd_internal_job_rope_cache(const spd::TcJob *job, const spd::Product *y, int normed, int layer, cudaStream_t s);
extern "C" cudaError_t spd_internal_job_swiglu(const spd::TcJob *job, const spd::Product *y, int normed, cudaStream_t s);
// The end of a prefix: last residual add, final norm, LM head, KeepTopK and first timestep of one token row (h + y).
extern "C" cudaError_t spd_internal_job_head(const spd::KParams *p, const float *h, const spd::Product *y, int sm_count, cudaStream_t s);
