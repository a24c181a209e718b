// Long-prefix prefill (the dense pass over the prefix that precedes Eq. 1): jobs of up to 512 prefix tokens at a
// time, their matrix products on the fifth-generation tensor cores (tcgen05.mma, operands staged in shared
// memory by tiled TMA copies, float32 accumulators in tensor memory), everything between the products in small
// row-wise kernels.  The job that ends a prefix goes on to the LM head and the first timestep of its last token
// (7B shape, host to host: 15 / 27 / 100 / 400 / 2048 tokens 3.0 / 3.1 / 5.0 / 18 / 81 ms; with 128 x 128 tiles of single
// blocks and the last 1..16 tokens in spd_prefill_kernel 4.7 / 9.2 / 12.2 / 24 / 110 ms).
//
// Product: Y[token][row] = sum_c X[token][c] W[row][c], W bf16 [rows][cols] as stored, X float32 activations
// split exactly into three bf16 terms (x = hi + mid + lo, 8 + 8 + 8 significant bits), so that the tensor
// cores see exact operands and the float32 accumulator receives what a float32 product would.  One persistent kernel
// for every number of token rows (a batch of requests, a short prefix, a job of 512 tokens): see spd_tc_product_kernel.
#include <cuda_runtime.h>
#include <math_constants.h>

#include "spd_params.h"
#include "spd_prefill_tc.h"
#include "spd_ptx.cuh"

namespace spd {

constexpr int kTcRows = 128;                   // weight rows of a tile in one block = lanes of tensor memory
constexpr int kTcKB = 64;                      // columns per stage: one 128-byte swizzle row of bf16
constexpr int kTcWBytes = kTcRows * kTcKB * 2;
constexpr int kTcThreads = 320;                // producer warp, issuing warp, eight warps for the accumulator
constexpr int kTcMaxStages = 10;
constexpr int kTcWBoxRows = 32;                // the weights' tensor maps describe boxes of 32 rows x 64 columns
constexpr int kTcMaxAccs = 4;                   // accumulator sets in rotation
constexpr unsigned long long kTcWaitNs = 1500ull * 1000ull * 1000ull;

// ---------------------------------------------------------------- PTX: tensor memory and tcgen05
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
// Shared-memory operand descriptor: K-major tile whose rows are 128 bytes (64 bf16) in the 128-byte swizzle,
// groups of 8 rows 1024 bytes apart.
__device__ __forceinline__ uint64_t tc_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);  // start address / 16
  d |= (uint64_t)1 << 16;                             // leading byte offset: unused for a swizzled K-major tile
  d |= (uint64_t)(1024 >> 4) << 32;                   // stride byte offset: one group of 8 rows
  d |= (uint64_t)1 << 46;                             // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                             // 128-byte swizzle
  return d;
}
// Instruction descriptor of kind::f16: float32 accumulator, bf16 x bf16, both operands K-major, M x N tile.
__device__ __forceinline__ constexpr uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// 8 or 16 consecutive float32 columns of this thread's lane of tensor memory (tc_ld_wait before their use).
__device__ __forceinline__ void tc_ld(uint32_t taddr, uint32_t (&r)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tc_ld(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]),
        "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
__device__ __forceinline__ void tc_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- block pairs (cta_group::2): the two blocks of a cluster multiply one tile of 256 rows; the even one ("leader") issues.
// One thread of a converged warp.  The compiler knows that it is one, which `lane == 0` does not say: tensor and copy
// instructions take their operands from the warp's uniform registers, and with `lane == 0` around them a stage of four
// instructions and seven copies cost the issuing threads about twice the cycles (QKV product of 15 tokens, 7B shape: 25.7 us
// against 22.7).
__device__ __forceinline__ bool tc_elect() {
  uint32_t p;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ uint32_t tc_cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// Address, in the cluster's shared-memory window, of the leader's object at this block's address.
__device__ __forceinline__ uint32_t tc_leader_addr(const void *p) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, 0;" : "=r"(r) : "r"(smem_u32(p)));
  return r;
}
__device__ __forceinline__ void tc_cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// The halves of a barrier of both blocks' threads.  (The arrival is a release: a warp's arrivals at the other block's mbarriers have
// been made by then.)
__device__ __forceinline__ void tc_cluster_arrive_all() { asm volatile("barrier.cluster.arrive.release;" ::: "memory"); }
__device__ __forceinline__ void tc_cluster_wait_all() { asm volatile("barrier.cluster.wait.acquire;" ::: "memory"); }
// A copy into this block's shared memory whose bytes are counted on the leader's barrier (`bar` from tc_leader_addr).
__device__ __forceinline__ void tc_pair_box_load(uint32_t dst, const void *tmap, int x, int y, uint32_t bar) {
  asm volatile("cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];" ::"r"(dst),
               "l"(tmap), "r"(x), "r"(y), "r"(bar)
               : "memory");
}
__device__ __forceinline__ void tc_pair_box_load_policy(uint32_t dst, const void *tmap, int x, int y, uint32_t bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst),
      "l"(tmap), "r"(x), "r"(y), "r"(bar), "l"(policy)
      : "memory");
}
__device__ __forceinline__ void tc_pair_alloc(uint32_t *slot, uint32_t cols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(slot)), "r"(cols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tc_pair_dealloc(uint32_t base, uint32_t cols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(cols) : "memory");
}
__device__ __forceinline__ void tc_pair_mma(uint32_t tmem_d, uint64_t da, uint64_t db, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\ttcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
// The mbarrier at this address in both blocks receives one arrival once every mma issued so far by this thread has completed.
__device__ __forceinline__ void tc_pair_commit(uint64_t *bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(smem_u32(bar)),
               "h"((uint16_t)3)
               : "memory");
}
// Arrival of a warp that has read an accumulator (tcgen05.wait::ld, tcgen05.fence::before_thread_sync): nothing written
// to memory hangs on it, so it is relaxed.  As a release it waits for the warp's stores to memory, about half a microsecond of the
// issuing thread's time per segment: 15 tokens, 7B shape, segments of 4 stages, 3.65 ms against 3.32.
__device__ __forceinline__ void tc_cluster_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.relaxed.cluster.shared::cluster.b64 _, [%0];" ::"r"(bar) : "memory");
}

struct TcShared {
  uint64_t full[kTcMaxStages], empty[kTcMaxStages], acc_full[kTcMaxAccs], acc_empty[kTcMaxAccs];
  uint32_t tmem_base;
  int dead;
};

// Bounded wait on an mbarrier phase; false when the block gave up (here or elsewhere).
__device__ __forceinline__ bool tc_wait(TcShared &sh, State *st, uint64_t *bar, uint32_t parity, int info) {
  if (mbar_try_wait(bar, parity)) return true;
  volatile int *dead = &sh.dead;
  unsigned long long t0 = globaltimer();
  uint32_t n = 0;
  while (!mbar_try_wait(bar, parity)) {
    if ((++n & 63u) == 0) {
      if (*dead) return false;
      if (globaltimer() - t0 > kTcWaitNs) {
        if (atomicCAS(&st->err, 0, -7) == 0) st->err_info = info;
        *dead = 1;
        return false;
      }
    }
  }
  return true;
}

// Y = X W^T for up to 512 token rows, by one pair of blocks per two SMs that stay for the whole product.
//
// Tile: 256 weight rows (tcgen05.mma.cta_group::2, M = 256, 128 rows in each block's shared and tensor memory) x the token
// rows of a tile.  The weights are the wide operand whatever the number of tokens, the terms the narrow one:
//   F = 16, 32, 64 (up to that many token rows): the three term tiles lie behind one another, so one instruction of
//     N = 3 x rows per 16 columns multiplies all three (N = 64 for 16 rows, whose 16 columns left over hold nothing that is
//     read: N goes in steps of 16, so 48 would do, which was not measured); each term has its own accumulator columns, added
//     in the epilogue's registers.
//   128, 256 (that many rows at most, N = the tile's rows rounded up to 16, 80 to 256): one instruction per term and 16
//     columns, all into the same columns.
// Each block brings its 128 weight rows and half of the tile's tokens.
//
// What bounds it: with up to about 64 tokens the weight stream; beyond, the tensor pipe (N = 128: 89 cycles an
// instruction of 64, N = 256: 136 of 128, measured with the copies left out), whose operands come from shared memory.
// Work is dealt in stages (64 columns of one tile): the product's stages, tile by tile and in a tile column by column, are
// cut into as many runs as there are pairs; a pair's ring of stages and its accumulators run on across tiles, so that a tile's
// epilogue overlaps the next one's stages.  Up to 256 token rows the runs are equal, so no pair idles in a last wave, and a
// tile that the cuts divide is summed by the reader: the part with the tile's first column is written to Y, a later part to its
// pair's own buffer (a pair has at most one: the start of its run).  More rows make uncut tiles of up to 128 rows: then pairs
// idle (7B shape, 512 tokens: 64 tiles on 74 pairs in the attention-output and down products, two or three a pair in QKV's
// 192), but every sum is one pair's, as in the earlier kernels, whose bits a bf16 cache behind a long prefix keeps.
// Measured (7B shape, gate / up product, ncu, one launch at a time): 512 tokens 168 us = 1.65 PFLOP/s counting the three terms,
// 0.98 of the bf16 burst peak (128 x 128 tiles of single blocks: 250 us); 200 tokens 75 us; 100 tokens 46 us; 64 tokens 37 us;
// 15 tokens 35 us where the bytes need 27.6 (the four products of a layer 93 us for 62; about 8 us of each are start and end,
// which the dependent launches hide in part).  Tried: asking the weights behind the first ring into L2 before dep_wait (8 to
// 32 stages): 2 to 5 % slower.
//
// Accumulation: an accumulator takes the sums of a segment of stages (pr.seg), then moves to registers, where the
// segments are added with round-to-nearest: the tensor cores add into their accumulator with truncation, whose error grows
// with the length of the chain.  First timestep's largest logit error, 7B shape, float32 cache, against 64 bits: 15 / 64 / 100 /
// 200 tokens 2.0e-5 / 2.4e-5 / 5.1e-5 / 5.2e-5 (segments of 24 stages, 8 from 65 rows on: 8.0e-5 / 9.6e-5 / 1.2e-4 / 1.4e-4; the
// 16-token kernel 1.3e-4), in the same time.
//
// tmap_x: the term tiles, a [3 * x_term_rows][C] bf16 matrix in boxes of kBoxRows rows x 64 columns (term j's tokens start
// at row j * x_term_rows); tmap_w: W [N][C] in boxes of 32 rows x 64 columns; rows and columns past either matrix arrive as
// zeros.  Barriers: a stage's copies by both blocks are counted on the leader's `full`; a commit signals `empty` and
// `acc_full` in both blocks; the epilogue warps of both arrive at the leader's `acc_empty`.  Every wait is bounded.
// Launched as a programmatic dependent: a block is set up and copies the weights of its whole first ring while the kernel
// before it still runs; the terms, which that kernel writes, are asked for after dep_wait.
// stall (test hook): the leader announces its first stage but no copies are issued for it, so the wait for it runs out.  In
// a run longer than the ring the producers give up too, in a shorter one they are done by then.
template <int NT>
struct TcShape {
  static constexpr bool kFused = NT <= 64;
  static constexpr int kTermRows = NT / 2;                              // token rows that a block brings per term
  static constexpr int kBoxRows = kTermRows < 64 ? kTermRows : 64;
  static constexpr int kTermBytes = kTermRows * kTcKB * 2;
  static constexpr int kCols = kFused ? (NT == 16 ? 64 : 3 * NT) : NT;  // accumulator columns (not fused: at most)
  static constexpr int kCopyBytes = kTcWBytes + 3 * kTermBytes;
  static constexpr int kStageBytes = NT == 16 ? kTcWBytes + 4096 : kCopyBytes;  // 16 rows: room for the 32 rows that N = 64 reads
  static constexpr int kStages = NT == 16 ? 10 : (NT == 32 ? 9 : (NT == 64 ? 7 : (NT == 128 ? 5 : 3)));  // 192 - 200 KB
  static constexpr int kAccs = NT == 64 || NT == 256 ? 2 : 4;
  static constexpr int kAccStride = 512 / kAccs;                        // columns from one accumulator set to the next
  static constexpr int kHalf = NT / 2;                                  // tokens whose sums one epilogue thread holds
  static constexpr int kLd = kFused && NT == 16 ? 8 : 16;               // columns per tensor-memory load
  static constexpr size_t kSmem = (size_t)kStages * kStageBytes + 1024;
  static_assert(kStages <= kTcMaxStages && kAccs <= kTcMaxAccs && kCols <= kAccStride && kSmem <= 227 * 1024, "ring, accumulators and barriers fit");
};

template <int NT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kTcThreads, 1)
    spd_tc_product_kernel(const void *tmap_x, const void *tmap_w, float *Y, float *parts, const __grid_constant__ Product pr, int n_tok,
                          int x_term_rows, State *st, int stall) {
  using S = TcShape<NT>;
  extern __shared__ __align__(16) uint8_t tc_smem_raw[];
  uint8_t *smem = tc_smem_raw + ((1024u - (smem_u32(tc_smem_raw) & 1023u)) & 1023u);
  __shared__ TcShared sh;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)tc_cluster_rank(), pair = (int)(blockIdx.x >> 1);
  const int u0 = product_cut(pr, pair), u1 = product_cut(pr, pair + 1);  // this pair's run of stages
  const int tile_tok = pr.tile_tok;                                      // tokens of a tile
  dep_launch();
  if (threadIdx.x == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"(tmap_w) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"(tmap_x) : "memory");
    sh.dead = 0;
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(&sh.full[s], 1);
      mbar_init(&sh.empty[s], 1);
    }
    for (int a = 0; a < S::kAccs; ++a) {
      mbar_init(&sh.acc_full[a], 1);
      mbar_init(&sh.acc_empty[a], 16);  // one arrival per warp that reads the accumulator, eight in each block
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  if (warp == 1) tc_pair_alloc(&sh.tmem_base, 512);
  tc_fence_before();
  tc_cluster_sync();
  tc_fence_after();
  const uint32_t tmem = sh.tmem_base;
  const uint32_t ring = smem_u32(smem);

  if (warp == 0) {
    if (tc_elect()) {
      bool ok = true;
      int issued = 0;
      const int tile0 = u0 / pr.nk;
      int kb = u0 - tile0 * pr.nk, rt = tile0 / pr.tok_tiles, tt = tile0 - rt * pr.tok_tiles;
      auto next = [&]() {
        if (++kb == pr.nk) {
          kb = 0;
          if (++tt == pr.tok_tiles) { tt = 0; ++rt; }
        }
      };
      const uint32_t bar0 = tc_leader_addr(&sh.full[0]);
      const uint64_t policy = evict_first_policy();
      auto weights = [&](uint32_t stage) {
        const uint32_t base = ring + stage * (uint32_t)S::kStageBytes, bar = bar0 + stage * 8u;
        const int row = rt * (2 * kTcRows) + rank * kTcRows;
#pragma unroll
        for (int j = 0; j < kTcRows / kTcWBoxRows; ++j)
          tc_pair_box_load_policy(base + j * (kTcWBoxRows * kTcKB * 2), tmap_w, kb * kTcKB, row + j * kTcWBoxRows, bar, policy);
      };
      auto terms = [&](uint32_t stage) {
        const uint32_t base = ring + stage * (uint32_t)S::kStageBytes + kTcWBytes, bar = bar0 + stage * 8u;
        const int t0 = tt * tile_tok + rank * (tile_tok / 2);
#pragma unroll
        for (int j = 0; j < 3; ++j)
#pragma unroll
          for (int b = 0; b < S::kTermRows / S::kBoxRows; ++b)
            tc_pair_box_load(base + j * S::kTermBytes + b * (S::kBoxRows * kTcKB * 2), tmap_x, kb * kTcKB, j * x_term_rows + t0 + b * S::kBoxRows, bar);
      };
      // the first round of the ring: every stage is free; the weights go first, the terms once they are written
      const int first = min(u1 - u0, S::kStages);
      const int kb0 = kb, rt0 = rt, tt0 = tt;
      for (int i = 0; i < first; ++i, next()) {
        if (rank == 0) mbar_expect_tx(&sh.full[i], (uint32_t)(2 * S::kCopyBytes));
        if (!(stall && i == 0)) weights(i);
      }
      dep_wait();
      asm volatile("fence.proxy.async;" ::: "memory");  // the terms were written with ordinary stores
      kb = kb0; rt = rt0; tt = tt0;
      for (int i = 0; i < first; ++i, next())
        if (!(stall && i == 0)) terms(i);
      issued = first;
      uint32_t stage = 0, phase = 0;
      for (int u = u0 + first; u < u1; ++u, next()) {
        if (!tc_wait(sh, st, &sh.empty[stage], phase, 400)) { ok = false; break; }
        if (rank == 0) mbar_expect_tx(&sh.full[stage], (uint32_t)(2 * S::kCopyBytes));
        weights(stage);
        terms(stage);
        ++issued;
        if (++stage == (uint32_t)S::kStages) { stage = 0; phase ^= 1u; }
      }
      // No copy may land, and no instruction read a stage, after the blocks have gone, also when the issuing thread or the
      // epilogue gives up behind a producer that is done (a run no longer than the ring).  So before the cluster barrier
      // below the leader waits for the bytes of its last stages, its own and the other block's, which are counted on its
      // barriers; the other block waits until its last stages have been multiplied.  Both are over by themselves in a run
      // that succeeds (the epilogue waits as long) and bounded; a producer that gave up itself leaves 10 ms, for copies that
      // the leader never announced.
      const unsigned long long t = globaltimer(), limit = ok || rank == 0 ? kTcWaitNs : 10ull * 1000ull * 1000ull;
      for (int i = max(0, issued - S::kStages); i < issued; ++i) {
        if (stall && i == 0) continue;  // nothing was copied for it
        uint64_t *bar = rank == 0 ? &sh.full[i % S::kStages] : &sh.empty[i % S::kStages];
        while (!mbar_try_wait(bar, (uint32_t)(i / S::kStages) & 1u) && globaltimer() - t < limit) {}
      }
    }
    __syncwarp();
    tc_cluster_arrive_all();
  } else if (warp == 1) {
    if (rank == 0 && tc_elect()) {
      const uint32_t idesc = tc_idesc(2 * kTcRows, S::kFused ? S::kCols : tile_tok);
      uint32_t stage = 0, phase = 0;
      int seg = 0, in_seg = 0, kb = u0 % pr.nk;
      for (int u = u0; u < u1; ++u) {
        const int a = seg % S::kAccs;
        if (in_seg == 0 && !tc_wait(sh, st, &sh.acc_empty[a], (uint32_t)((seg / S::kAccs) & 1) ^ 1u, 430)) break;  // its last sum has been read
        if (!tc_wait(sh, st, &sh.full[stage], phase, 410)) break;
        tc_fence_after();
        const uint32_t base = ring + stage * (uint32_t)S::kStageBytes, acc = tmem + (uint32_t)(a * S::kAccStride);
        const uint32_t term0 = base + kTcWBytes + (!S::kFused && pr.small_first ? 2 * S::kTermBytes : 0);
        const int term_step = pr.small_first ? -S::kTermBytes : S::kTermBytes;
#pragma unroll
        for (int j = 0; j < (S::kFused ? 1 : 3); ++j)
#pragma unroll
          for (int kk = 0; kk < kTcKB / 16; ++kk)  // 16 columns = 32 bytes further into the swizzled rows
            tc_pair_mma(acc, tc_desc(base + kk * 32), tc_desc(term0 + j * term_step + kk * 32), idesc, (uint32_t)((in_seg | j | kk) != 0));
        tc_pair_commit(&sh.empty[stage]);  // the stage is free in both blocks once these have read it
        if (++stage == (uint32_t)S::kStages) { stage = 0; phase ^= 1u; }
        ++kb;
        if (++in_seg == pr.seg || kb == pr.nk || u + 1 == u1) {
          tc_pair_commit(&sh.acc_full[a]);  // the segment's sum is complete
          ++seg;
          in_seg = 0;
        }
        if (kb == pr.nk) kb = 0;
      }
    }
    __syncwarp();
    tc_fence_before();
    tc_cluster_arrive_all();
  } else {
    // Warp w may read lanes 32 (w % 4) .. 32 (w % 4) + 31 of tensor memory: a weight row per thread, a token per column;
    // warps 2..5 take the first half of the tile's tokens, 6..9 the second.
    const int quarter = warp & 3, half = (warp - 2) >> 2, half_tok = tile_tok / 2;
    const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
    int seg = 0;
    bool ok = true, left = false;
    dep_wait();  // Y and the pairs' buffers are written below (the kernel before this one may still be reading them)
    for (int u = u0; u < u1 && ok;) {
      const int tile = u / pr.nk, kb = u - tile * pr.nk, stages = min(pr.nk - kb, u1 - u);
      float sum[S::kHalf];
#pragma unroll
      for (int j = 0; j < S::kHalf; ++j) sum[j] = 0.f;
      for (int done = 0; done < stages; done += pr.seg, ++seg) {
        const int a = seg % S::kAccs;
        if (!tc_wait(sh, st, &sh.acc_full[a], (uint32_t)((seg / S::kAccs) & 1), 420)) { ok = false; break; }
        tc_fence_after();
        const uint32_t acc = lanes + (uint32_t)(a * S::kAccStride);
        if constexpr (S::kFused) {
          // a half's columns: its tokens' first terms, second terms, third terms; the small ones are added first (one load
          // in flight: with three of 16 columns 64 tokens took 4.29 ms instead of 4.15)
          const uint32_t from = acc + (uint32_t)(half * (S::kCols / 2));
#pragma unroll
          for (int c0 = 3 * S::kHalf - S::kLd; c0 >= 0; c0 -= S::kLd) {
            uint32_t r[S::kLd];
            tc_ld(from + (uint32_t)c0, r);
            tc_ld_wait();
#pragma unroll
            for (int j = 0; j < S::kLd; ++j) sum[(c0 + j) % S::kHalf] += __uint_as_float(r[j]);
          }
        } else {
          const uint32_t from = acc + (uint32_t)(half * half_tok);
#pragma unroll
          for (int c0 = 0; c0 < S::kHalf; c0 += 32)
            if (c0 < half_tok) {  // (a multiple of 8: the last load may bring columns behind the half, whose sums go nowhere)
              uint32_t r[16], q[16];
              tc_ld(from + (uint32_t)c0, r);
              if (c0 + 16 < half_tok) tc_ld(from + (uint32_t)(c0 + 16), q);
              tc_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) sum[c0 + j] += __uint_as_float(r[j]);
              if (c0 + 16 < half_tok) {
#pragma unroll
                for (int j = 0; j < 16; ++j) sum[c0 + 16 + j] += __uint_as_float(q[j]);
              }
            }
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) tc_cluster_arrive(tc_leader_addr(&sh.acc_empty[a]));
      }
      // The last sums are in registers: the tensor memory may go while they are stored.  Up to 32 token rows, where a product's end is
      // felt (spd_prefill of 15 tokens, 7B shape, 3.009 -> 2.968 ms, 27 3.055 -> 3.022, three timesteps of 8 requests 9.17 -> 9.08;
      // 100 tokens 5.02 -> 5.04, 64 requests 14.66 -> 14.76).
      if (NT <= 32 && u + stages == u1) {
        tc_fence_before();
        tc_cluster_arrive_all();
        left = true;
      }
      const int in_tile = rank * kTcRows + quarter * 32 + lane, row = tile / pr.tok_tiles * (2 * kTcRows) + in_tile;
      const int t_lo = half * half_tok, t0 = tile % pr.tok_tiles * tile_tok + t_lo;  // first token of this half in the tile, overall
      if (ok && row < pr.N) {
        // the lanes of a warp write 32 consecutive floats of a token's row
        float *out = kb == 0 ? Y + (size_t)t0 * pr.N + row : parts + ((size_t)pair * tile_tok + t_lo) * (2 * kTcRows) + in_tile;
        const size_t step = kb == 0 ? (size_t)pr.N : (size_t)(2 * kTcRows);
#pragma unroll
        for (int j = 0; j < S::kHalf; ++j)
          if (j < half_tok && t0 + j < n_tok) out[j * step] = sum[j];
      }
      u += stages;
    }
    if (!left) {
      tc_fence_before();
      tc_cluster_arrive_all();
    }
  }
  // neither block leaves while the other may still signal or read its shared memory
  tc_cluster_wait_all();
  if (warp == 1) {
    tc_fence_after();
    tc_pair_dealloc(tmem, 512);
  }
}

// ---------------------------------------------------------------- attention of a job
// The three bf16 terms of v (v = hi + mid + lo exactly: each takes the leading 8 significant bits of what is left, by truncation), each in the upper half of a word.
__device__ __forceinline__ void tc_split3(float v, uint32_t &hi, uint32_t &mid, uint32_t &lo) {
  hi = __float_as_uint(v) & 0xffff0000u;
  const float r1 = v - __uint_as_float(hi);
  mid = __float_as_uint(r1) & 0xffff0000u;
  lo = __float_as_uint(r1 - __uint_as_float(mid)) & 0xffff0000u;
}
// Two neighbouring values of the output as terms.
__device__ __forceinline__ void tc_put_pair(uint16_t *dst, size_t term_stride, float a, float b) {
  uint32_t h0, m0, l0, h1, m1, l1;
  tc_split3(a, h0, m0, l0);
  tc_split3(b, h1, m1, l1);
  *reinterpret_cast<uint32_t *>(dst) = h1 | (h0 >> 16);
  *reinterpret_cast<uint32_t *>(dst + term_stride) = m1 | (m0 >> 16);
  *reinterpret_cast<uint32_t *>(dst + 2 * term_stride) = l1 | (l0 >> 16);
}

// Causal attention over a float32 cache (a bf16 cache takes spd_tc_attn_mma_kernel below): 16 consecutive tokens
// of one head.  The block brings 32 cached positions at
// a time into shared memory as float32 (keys with padded rows, so that a lane per position reads its row without
// bank conflicts); a warp owns two tokens: scores with a lane per position, the tile's softmax weights by warp
// reductions (online softmax across tiles), weighted value sums with HD / 32 dimensions per lane and the weights
// passed round by shuffles.  Every cache row is read once per 16 tokens.  Output as three bf16 terms.
// What bounds it: for few tokens the trips to L2 before the first score, which are made side by side (15 tokens, 7B shape, 9.4 -> 5.2
// us a layer, 64 tokens of 13B 17.0 -> 12.9), for many the score and value loops, behind which the next tile travels (spd_prefill
// of 200 tokens 10.1 -> 8.6 ms, 500 23.3 -> 22.1).
template <int HD>
__global__ void __launch_bounds__(256) spd_tc_attn_kernel(const float *Q, const float *kcache, const float *vcache, uint16_t *X,
                                                          size_t term_stride, int d, int max_pos, int layer, int pos0, int n_tok) {
  dep_launch();
  dep_wait();
  constexpr int kTok = 16, kPos = 32;
  constexpr int KS = HD + 4;    // key row stride in floats: 16-byte aligned, rows 4 banks apart
  constexpr int DPL = HD / 32;  // value dimensions per lane
  __shared__ __align__(16) float sq[kTok * HD];
  __shared__ __align__(16) float sk[kPos * KS];
  __shared__ __align__(16) float sv[kPos * HD];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, tid = threadIdx.x;
  const int head = blockIdx.y, t0 = blockIdx.x * kTok;
  const float scale = 1.f / sqrtf((float)HD);
  const int last_pos = pos0 + min(t0 + kTok - 1, n_tok - 1);  // the last position a token of this block sees
  // A tile's rows on their way through registers: the first tile's are asked for before the queries, a later one's while the tile
  // before it is used (a trip to L2 each, which the block otherwise spends idle).
  constexpr int kMine = kPos * HD / 4 / 256;  // 16-byte vectors of keys that a thread brings, and of values
  float4 kf[kMine], vf[kMine];
  auto ask = [&](int tile0) {
#pragma unroll
    for (int u = 0; u < kMine; ++u) {
      const int i = tid + u * 256, r = i / (HD / 4), c4 = i - r * (HD / 4), pos = tile0 + r;
      const size_t at = ((size_t)layer * max_pos + min(pos, last_pos)) * d + head * HD + c4 * 4;
      kf[u] = *reinterpret_cast<const float4 *>(kcache + at);
      vf[u] = *reinterpret_cast<const float4 *>(vcache + at);
      if (pos > last_pos) kf[u] = vf[u] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
  };
  ask(0);
#pragma unroll
  for (int u = 0; u < kTok * HD / 4 / 256; ++u) {
    const int i = tid + u * 256, tt = i / (HD / 4), c = (i - tt * (HD / 4)) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t0 + tt < n_tok) v = *reinterpret_cast<const float4 *>(Q + (size_t)(t0 + tt) * d + head * HD + c);
    *reinterpret_cast<float4 *>(sq + tt * HD + c) = make_float4(v.x * scale, v.y * scale, v.z * scale, v.w * scale);
  }
  const int ta = t0 + 2 * warp, tb = ta + 1;
  const int pa = pos0 + ta, pb = pos0 + tb;
  float ma = -CUDART_INF_F, mb = -CUDART_INF_F, la = 0.f, lb = 0.f;
  float acca[DPL], accb[DPL];
#pragma unroll
  for (int e = 0; e < DPL; ++e) acca[e] = accb[e] = 0.f;
  for (int tile0 = 0; tile0 <= last_pos; tile0 += kPos) {
    __syncthreads();  // the previous tile has been used (first round: nothing)
#pragma unroll
    for (int u = 0; u < kMine; ++u) {
      const int i = tid + u * 256, r = i / (HD / 4), c4 = i - r * (HD / 4);
      *reinterpret_cast<float4 *>(sk + r * KS + c4 * 4) = kf[u];
      *reinterpret_cast<float4 *>(sv + r * HD + c4 * 4) = vf[u];
    }
    __syncthreads();
    if (tile0 + kPos <= last_pos) ask(tile0 + kPos);
    // scores of position tile0 + lane for the warp's two tokens
    float sa = 0.f, sb = 0.f;
    {
      const float4 *kr = reinterpret_cast<const float4 *>(sk + lane * KS);
      const float4 *qa = reinterpret_cast<const float4 *>(sq + (2 * warp) * HD), *qb = qa + HD / 4;
#pragma unroll 8
      for (int c = 0; c < HD / 4; ++c) {
        const float4 k4 = kr[c], a4 = qa[c], b4 = qb[c];
        sa = fmaf(a4.x, k4.x, sa); sa = fmaf(a4.y, k4.y, sa); sa = fmaf(a4.z, k4.z, sa); sa = fmaf(a4.w, k4.w, sa);
        sb = fmaf(b4.x, k4.x, sb); sb = fmaf(b4.y, k4.y, sb); sb = fmaf(b4.z, k4.z, sb); sb = fmaf(b4.w, k4.w, sb);
      }
    }
    const int pos = tile0 + lane;
    sa = pos <= pa ? sa : -CUDART_INF_F;
    sb = pos <= pb ? sb : -CUDART_INF_F;
    float xa = sa, xb = sb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      xa = fmaxf(xa, __shfl_xor_sync(0xffffffffu, xa, o));
      xb = fmaxf(xb, __shfl_xor_sync(0xffffffffu, xb, o));
    }
    // position 0 is visible to every token, so the running maxima are finite from the first tile on
    const float mna = fmaxf(ma, xa), mnb = fmaxf(mb, xb);
    const float ca = __expf(ma - mna), cb = __expf(mb - mnb);
    const float wa = __expf(sa - mna), wb = __expf(sb - mnb);
    float ua = wa, ub = wb;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      ua += __shfl_xor_sync(0xffffffffu, ua, o);
      ub += __shfl_xor_sync(0xffffffffu, ub, o);
    }
    la = fmaf(la, ca, ua);
    lb = fmaf(lb, cb, ub);
    ma = mna;
    mb = mnb;
#pragma unroll
    for (int e = 0; e < DPL; ++e) {
      acca[e] *= ca;
      accb[e] *= cb;
    }
    const int used = min(kPos, last_pos + 1 - tile0);  // positions behind the last have no weight
#pragma unroll 8
    for (int j = 0; j < used; ++j) {
      const float ja = __shfl_sync(0xffffffffu, wa, j), jb = __shfl_sync(0xffffffffu, wb, j);
      const float *vr = sv + j * HD + lane * DPL;
      float v[DPL];
      if (DPL == 4) {
        const float4 v4 = *reinterpret_cast<const float4 *>(vr);
        v[0] = v4.x; v[1] = v4.y; v[DPL - 2] = v4.z; v[DPL - 1] = v4.w;
      } else {
        const float2 v2 = *reinterpret_cast<const float2 *>(vr);
        v[0] = v2.x; v[1] = v2.y;
      }
#pragma unroll
      for (int e = 0; e < DPL; ++e) {
        acca[e] = fmaf(ja, v[e], acca[e]);
        accb[e] = fmaf(jb, v[e], accb[e]);
      }
    }
  }
  const float ia = 1.f / la, ib = 1.f / lb;
  uint16_t *out = X + (size_t)ta * d + head * HD + lane * DPL;
#pragma unroll
  for (int e = 0; e < DPL; e += 2) {
    if (ta < n_tok) tc_put_pair(out + e, term_stride, acca[e] * ia, acca[e + 1] * ia);
    if (tb < n_tok) tc_put_pair(out + d + e, term_stride, accb[e] * ib, accb[e + 1] * ib);
  }
}

// ---------------------------------------------------------------- attention over a bf16 cache on tensor cores
__device__ __forceinline__ void tc_mma_sync(float (&c)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void tc_ldsm_x4(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(addr));
}
__device__ __forceinline__ void tc_ldsm_x4_trans(uint32_t addr, uint32_t (&r)[4]) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr));
}

__device__ __forceinline__ void tc_cp16(uint32_t dst, const void *src, uint32_t bytes) {  // 16 bytes, zeros past `bytes` (0 or 16)
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

// Four scaled values as terms, 8 bytes of each.
__device__ __forceinline__ void tc_put_terms(uint8_t *dst, int term_step, const float4 &v, float scale) {
  uint32_t h[4], m[4], l[4];
  tc_split3(v.x * scale, h[0], m[0], l[0]);
  tc_split3(v.y * scale, h[1], m[1], l[1]);
  tc_split3(v.z * scale, h[2], m[2], l[2]);
  tc_split3(v.w * scale, h[3], m[3], l[3]);
  *reinterpret_cast<uint2 *>(dst) = make_uint2(h[1] | (h[0] >> 16), h[3] | (h[2] >> 16));
  *reinterpret_cast<uint2 *>(dst + term_step) = make_uint2(m[1] | (m[0] >> 16), m[3] | (m[2] >> 16));
  *reinterpret_cast<uint2 *>(dst + 2 * term_step) = make_uint2(l[1] | (l[0] >> 16), l[3] | (l[2] >> 16));
}
// The softmax weights of 16 positions (two score fragments) as terms, repacked as a left operand; their sums join l.
__device__ __forceinline__ void tc_weight_terms(const float (&sa)[4], const float (&sb)[4], const float (&m)[2], float (&l)[2], uint32_t (&pt)[3][4]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float pw[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) pw[e] = __expf((h ? sb : sa)[e] - m[e >> 1]);
    l[0] += pw[0] + pw[1];
    l[1] += pw[2] + pw[3];
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      uint32_t h0, m0, l0, h1, m1, l1;
      tc_split3(pw[2 * r], h0, m0, l0);
      tc_split3(pw[2 * r + 1], h1, m1, l1);
      pt[0][h * 2 + r] = h1 | (h0 >> 16);
      pt[1][h * 2 + r] = m1 | (m0 >> 16);
      pt[2][h * 2 + r] = l1 | (l0 >> 16);
    }
  }
}

// Causal attention of 16 x WARPS consecutive tokens of one head over a bf16 cache, on tensor cores (mma.sync m16n8k16:
// the attention's share of the arithmetic is small, so the warp-level instructions serve).  Keys and values
// are bf16 already and therefore exact operands; the scaled queries and the softmax weights are float32 and go
// in as three bf16 terms each, as the activations of the products do.  A warp owns 16 tokens: scores of a tile of
// 64 cached positions (tokens x positions), online softmax on the accumulator fragments, the weights' terms repacked in
// registers as the next product's left operand, values through transposing matrix loads.  Rows of every shared-memory
// tile are 16 bytes longer than their data: eight consecutive rows then start in different bank groups.
// What bounds it: the 384 instructions of a tile and warp; so the next tile's rows travel (cp.async, two buffers) while
// a tile is multiplied, consecutive instructions go to different accumulators, and tiles wholly behind a warp's tokens
// skip the mask.  One block per SM: eight warps when 64-token blocks would outnumber the SMs, else four.
// spd_prefill of 400 / 2048 tokens, 7B shape, 0.6 / 2.5 ms shorter than with one tile buffer, two blocks of four warps per SM
// and three dependent instructions in a row; a job of 512 tokens at position 0 takes 49 us a layer (ncu).
template <int HD, int WARPS>
__global__ void __launch_bounds__(WARPS * 32, 1)
    spd_tc_attn_mma_kernel(const float *Q, const uint16_t *kcache, const uint16_t *vcache, uint16_t *X, size_t term_stride, int d, int max_pos,
                           int layer, int pos0, int n_tok) {
  dep_launch();
  dep_wait();
  constexpr int kTok = 16 * WARPS, kPos = 64, kThr = WARPS * 32;
  constexpr int RS = HD * 2 + 16;  // bytes per tile row
  constexpr int KS = HD / 16;      // k-steps over the head's dimensions
  constexpr int DT = HD / 8;       // output tiles of 8 dimensions
  constexpr int kBuf = 2 * kPos * RS;
  extern __shared__ __align__(16) uint8_t at_smem[];
  const uint32_t sq_u = smem_u32(at_smem);            // [3 terms][tokens][RS]
  const uint32_t kv_u = sq_u + 3 * kTok * RS;         // two buffers of [64 positions][RS] keys, then values
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
  const int head = blockIdx.y, t0 = blockIdx.x * kTok;
  const int last_pos = pos0 + min(t0 + kTok - 1, n_tok - 1);  // the last position a token of this block sees
  auto fetch = [&](int tile0, int buf) {
    const uint32_t dst = kv_u + (uint32_t)(buf * kBuf);
    for (int i = tid; i < kPos * HD / 8; i += kThr) {
      const int r = i / (HD / 8), c8 = i - r * (HD / 8), pos = tile0 + r;
      const size_t at = ((size_t)layer * max_pos + min(pos, last_pos)) * d + head * HD + c8 * 8;
      const uint32_t bytes = pos <= last_pos ? 16u : 0u, off = (uint32_t)(r * RS + c8 * 16);
      tc_cp16(dst + off, kcache + at, bytes);
      tc_cp16(dst + kPos * RS + off, vcache + at, bytes);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0, 0);
  const float scale = 1.f / sqrtf((float)HD);
  for (int i = tid; i < kTok * HD / 4; i += kThr) {
    const int tt = i / (HD / 4), c = (i - tt * (HD / 4)) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t0 + tt < n_tok) v = *reinterpret_cast<const float4 *>(Q + (size_t)(t0 + tt) * d + head * HD + c);
    tc_put_terms(at_smem + tt * RS + c * 2, kTok * RS, v, scale);
  }
  const int tw = t0 + warp * 16;
  const int p_first = pos0 + tw, p_lo = p_first + g, p_hi = p_lo + 8, warp_last = p_first + 15;
  float m[2] = {-CUDART_INF_F, -CUDART_INF_F}, l[2] = {0.f, 0.f};
  float o[DT][4];
#pragma unroll
  for (int i = 0; i < DT; ++i) o[i][0] = o[i][1] = o[i][2] = o[i][3] = 0.f;
  // per-lane offsets: left operand (tokens x dimensions), keys (two tiles of 8 positions x 16 dimensions), values (transposed)
  const uint32_t a_off = sq_u + (uint32_t)((warp * 16 + (lane & 7) + ((lane >> 3) & 1) * 8) * RS + (lane >> 4) * 16);
  const uint32_t k_off = (uint32_t)(((lane >> 4) * 8 + (lane & 7)) * RS + ((lane >> 3) & 1) * 16);
  const uint32_t v_off = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * RS + (lane >> 4) * 16 + kPos * RS);
  int buf = 0;
  for (int tile0 = 0; tile0 <= last_pos; tile0 += kPos, buf ^= 1) {
    if (tile0 + kPos <= last_pos) {
      fetch(tile0 + kPos, buf ^ 1);  // (every warp has left that buffer: the barrier at the end of the round)
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();  // the tile (first round: and the queries) is in place for all
    if (tile0 <= warp_last) {  // else nothing of this tile is visible to the warp's tokens
      const uint32_t sk_u = kv_u + (uint32_t)(buf * kBuf);
      float s[kPos / 8][4];
#pragma unroll
      for (int i = 0; i < kPos / 8; ++i) s[i][0] = s[i][1] = s[i][2] = s[i][3] = 0.f;
#pragma unroll
      for (int ks = 0; ks < KS; ++ks) {
        uint32_t kb[kPos / 16][4];
#pragma unroll
        for (int np = 0; np < kPos / 16; ++np) tc_ldsm_x4(sk_u + k_off + (uint32_t)(np * 16 * RS + ks * 32), kb[np]);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          uint32_t a[4];
          tc_ldsm_x4(a_off + (uint32_t)(j * kTok * RS + ks * 32), a);
#pragma unroll
          for (int np = 0; np < kPos / 16; ++np) {
            tc_mma_sync(s[2 * np], a, kb[np][0], kb[np][1]);
            tc_mma_sync(s[2 * np + 1], a, kb[np][2], kb[np][3]);
          }
        }
      }
      // causal mask, row maxima (rows g and g + 8 of the warp's 16 tokens; a row lives in the four lanes of a quad)
      if (tile0 + kPos - 1 > p_first) {
#pragma unroll
        for (int nt = 0; nt < kPos / 8; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) {
            const int pos = tile0 + nt * 8 + 2 * q + (e & 1);
            if (pos > (e < 2 ? p_lo : p_hi)) s[nt][e] = -CUDART_INF_F;
          }
      }
      float mx[2] = {-CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
      for (int nt = 0; nt < kPos / 8; ++nt)
#pragma unroll
        for (int e = 0; e < 4; ++e) mx[e >> 1] = fmaxf(mx[e >> 1], s[nt][e]);
      float c[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
        const float mn = fmaxf(m[r], mx[r]);  // finite: position 0 is visible to every token in the first tile
        c[r] = __expf(m[r] - mn);
        m[r] = mn;
        l[r] *= c[r];
      }
#pragma unroll
      for (int i = 0; i < DT; ++i) {
        o[i][0] *= c[0]; o[i][1] *= c[0]; o[i][2] *= c[1]; o[i][3] *= c[1];
      }
      // per 16 positions: the weights and their terms, repacked as the left operand, times the values
#pragma unroll
      for (int kk = 0; kk < kPos / 16; ++kk) {
        uint32_t pt[3][4];
        tc_weight_terms(s[2 * kk], s[2 * kk + 1], m, l, pt);
#pragma unroll
        for (int dq = 0; dq < DT / 2; dq += 4) {
          uint32_t vb[4][4];
#pragma unroll
          for (int i = 0; i < 4; ++i) tc_ldsm_x4_trans(sk_u + v_off + (uint32_t)(kk * 16 * RS + (dq + i) * 32), vb[i]);
#pragma unroll
          for (int j = 0; j < 3; ++j)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              tc_mma_sync(o[2 * (dq + i)], pt[j], vb[i][0], vb[i][1]);
              tc_mma_sync(o[2 * (dq + i) + 1], pt[j], vb[i][2], vb[i][3]);
            }
        }
      }
    }
    __syncthreads();  // the tile's buffer may be filled again
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
  }
  const float inv[2] = {1.f / l[0], 1.f / l[1]};
#pragma unroll
  for (int i = 0; i < DT; ++i)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int t = tw + g + r * 8;
      if (t < n_tok) {
        tc_put_pair(X + (size_t)t * d + head * HD + i * 8 + 2 * q, term_stride, o[i][2 * r] * inv[r], o[i][2 * r + 1] * inv[r]);
      }
    }
}

// The same for few tokens: 16 tokens of one head, the eight warps sharing them.  With a warp per 16 tokens a short job keeps one to
// four warps of a few SMs busy with 384 instructions a tile; here a warp takes 8 of a tile's 64 positions (the scores meet in shared
// memory), then, with all warps repeating the softmax of the 16 tokens for themselves, 16 of the head's dimensions of the weighted
// values.  Every score and every sum is made of the same instructions in the same order, so the results are that kernel's bit for bit.
// What bounds it is latency: 24 dependent instructions for the scores, 12 for the values, two barriers a tile.  A job of 27 tokens,
// 7B shape, 9.6 -> 5.3 us of the layer's 99; 16 tokens behind 384 positions 27.5 -> 21; 100 tokens 13.9 -> 10.5.
template <int HD>
__global__ void __launch_bounds__(256, 2)
    spd_tc_attn_few_kernel(const float *Q, const uint16_t *kcache, const uint16_t *vcache, uint16_t *X, size_t term_stride, int d, int max_pos,
                           int layer, int pos0, int n_tok) {
  dep_launch();
  dep_wait();
  constexpr int kTok = 16, kPos = 64, kThr = 256;
  constexpr int RS = HD * 2 + 16, KS = HD / 16;
  constexpr int kBuf = 2 * kPos * RS;
  extern __shared__ __align__(16) uint8_t at_smem[];
  const uint32_t sq_u = smem_u32(at_smem);            // [3 terms][tokens][RS]
  const uint32_t kv_u = sq_u + 3 * kTok * RS;         // two buffers of [64 positions][RS] keys, then values
  float4 *sc = reinterpret_cast<float4 *>(at_smem + 3 * kTok * RS + 2 * kBuf);  // two buffers of [8 positions' scores][lane]
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, g = lane >> 2, q = lane & 3;
  const int head = blockIdx.y, t0 = blockIdx.x * kTok;
  const int last_pos = pos0 + min(t0 + kTok - 1, n_tok - 1);
  auto fetch = [&](int tile0, int buf) {
    const uint32_t dst = kv_u + (uint32_t)(buf * kBuf);
    for (int i = tid; i < kPos * HD / 8; i += kThr) {
      const int r = i / (HD / 8), c8 = i - r * (HD / 8), pos = tile0 + r;
      const size_t at = ((size_t)layer * max_pos + min(pos, last_pos)) * d + head * HD + c8 * 8;
      const uint32_t bytes = pos <= last_pos ? 16u : 0u, off = (uint32_t)(r * RS + c8 * 16);
      tc_cp16(dst + off, kcache + at, bytes);
      tc_cp16(dst + kPos * RS + off, vcache + at, bytes);
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  fetch(0, 0);
  const float scale = 1.f / sqrtf((float)HD);
  for (int i = tid; i < kTok * HD / 4; i += kThr) {
    const int tt = i / (HD / 4), c = (i - tt * (HD / 4)) * 4;
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (t0 + tt < n_tok) v = *reinterpret_cast<const float4 *>(Q + (size_t)(t0 + tt) * d + head * HD + c);
    tc_put_terms(at_smem + tt * RS + c * 2, kTok * RS, v, scale);
  }
  const int p_first = pos0 + t0, p_lo = p_first + g, p_hi = p_lo + 8;
  float m[2] = {-CUDART_INF_F, -CUDART_INF_F}, l[2] = {0.f, 0.f};
  float o[2][4] = {};
  const uint32_t a_off = sq_u + (uint32_t)(((lane & 7) + ((lane >> 3) & 1) * 8) * RS + (lane >> 4) * 16);
  const uint32_t k_off = (uint32_t)((warp * 8 + (lane & 7)) * RS + (lane >> 3) * 16);  // 8 positions x 32 dimensions
  const uint32_t v_off = (uint32_t)((((lane >> 3) & 1) * 8 + (lane & 7)) * RS + (lane >> 4) * 16 + kPos * RS + warp * 32);
  int buf = 0;
  for (int tile0 = 0; tile0 <= last_pos; tile0 += kPos, buf ^= 1) {
    asm volatile("cp.async.wait_group 0;" ::: "memory");
    __syncthreads();  // the tile (first round: and the queries) is in place for all, the other buffer has been used
    if (tile0 + kPos <= last_pos) fetch(tile0 + kPos, buf ^ 1);
    const uint32_t sk_u = kv_u + (uint32_t)(buf * kBuf);
    {
      float s[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int ks = 0; ks < KS; ks += 2) {
        uint32_t kb[4];
        tc_ldsm_x4(sk_u + k_off + (uint32_t)(ks * 32), kb);
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            uint32_t a[4];
            tc_ldsm_x4(a_off + (uint32_t)(j * kTok * RS + (ks + h) * 32), a);
            tc_mma_sync(s, a, kb[2 * h], kb[2 * h + 1]);
          }
      }
      sc[(buf * 8 + warp) * 32 + lane] = make_float4(s[0], s[1], s[2], s[3]);
    }
    __syncthreads();
    if (warp * 16 < HD) {
      float s[kPos / 8][4];
      float mx[2] = {-CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
      for (int nt = 0; nt < kPos / 8; ++nt) {
        const float4 v = sc[(buf * 8 + nt) * 32 + lane];
        s[nt][0] = v.x; s[nt][1] = v.y; s[nt][2] = v.z; s[nt][3] = v.w;
        const int pos = tile0 + nt * 8 + 2 * q;
        if (pos > p_lo) s[nt][0] = -CUDART_INF_F;
        if (pos + 1 > p_lo) s[nt][1] = -CUDART_INF_F;
        if (pos > p_hi) s[nt][2] = -CUDART_INF_F;
        if (pos + 1 > p_hi) s[nt][3] = -CUDART_INF_F;
#pragma unroll
        for (int e = 0; e < 4; ++e) mx[e >> 1] = fmaxf(mx[e >> 1], s[nt][e]);
      }
      float c[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 1));
        mx[r] = fmaxf(mx[r], __shfl_xor_sync(0xffffffffu, mx[r], 2));
        const float mn = fmaxf(m[r], mx[r]);
        c[r] = __expf(m[r] - mn);
        m[r] = mn;
        l[r] *= c[r];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        o[i][0] *= c[0]; o[i][1] *= c[0]; o[i][2] *= c[1]; o[i][3] *= c[1];
      }
#pragma unroll
      for (int kk = 0; kk < kPos / 16; ++kk) {
        uint32_t pt[3][4], vb[4];
        tc_weight_terms(s[2 * kk], s[2 * kk + 1], m, l, pt);
        tc_ldsm_x4_trans(sk_u + v_off + (uint32_t)(kk * 16 * RS), vb);
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          tc_mma_sync(o[0], pt[j], vb[0], vb[1]);
          tc_mma_sync(o[1], pt[j], vb[2], vb[3]);
        }
      }
    }
  }
  if (warp * 16 >= HD) return;
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 1);
    l[r] += __shfl_xor_sync(0xffffffffu, l[r], 2);
  }
  const float inv[2] = {1.f / l[0], 1.f / l[1]};
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int t = t0 + g + r * 8;
      if (t < n_tok) tc_put_pair(X + (size_t)t * d + head * HD + (2 * warp + i) * 8 + 2 * q, term_stride, o[i][2 * r] * inv[r], o[i][2 * r + 1] * inv[r]);
    }
}

}  // namespace spd

namespace {

template <int HD>
constexpr size_t attn_few_smem() { return (size_t)(3 * 16 + 4 * 64) * (HD * 2 + 16) + 2 * 8 * 32 * 16; }  // query terms, keys and values, scores

template <int HD, int WARPS>
constexpr size_t attn_mma_smem() { return (size_t)(3 * 16 * WARPS + 4 * 64) * (HD * 2 + 16); }  // query terms; two buffers of keys and values

template <int HD, int WARPS>
cudaError_t launch_attn_mma(const spd::TcJob &j, int layer, int n_tok, cudaStream_t s) {
  return spd::launch_dep(spd::spd_tc_attn_mma_kernel<HD, WARPS>, dim3((n_tok + 16 * WARPS - 1) / (16 * WARPS), j.H), dim3(WARPS * 32),
                         attn_mma_smem<HD, WARPS>(), s, j.q, static_cast<const uint16_t *>(j.kcache), static_cast<const uint16_t *>(j.vcache), j.x,
                         (size_t)j.x_term_rows * j.d, j.d, j.max_pos, layer, j.pos0, n_tok);
}

template <int HD>
cudaError_t launch_attn(const spd::TcJob &j, int layer, int n_tok, cudaStream_t s) {
  // Up to 128 tokens a block's warps share 16 of them; beyond, where blocks of 64 tokens keep the SMs as busy and read the cache less
  // often, a warp has 16 (7B shape, spd_prefill, shared / apart: 15 tokens 3.06 / 3.15 ms, 27 3.12 / 3.27, 64 3.46 / 3.66, 100 4.48 /
  // 4.53, 128 4.87 / 4.95; 200 7.53 / 7.45, 300 12.50 / 12.44).
  if (j.kv_bf16 && n_tok <= spd::kTcTile)
    return spd::launch_dep(spd::spd_tc_attn_few_kernel<HD>, dim3((n_tok + 15) / 16, j.H), dim3(256), attn_few_smem<HD>(), s, j.q,
                           static_cast<const uint16_t *>(j.kcache), static_cast<const uint16_t *>(j.vcache), j.x, (size_t)j.x_term_rows * j.d, j.d,
                           j.max_pos, layer, j.pos0, n_tok);
  if (j.kv_bf16) return (n_tok + 63) / 64 * j.H > j.sm_count ? launch_attn_mma<HD, 8>(j, layer, n_tok, s) : launch_attn_mma<HD, 4>(j, layer, n_tok, s);
  return spd::launch_dep(spd::spd_tc_attn_kernel<HD>, dim3((n_tok + 15) / 16, j.H), dim3(256), 0, s, j.q, static_cast<const float *>(j.kcache),
                         static_cast<const float *>(j.vcache), j.x, (size_t)j.x_term_rows * j.d, j.d, j.max_pos, layer, j.pos0, n_tok);
}

template <int HD>
cudaError_t allow_attn_few_smem() {
  return cudaFuncSetAttribute(reinterpret_cast<const void *>(&spd::spd_tc_attn_few_kernel<HD>), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)attn_few_smem<HD>());
}

template <int HD, int WARPS>
cudaError_t allow_attn_smem() {
  return cudaFuncSetAttribute(reinterpret_cast<const void *>(&spd::spd_tc_attn_mma_kernel<HD, WARPS>), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)attn_mma_smem<HD, WARPS>());
}

template <int NT>
cudaError_t launch_product(const spd::TcJob &j, int wide, const void *wmap, float *Y, const spd::Product &pr, int n_tok, cudaStream_t s, int stall) {
  using S = spd::TcShape<NT>;
  // the term buffer's tensor maps, two each (d_model and d_ffn columns): boxes of 8, 16, 32 and 64 rows
  const int slot = (S::kBoxRows == 8 ? 0 : (S::kBoxRows == 16 ? 1 : (S::kBoxRows == 32 ? 2 : 3))) * 2 + (wide ? 1 : 0);
  return spd::launch_dep(spd::spd_tc_product_kernel<NT>, dim3(2 * pr.pairs), dim3(spd::kTcThreads), S::kSmem, s,
                         j.x_tmaps + (size_t)slot * spd::kTensorMapBytes, wmap, Y, j.parts, pr, n_tok, j.x_term_rows, j.st, stall);
}

template <int NT>
cudaError_t allow_product_smem() {
  return cudaFuncSetAttribute(reinterpret_cast<const void *>(&spd::spd_tc_product_kernel<NT>), cudaFuncAttributeMaxDynamicSharedMemorySize,
                              (int)spd::TcShape<NT>::kSmem);
}

}  // namespace

extern "C" cudaError_t spd_internal_tc_prepare(void) {
  cudaError_t e = allow_product_smem<16>();
  if (e == cudaSuccess) e = allow_product_smem<32>();
  if (e == cudaSuccess) e = allow_product_smem<64>();
  if (e == cudaSuccess) e = allow_product_smem<128>();
  if (e == cudaSuccess) e = allow_product_smem<256>();
  if (e == cudaSuccess) e = allow_attn_smem<64, 4>();
  if (e == cudaSuccess) e = allow_attn_smem<64, 8>();
  if (e == cudaSuccess) e = allow_attn_smem<128, 4>();
  if (e == cudaSuccess) e = allow_attn_smem<128, 8>();
  if (e == cudaSuccess) e = allow_attn_few_smem<64>();
  if (e == cudaSuccess) e = allow_attn_few_smem<128>();
  return e;
}

// Product of n_tok token rows (<= x_term_rows) with matrix `which` of the layers' tensor maps: `wide` terms have d_ffn
// columns, else d_model.  *out tells the readers of Y where its sums are (product_sum4).
extern "C" cudaError_t spd_internal_product(const spd::TcJob *job, int n_tok, int wide, int which, float *Y, int N, spd::Product *out, cudaStream_t s) {
  const spd::TcJob &j = *job;
  const void *wmap = j.w_tmaps + (size_t)which * spd::kTensorMapBytes;
  const spd::Product pr = spd::plan_product(n_tok, N, wide ? j.f : j.d, j.sm_count, Y, j.parts);
  *out = pr;
  switch (pr.shape) {
    case 16: return launch_product<16>(j, wide, wmap, Y, pr, n_tok, s, 0);
    case 32: return launch_product<32>(j, wide, wmap, Y, pr, n_tok, s, 0);
    case 64: return launch_product<64>(j, wide, wmap, Y, pr, n_tok, s, 0);
    case 128: return launch_product<128>(j, wide, wmap, Y, pr, n_tok, s, 0);
    default: return launch_product<256>(j, wide, wmap, Y, pr, n_tok, s, 0);
  }
}

// Test hook: one pair whose first stage never arrives (see the kernel's `stall`), on the first layer's QKV product or, `few`,
// on four stages of it at most (256 rows, 256 columns).
extern "C" cudaError_t spd_internal_tc_stall(const spd::TcJob *job, int few, cudaStream_t s) {
  const spd::TcJob &j = *job;
  const spd::Product pr = spd::plan_product(1, few ? 256 : 3 * j.d, few && j.d > 256 ? 256 : j.d, 2, j.y, j.parts);
  return launch_product<16>(j, 0, j.w_tmaps, j.y, pr, 1, s, 1);
}

// Enqueues the decoder over j.n_tok tokens (at most j.x_term_rows) at positions j.pos0 ..: their keys and values
// enter the cache.  The term rows past n_tok hold whatever an earlier job left and give rows of Y that nothing reads
// (a row of Y depends on its own token only).
// head: the context's parameters when the job ends the prefix, else null.  Then the last layer carries on with the last
// token's row alone once the keys and values are in the cache (nothing reads the other rows), and one more launch adds
// the last product to the residual row, multiplies the LM head and takes the first timestep.
// *launches receives the number of kernels enqueued.
extern "C" cudaError_t spd_internal_tc_prefill(const spd::TcJob *job, const spd::KParams *head, cudaStream_t s, int *launches) {
  const spd::TcJob &j = *job;
  const int n = j.n_tok, d = j.d, f = j.f;
  int count = 0;
  cudaError_t e = cudaSuccess;
  spd::Product pr;  // where the last product's sums are
  auto done = [&](cudaError_t r) {  // a kernel enqueued (after an error: not)
    e = r;
    ++count;
  };
  auto product = [&](int rows, int wide, int which, int N) {
    if (e == cudaSuccess) done(spd_internal_product(job, rows, wide, which, j.y, N, &pr, s));
  };
  const bool normed = n > spd::kTcTile;  // long jobs: the norm before the product
  auto resid = [&](const spd::TcJob &part, const spd::Product *y, const __nv_bfloat16 *gain) {
    if (e == cudaSuccess) done(normed && part.n_tok == n ? spd_internal_job_norm(&part, y, gain, s) : spd_internal_job_resid(&part, y, gain, s));
  };
  resid(j, nullptr, j.layers[0].attn_norm);
  for (int l = 0; l < j.L && e == cudaSuccess; ++l) {
    product(n, 0, 4 * l, 3 * d);
    if (e == cudaSuccess) done(spd_internal_job_rope_cache(job, &pr, normed, l, s));
    const bool end = head && l + 1 == j.L;
    spd::TcJob part = j;  // the rows that carry on
    if (end) {
      part.h += (size_t)(n - 1) * d;
      part.q += (size_t)(n - 1) * d;
      part.pos0 += n - 1;
      part.n_tok = 1;
    }
    if (e == cudaSuccess)
      done(j.hd == 128 ? launch_attn<128>(part, l, part.n_tok, s) : launch_attn<64>(part, l, part.n_tok, s));  // other head sizes never get here
    product(part.n_tok, 0, 4 * l + 1, d);
    resid(part, &pr, j.layers[l].ffn_norm);
    product(part.n_tok, 0, 4 * l + 2, 2 * f);
    if (e == cudaSuccess) done(spd_internal_job_swiglu(&part, &pr, normed && !end, s));
    product(part.n_tok, 1, 4 * l + 3, d);
    if (end && e == cudaSuccess) done(spd_internal_job_head(head, part.h, &pr, j.sm_count, s));
    else if (l + 1 < j.L) resid(part, &pr, j.layers[l + 1].attn_norm);  // without a head the last layer's output feeds nothing
  }
  if (launches) *launches = count;
  return e;
}
