// The two kernels of a job's attention over a bf16 cache, side by side on the same queries and cache.
#include "spd_prefill_tc.cu"

// (what a job's other kernels would be called by; no test of this file gets there)
extern "C" {
cudaError_t spd_internal_job_resid(const spd::TcJob *, const spd::Product *, const __nv_bfloat16 *, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t spd_internal_job_norm(const spd::TcJob *, const spd::Product *, const __nv_bfloat16 *, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t spd_internal_job_rope_cache(const spd::TcJob *, const spd::Product *, int, int, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t spd_internal_job_swiglu(const spd::TcJob *, const spd::Product *, int, cudaStream_t) { return cudaErrorNotSupported; }
cudaError_t spd_internal_job_head(const spd::KParams *, const float *, const spd::Product *, int, cudaStream_t) { return cudaErrorNotSupported; }

cudaError_t attn_prepare() { return spd_internal_tc_prepare(); }

// which: 0 the kernel of up to 128 tokens, 4 and 8 the longer jobs' with as many warps a block
cudaError_t attn_run(int which, int hd, float *q, void *k, void *v, uint16_t *x, int heads, int rows, int max_pos, int layer, int pos0, int n_tok) {
  spd::TcJob j = {};
  j.q = q;
  j.kcache = k;
  j.vcache = v;
  j.x = x;
  j.d = heads * hd;
  j.hd = hd;
  j.H = heads;
  j.x_term_rows = rows;
  j.max_pos = max_pos;
  j.kv_bf16 = 1;
  j.pos0 = pos0;
  cudaError_t e;
  if (which == 4) e = hd == 128 ? launch_attn_mma<128, 4>(j, layer, n_tok, 0) : launch_attn_mma<64, 4>(j, layer, n_tok, 0);
  else if (which == 8) e = hd == 128 ? launch_attn_mma<128, 8>(j, layer, n_tok, 0) : launch_attn_mma<64, 8>(j, layer, n_tok, 0);
  else e = n_tok > spd::kTcTile ? cudaErrorInvalidValue : (hd == 128 ? launch_attn<128>(j, layer, n_tok, 0) : launch_attn<64>(j, layer, n_tok, 0));
  return e == cudaSuccess ? cudaDeviceSynchronize() : e;
}
}
