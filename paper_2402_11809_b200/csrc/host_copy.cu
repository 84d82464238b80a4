// Transfers of space_step_host between pinned host memory and the context's staging, as kernels that read and
// write host memory through its device mapping.
//
// What a resident-cache step moves besides the logits and the attention output are many small pieces: the
// query rows, one run of block rows per kv head of K and of V, a handful of numbers per sequence, and back one
// run of k+1 rows per kv head and the results.  A copy command costs 6-7 us on its stream whatever it moves
// (13-20 us alone), a strided one more, and they queue behind one another: with five up and three down, half of
// the step on one 7B-shaped sequence (141 us in a steady loop, 88 now).  One kernel each way moves the same bytes
// with all pieces in flight together.  Bound by PCIe: measured 46 GB/s plus 4 us either way, whatever the number
// of blocks.
#include "common.cuh"

namespace {

constexpr int HC_THREADS = 256;

// First row moved of one (sequence, kv head), in 16-byte pieces from the cache's base.
__device__ __forceinline__ size_t run_offset(const HostCopyParams& p, int b, int h) {
  return (((size_t)b * p.H_kv + h) * p.s_cap + (size_t)p.len[b]) * p.row_vecs;
}

// The query rows, then [b][h][K, V][run_vecs] of the block's rows; the small arrays by the first block.
__global__ void __launch_bounds__(HC_THREADS) host_upload_kernel(const HostCopyParams p) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr int U = 4;
  const int64_t total = p.q_vecs + (int64_t)p.B * p.H_kv * 2 * p.run_vecs;
  const int64_t stride = (int64_t)gridDim.x * HC_THREADS;
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < p.small_words; i += HC_THREADS) p.d_small[i] = p.h_small[i];
    for (int i = threadIdx.x; i < p.B; i += HC_THREADS) p.d_status[i] = 0;
  }
  for (int64_t i0 = (int64_t)blockIdx.x * HC_THREADS + threadIdx.x; i0 < total; i0 += U * stride) {
    uint4 v[U];
    uint4* dst[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {                           // all loads of a batch are issued before its stores
      const int64_t i = i0 + u * stride;
      dst[u] = nullptr;
      if (i < p.q_vecs) {
        v[u] = p.h_q[i]; dst[u] = p.d_q + i;
      } else if (i < total) {
        int64_t r = i - p.q_vecs;
        const int x = (int)(r % p.run_vecs); r /= p.run_vecs;
        const int which = (int)(r & 1);      r >>= 1;
        const int h = (int)(r % p.H_kv), b = (int)(r / p.H_kv);
        if (p.len[b] >= 0) {
          const size_t at = run_offset(p, b, h) + x;
          v[u] = (which ? p.h_v : p.h_k)[at];
          dst[u] = (which ? p.d_v : p.d_k) + at;
        }
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u) if (dst[u]) *dst[u] = v[u];
  }
}

// The commit and the way down in one: [b][h][K, V][row g = 0..k][piece].  Row L+g(k+1) goes to row L+g of both the
// device's and the host's cache for the accepted candidates g = 1..i* (all k of them when speculative: rows beyond
// the new length, see space_verify_commit); the host's other rows of L .. L+k become the device's.  Sources and
// destinations never overlap.
__global__ void __launch_bounds__(HC_THREADS) host_download_kernel(const HostCopyParams p) {
  pdl_launch_dependents();
  pdl_wait();
  const int k1 = p.k + 1;
  const int64_t total = (int64_t)p.B * p.H_kv * 2 * p.run_vecs;
  const int64_t stride = (int64_t)gridDim.x * HC_THREADS;
  for (int64_t i = (int64_t)blockIdx.x * HC_THREADS + threadIdx.x; i < total; i += stride) {
    int64_t r = i;
    const int x = (int)(r % p.run_vecs); r /= p.run_vecs;
    const int which = (int)(r & 1);      r >>= 1;
    const int h = (int)(r % p.H_kv), b = (int)(r / p.H_kv);
    if (p.len[b] < 0) continue;
    const int g = x / p.row_vecs, v = x - g * p.row_vecs;
    const bool moves = g > 0 && (p.speculative || g <= p.n_accept[b]);
    const size_t base = run_offset(p, b, h) + v;
    uint4* dev = which ? p.d_v : p.d_k;
    const uint4 val = dev[base + (size_t)(moves ? g * k1 : g) * p.row_vecs];
    if (moves) dev[base + (size_t)g * p.row_vecs] = val;
    (which ? p.h_v : p.h_k)[base + (size_t)g * p.row_vecs] = val;
  }
  if (blockIdx.x == 0) {
    for (int i = threadIdx.x; i < p.small_words; i += HC_THREADS) p.h_small[i] = p.d_small[i];
    for (int b = threadIdx.x; b < p.B; b += HC_THREADS) {
      p.h_status[b] = p.d_status[b] | p.d_vstatus[b];
      p.d_vstatus[b] = 0;
      p.h_len_out[b] = p.len[b] < 0 ? p.old_len[b] : p.len[b] + p.n_accept[b] + 1;
    }
  }
}

int blocks_for(const space_ctx* ctx, int64_t vecs, int per_thread) {
  int64_t n = (vecs + (int64_t)HC_THREADS * per_thread - 1) / ((int64_t)HC_THREADS * per_thread);
  if (n > ctx->sm_count) n = ctx->sm_count;
  return n < 1 ? 1 : (int)n;
}

}  // namespace

int launch_host_upload(space_ctx* ctx, const HostCopyParams& p, cudaStream_t st) {
  const int64_t vecs = p.q_vecs + (int64_t)p.B * p.H_kv * 2 * p.run_vecs;
  const cudaError_t e = launch_pdl(host_upload_kernel, dim3(blocks_for(ctx, vecs, 4)), dim3(HC_THREADS), 0, st, p);
  ctx->launches += 1;
  return cuda_ok(e);
}

int launch_host_download(space_ctx* ctx, const HostCopyParams& p, cudaStream_t st) {
  const int64_t vecs = (int64_t)p.B * p.H_kv * 2 * p.run_vecs;
  const cudaError_t e = launch_pdl(host_download_kernel, dim3(blocks_for(ctx, vecs, 1)), dim3(HC_THREADS), 0, st, p);
  ctx->launches += 1;
  return cuda_ok(e);
}
