// The launchers that csrc/space_api.cu calls, as work of the stand-in runtime (fake_cuda_runtime.cpp).
#include "../paper_2402_11809_b200/csrc/common.cuh"

cudaError_t fake_issue(cudaStream_t s);

namespace {
int launch(space_ctx* ctx, cudaStream_t s) {
  if (fake_issue(s) != cudaSuccess) return SPACE_E_CUDA;
  ctx->launches += 1;
  return SPACE_OK;
}
}  // namespace

extern "C" int fake_vstatus(space_ctx* ctx, int b) { return ctx->vstatus[b]; }

int launch_host_upload(space_ctx* ctx, const HostCopyParams&, cudaStream_t s) { return launch(ctx, s); }
int launch_host_download(space_ctx* ctx, const HostCopyParams& p, cudaStream_t s) {
  const int rc = launch(ctx, s);
  if (rc == SPACE_OK) for (int b = 0; b < p.B; ++b) { p.h_status[b] = p.d_vstatus[b]; p.d_vstatus[b] = 0; }
  return rc;
}
// (a verification that finds an out-of-range candidate in sequence 0)
int launch_verify(space_ctx* ctx, const space_verify_args* a, const space_commit_args*, cudaStream_t s, bool) {
  const int rc = launch(ctx, s);
  if (rc == SPACE_OK && a->status) a->status[0] |= SPACE_ST_BAD_CANDIDATE;
  return rc;
}
bool verify_is_fused(const space_verify_args*) { return true; }
int launch_attn_tensor(space_ctx* ctx, const space_attn_args*, const uint64_t*, cudaStream_t s) { return launch(ctx, s); }
int launch_attn_simt(space_ctx* ctx, const space_attn_args*, const uint64_t*, cudaStream_t s) { return launch(ctx, s); }
int launch_commit(space_ctx* ctx, const space_commit_args*, cudaStream_t s) { return launch(ctx, s); }
int launch_lmhead_verify(space_ctx* ctx, const space_lmhead_args*, cudaStream_t s) { return launch(ctx, s); }
int launch_verify_noalloc(const space_verify_args*, cudaStream_t) { return SPACE_OK; }
int launch_philox_debug(uint64_t, int64_t, const uint32_t*, const uint32_t*, const uint32_t*, const uint32_t*, uint32_t*, cudaStream_t) { return SPACE_OK; }
size_t attn_tensor_partial_floats(const space_config*, int, size_t* slots) { *slots = 1; return 64; }
size_t verify_filter_scratch_bytes(int, int) { return 256; }
size_t lmhead_partial_bytes(int) { return 256; }
size_t lmhead_gather_bytes() { return 256; }
