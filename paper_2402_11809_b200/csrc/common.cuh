// Internal declarations shared by the translation units of libspace.
#pragma once
#include <cuda_runtime.h>
#include <cuda_bf16.h>
#include <stdint.h>
#include "../../include/space.h"
#include <cstring>

#define SPACE_VERIFY_MAX_CHUNKS 64
#define SPACE_VERIFY_THREADS 256
#define SPACE_FUSED_MAX_CHUNKS 16

// ---- Philox4x32-10 (Salmon et al., SC'11) ---------------------------------
struct Philox4 { uint32_t x, y, z, w; };

__host__ __device__ __forceinline__ Philox4 philox4x32_10(uint32_t c0, uint32_t c1, uint32_t c2,
                                                          uint32_t c3, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    const uint64_t p0 = (uint64_t)0xD2511F53u * c0;
    const uint64_t p1 = (uint64_t)0xCD9E8D57u * c2;
    const uint32_t n0 = (uint32_t)(p1 >> 32) ^ c1 ^ k0;
    const uint32_t n2 = (uint32_t)(p0 >> 32) ^ c3 ^ k1;
    c1 = (uint32_t)p1;
    c3 = (uint32_t)p0;
    c0 = n0;
    c2 = n2;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return Philox4{c0, c1, c2, c3};
}

// 32-bit word -> uniform in (0,1), exactly representable in binary32.
// ((w >> 9) + 1/2) 2^-23, built without an integer-to-float conversion: the 23 bits
// become the mantissa of a float in [1, 2), and subtracting 1 - 2^-24 (the largest
// float below 1) leaves (2m + 1) 2^-24 exactly.
__host__ __device__ __forceinline__ float uniform_open(uint32_t w) {
  const uint32_t bits = 0x3F800000u | (w >> 9);
  float f;
#ifdef __CUDA_ARCH__
  f = __uint_as_float(bits);
#else
  memcpy(&f, &bits, sizeof(f));
#endif
  return f - 0.99999994f;
}

enum { PURPOSE_ACCEPT = 0, PURPOSE_TOKEN = 1, PURPOSE_DRAFT = 2 };

// Gumbel noise in units of log 2:  -log2(-log2 u)  for u = (m + 1/2) 2^-23.
// arg-max_x (z_x/T - log(-log u_x)) = arg-max_x (z_x*log2(e)/T - log2(-log2 u_x)):
// the two scores differ by the factor log 2 and a constant, so the hardware
// base-2 logarithm serves without rescaling.  Near u = 1 the inner logarithm is
// taken from its series in d = 1 - u (exact in binary32); the error of the result
// stays below 3e-5, inside the 1e-4 band within which two scores count as tied.
__device__ __forceinline__ float fast_log2(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float gumbel2_from_uniform(float u) {
  const float d = 1.0f - u;
  const float t = (d < 0.0078125f) ? d * (1.0f + d * (0.5f + d * 0.33333334f)) * 1.4426950408889634f
                                   : -fast_log2(u);
  return -fast_log2(t);
}


// Sixteen bytes of logits from a row that starts at any element-aligned address (an odd vocabulary leaves
// most rows off the 16-byte grid): the two aligned pieces that hold them, each with at least one byte of
// the vector, shifted into place by the row's offset (the same for the whole row, so no branch diverges).
// About two instructions per logit; the second piece is the neighbouring lane's first one and hits L1.
struct Piece2 { uint4 a, b; };
template <typename T>
__device__ __forceinline__ Piece2 load_pieces(const T* row, int x) {
  const uintptr_t at = reinterpret_cast<uintptr_t>(row + x);
  const uint4* q = reinterpret_cast<const uint4*>(at & ~(uintptr_t)15);
  Piece2 r;
  r.a = __ldg(q);
  r.b = (at & 15) ? __ldg(q + 1) : r.a;
  return r;
}
template <typename T>
__device__ __forceinline__ uint4 shift_pieces(const Piece2& r, const T* row) {
  const uint32_t off = (uint32_t)(reinterpret_cast<uintptr_t>(row) & 15);   // (vectors start at multiples of 16 bytes of the row)
  uint32_t w[8] = {r.a.x, r.a.y, r.a.z, r.a.w, r.b.x, r.b.y, r.b.z, r.b.w};
  if (off & 8) {
#pragma unroll
    for (int i = 0; i < 6; ++i) w[i] = w[i + 2];
  }
  if (off & 4) {
#pragma unroll
    for (int i = 0; i < 5; ++i) w[i] = w[i + 1];
  }
  if (sizeof(T) == 2 && (off & 2)) {
#pragma unroll
    for (int i = 0; i < 4; ++i) w[i] = __funnelshift_r(w[i], w[i + 1], 16);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// Asks L2 for a chunk's first sweep of logits, for the time before a kernel's dependency wait: with a programmatic
// launch the blocks are resident while the kernel before them still runs.  Only a request to the point of
// coherence: whatever is still being written is what the loads after the wait will see.  (Without / with, us:
// sixteen sequences of 36 rows of 32000 behind a short attention, graph replay, 24.9 / 24.4 a step; eight decoding
// steps for two sequences, steady loop, 185 / 182; one sequence's step the same either way.)
template <typename T>
__device__ __forceinline__ void prefetch_chunk(const T* row, int begin, int end) {
  constexpr int N = 16 / (int)sizeof(T);
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const int x = begin + (u * SPACE_VERIFY_THREADS + (int)threadIdx.x) * N;
    if ((threadIdx.x & 7) == 0 && x < end) asm volatile("prefetch.global.L2 [%0];" ::"l"(row + x));   // (a 128-byte line)
  }
}

// Blocks that a launch over rows and chunks may have to be resident at once: three per SM, and a few more.
static inline int64_t row_chunk_slots(int sm_count) { return 3 * (int64_t)sm_count * 21 / 20; }
// Chunks per row and their length.  A sweep of a block is four vectors per thread (8192 bf16 logits); a
// block costs about 3 us whatever it scans (reduction, fence, arrival).  So: as few sweeps per block as let all
// blocks be resident at once, four where they cannot be.  Measured, us per call
// (graph replay of space_verify_commit) with 1 / 2 / 3 / 4 sweeps per block: 80 rows of 50257 10.7 / 9.4 / 10.9 /
// 13.6, 98 rows of 128256 16.6 / 12.5 / 13.1 / 10.5, 576 rows of 32000 22.7 / 16.5 / 16.6 / 15.2, top-10 lists of 72
// and 48 rows of 128256 39 / 31 / 29 / 32 (27.7 with three and two), sampling 64 x 5 rows of 128256 106 / 71 / 66 / 57.
static inline int row_chunks(int vocab, int rows, int vec, int sm_count, int max_chunks, int* chunk_out) {
  const int sweep = SPACE_VERIFY_THREADS * vec * 4;
  const int64_t slots = row_chunk_slots(sm_count);
  int64_t nc = 1;
  for (int per_block = 1; per_block <= 4; ++per_block) {
    nc = (vocab + (int64_t)per_block * sweep - 1) / ((int64_t)per_block * sweep);
    if (nc * rows <= slots) break;
  }
  if (nc > max_chunks) nc = max_chunks;
  int chunk = (int)((vocab + nc - 1) / nc);
  chunk = (chunk + vec - 1) / vec * vec;
  *chunk_out = chunk;
  return (vocab + chunk - 1) / chunk;
}

// ---- context ---------------------------------------------------------------
struct VerifyPartial { float m, s, gs; int idx, gidx, pad0, pad1, pad2; };   // 32 bytes
struct VerifyRow     { float m, s; int idx, pad; };

struct AttnPlanHost {
  int n_ctas;         // persistent grid size
  int n_mblocks;      // query-row blocks per (sequence, kv head)
  int rows_per_mblock;// block rows (i) per query-row block
};

struct space_ctx {
  space_config cfg;
  int sm_count;
  int64_t launches;
  // one allocation, carved up
  char* ws;
  size_t ws_bytes;
  float* attn_part;        // split partials
  size_t attn_part_slots;
  int* counters;           // [3][max_batch] self-resetting arrival counters (two verify launches, commit), then an error word
  int* merge_cnt;          // attention, row kernel: cut descriptors, one per (sequence, kv head, row block), and owners
  int* arrived;            // attention: pieces of a cut that are stored, one per (sequence, kv head, row block)
  VerifyPartial* vpart;    // [max_batch][k_max+2][SPACE_VERIFY_MAX_CHUNKS]
  VerifyRow* vrow;         // [max_batch][k_max+1]
  VerifyPartial* vfused;   // [max_batch][SPACE_MAX_ROWS][16] single-launch greedy path
  char* vtopk;             // filtered sampling: top-k lists per (sequence, row, chunk)
  int32_t* vstatus;        // [max_batch] status bits of a verification that runs beside the attention (space_step_host)
  char* lm_part;           // output-projection statistics [256 block rows][sm_count] x 16 bytes
  char* lm_gather;         // gathered mask rows of the projection's second phase
  int* lm_counter;         // {arrival counter, first timeout site}
  // staging for space_step_host
  char* stage;
  char* host_small;        // pinned host mirror of the staging area's small per-sequence arrays (host_staging only)
  cudaStream_t aux_stream; // space_step_host: second stream, so that the logits upload and the download of the
  cudaEvent_t aux_ev[4];   //   attention output overlap the kernels (host_staging only)
  size_t stage_bytes;
  // per-kernel event timing (space_profile_*)
  int prof_on;
  int prof_n[SPACE_K_COUNT];
  cudaEvent_t* prof_ev[SPACE_K_COUNT];   // [2 * SPACE_PROFILE_MAX_STEPS] start/stop pairs, lazily created
  // cached block layout (Eq. 5 mask rows) and the attention kernel's visibility words, per (k, mask variant)
  int lay_k, lay_variant;                // lay_k = 0: nothing cached
  uint64_t lay_mask[SPACE_MAX_ROWS];
  int cluster_fit[2][17];                // transposed and row attention kernel: resident clusters of that many blocks (0: not asked yet)
  int visq_k, visq_variant;
  uint64_t visq[2][SPACE_MAX_ROWS];
  // cached TMA descriptors
  const void* tm_q_ptr; const void* tm_k_ptr; const void* tm_v_ptr;
  int64_t tm_key[8];
  alignas(64) unsigned char tm_q[128];
  alignas(64) unsigned char tm_k[128];
  alignas(64) unsigned char tm_v[128];
};

// ---- KV commit: shared by kv_commit_kernel and the verify kernels that carry the commit ----
// Rows L + g(k+1) -> L + g, g = 1..i*, of K and V for every kv head (16-byte pieces).
struct CommitParams {
  int B, k, H_kv, d, blocks_per_seq, in_place;
  int64_t s_cap;
  __nv_bfloat16* kc; __nv_bfloat16* vc;
  int64_t sb, sh, ss;
  const int32_t* n_accept; const int32_t* kv_len;
  int32_t* kv_len_out; int32_t* src; int32_t* dst; int32_t* status;
  int* counter;
  const int32_t* page_table; int pages_per_seq, n_pages;   // paged cache (page_table != nullptr): kc / vc are page pools
};

// Row s of sequence b, head h, of a cache that is contiguous (page_table == nullptr) or paged:
// offset in elements from the cache base, or -1 for a page-table entry outside the pool.
__device__ __forceinline__ int64_t kv_row_offset(const int32_t* page_table, int pages_per_seq, int n_pages,
                                                 int64_t sb, int64_t sh, int64_t ss, int b, int h, int s) {
  if (!page_table) return (int64_t)b * sb + (int64_t)h * sh + (int64_t)s * ss;
  const int pg = page_table[(int64_t)b * pages_per_seq + s / SPACE_PAGE_SIZE];
  if (pg < 0 || pg >= n_pages) return -1;
  return (int64_t)pg * sb + (int64_t)h * sh + (int64_t)(s % SPACE_PAGE_SIZE) * ss;
}

__device__ __forceinline__ bool commit_fits(const CommitParams& p, int L) {
  return L >= 0 && (int64_t)L + (int64_t)(p.k + 1) * (p.k + 1) <= p.s_cap;
}

// 16-byte pieces in the move of n rows of a sequence, and piece t of it: its bytes and where they go (nullptr: a bad page).
__device__ __forceinline__ int commit_pieces(const CommitParams& p, int n) { return n * p.H_kv * 2 * (p.d / 8); }
template <bool PAGED>
__device__ __forceinline__ uint4* commit_piece(const CommitParams& p, int b, int L, int t, uint4& val) {
  const int k1 = p.k + 1, vec_per_row = p.d / 8;
  int r = t;
  const int v = r % vec_per_row; r /= vec_per_row;
  const int which = r % 2;       r /= 2;
  const int h = r % p.H_kv;      r /= p.H_kv;
  const int g = r + 1;                                // candidate g
  __nv_bfloat16* base = which ? p.vc : p.kc;
  if (!PAGED) {
    base += (int64_t)b * p.sb + (int64_t)h * p.sh;
    val = *(reinterpret_cast<const uint4*>(base + (int64_t)(L + g * k1) * p.ss) + v);
    return reinterpret_cast<uint4*>(base + (int64_t)(L + g) * p.ss) + v;
  }
  const int64_t so = kv_row_offset(p.page_table, p.pages_per_seq, p.n_pages, p.sb, p.sh, p.ss, b, h, L + g * k1);
  const int64_t dof = kv_row_offset(p.page_table, p.pages_per_seq, p.n_pages, p.sb, p.sh, p.ss, b, h, L + g);
  if (so >= 0 && dof >= 0) {
    val = *(reinterpret_cast<const uint4*>(base + so) + v);
    return reinterpret_cast<uint4*>(base + dof) + v;
  }
  if (p.status && v == 0 && which == 0 && h == 0) atomicOr(p.status + b, SPACE_ST_BAD_PAGE);   // the row stays where it is
  return nullptr;
}

// Slice `part` of `nparts` of sequence b's move, by `nthreads` threads (this one is `tid`).
// All loads of a batch of U pieces are issued before its stores.
template <bool PAGED, int U = 8>
__device__ __forceinline__ void commit_rows_impl(const CommitParams& p, int b, int L, int i_star, int part, int nparts,
                                                 int tid, int nthreads) {
  const int total = commit_pieces(p, i_star);
  const int stride = nparts * nthreads;
  for (int t0 = part * nthreads + tid; t0 < total; t0 += U * stride) {
    uint4 val[U];
    uint4* dd[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int t = t0 + u * stride;
      dd[u] = nullptr;
      if (t < total) {
        dd[u] = commit_piece<PAGED>(p, b, L, t, val[u]);
      }
    }
#pragma unroll
    for (int u = 0; u < U; ++u)
      if (dd[u]) *dd[u] = val[u];
  }
}

// Contiguous cache only: the form the verify kernels carry (it sits in their critical path; with a
// paged cache space_verify_commit runs the commit kernel after them instead).
__device__ __forceinline__ void commit_rows(const CommitParams& p, int b, int L, int i_star, int part, int nparts,
                                            int tid, int nthreads) {
  commit_rows_impl<false>(p, b, L, i_star, part, nparts, tid, nthreads);
}
// Either cache form (the commit kernel).
__device__ __forceinline__ void commit_rows_any(const CommitParams& p, int b, int L, int i_star, int part, int nparts,
                                                int tid, int nthreads) {
  if (p.page_table) commit_rows_impl<true>(p, b, L, i_star, part, nparts, tid, nthreads);
  else commit_rows_impl<false>(p, b, L, i_star, part, nparts, tid, nthreads);
}

// New length and index tables of sequence b (one thread).
__device__ __forceinline__ void commit_tables(const CommitParams& p, int b, int L, int i_star, bool fits) {
  const int k1 = p.k + 1;
  if (!fits) {
    if (p.status) atomicOr(p.status + b, SPACE_ST_CAPACITY);
    i_star = -1;                                        // nothing committed, length unchanged
  }
  if (p.kv_len_out) p.kv_len_out[b] = L + i_star + 1;
  for (int g = 0; g < k1; ++g) {
    if (p.src) p.src[b * k1 + g] = (g <= i_star) ? L + g * k1 : -1;
    if (p.dst) p.dst[b * k1 + g] = (g <= i_star) ? L + g : -1;
  }
}

// ---- space_step_host: transfers by kernels over the device mapping of pinned host memory (host_copy.cu) ----
struct HostCopyParams {
  int B, H_kv;
  int row_vecs, run_vecs;              // 16-byte pieces per cache row, and per run of rows moved
  int small_words;                     // 4-byte words of the small arrays
  int64_t s_cap, q_vecs;
  const uint4* h_q; uint4* d_q;
  uint4* h_k; uint4* h_v; uint4* d_k; uint4* d_v;      // [B, H_kv, s_cap, d] on both sides
  int32_t* h_small; int32_t* d_small; int32_t* d_status;
  // way down: the commit's part
  int k, speculative;                  // speculative: all k candidate rows move, as in the single-launch verify
  const int32_t* n_accept; int32_t* d_vstatus;         // the verification's status bits (cleared for the next call)
  int32_t* h_status; int32_t* h_len_out;
  int32_t len[128];                    // first row moved of every sequence, -1: none (it does not fit)
  int32_t old_len[128];
};
int launch_host_upload(space_ctx* ctx, const HostCopyParams& p, cudaStream_t st);
int launch_host_download(space_ctx* ctx, const HostCopyParams& p, cudaStream_t st);

// ---- per-stage launchers (defined next to their kernels) -------------------
// cm != nullptr: the verify kernels also carry out the commit described by cm (one launch less)
// mapped: the logits lie in host memory (read where they are, by the launches that read only the rows they need)
int launch_verify(space_ctx* ctx, const space_verify_args* a, const space_commit_args* cm, cudaStream_t st, bool mapped = false);
bool verify_is_fused(const space_verify_args* a);   // whether a call on device logits takes one launch
int launch_verify_filtered(space_ctx* ctx, const space_verify_args* a, const space_commit_args* cm, cudaStream_t st);
size_t verify_filter_scratch_bytes(int max_batch, int k_max);
void fill_commit_params(const space_ctx* ctx, const space_commit_args* a, CommitParams* p);
int launch_verify_noalloc(const space_verify_args* a, cudaStream_t st);
int launch_commit(space_ctx* ctx, const space_commit_args* a, cudaStream_t st);
int launch_lmhead_verify(space_ctx* ctx, const space_lmhead_args* a, cudaStream_t st);
size_t lmhead_partial_bytes(int sm_count);
size_t lmhead_gather_bytes();
int launch_attn_simt(space_ctx* ctx, const space_attn_args* a, const uint64_t* mask_rows,
                     cudaStream_t st);
int launch_attn_tensor(space_ctx* ctx, const space_attn_args* a, const uint64_t* mask_rows,
                       cudaStream_t st);
int launch_attn_rows(space_ctx* ctx, const space_attn_args* a, const uint64_t* mask_rows, cudaStream_t st);
size_t attn_tensor_partial_floats(const space_config* cfg, int sm_count, size_t* slots);
int launch_philox_debug(uint64_t seed, int64_t n, const uint32_t* c0, const uint32_t* c1,
                        const uint32_t* c2, const uint32_t* c3, uint32_t* out, cudaStream_t st);

// Event pair around one kernel launch when profiling is on.
struct ProfScope {
  space_ctx* ctx; int which; cudaStream_t st; int slot;
  ProfScope(space_ctx* c, int w, cudaStream_t s) : ctx(c), which(w), st(s), slot(-1) {
    if (!c->prof_on || !c->prof_ev[w] || c->prof_n[w] >= SPACE_PROFILE_MAX_STEPS) return;
    slot = c->prof_n[w];
    cudaEventRecord(c->prof_ev[w][2 * slot], st);
  }
  ~ProfScope() {
    if (slot < 0) return;
    cudaEventRecord(ctx->prof_ev[which][2 * slot + 1], st);
    ctx->prof_n[which] = slot + 1;
  }
};

// Programmatic dependent launch: the kernel may be scheduled while the previous
// kernel of the stream is still draining; every kernel calls pdl_wait() before
// it touches global memory, which blocks until the previous kernel has finished
// and its writes are visible.  Both are no-ops without the launch attribute.
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <typename... KArgs, typename... Args>
static inline cudaError_t launch_pdl(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem,
                                     cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, KArgs(args)...);
}

static inline int cuda_ok(cudaError_t e) { return e == cudaSuccess ? SPACE_OK : SPACE_E_CUDA; }
