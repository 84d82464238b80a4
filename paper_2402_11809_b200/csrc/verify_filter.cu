// Verification with filtered target distributions (App. A.4 runs random sampling with top-k = 10 and
// top-p = 0.95): every distribution that Algorithm 1 tests against or samples from is softmax(z / T)
// restricted to its top_k largest logits (lowest token first on ties), then to the shortest prefix of
// those, in descending order, whose probability reaches top_p, and renormalised.
//
// Two launches of one kernel.  Phase 0 finds the top_k logits of the k+1 target rows; the last block
// of a sequence builds the filtered distributions, runs the acceptance loop (r <= Q'(c) / P_c), draws
// the extra token from row i* (Gumbel arg-max over the kept tokens, Philox noise keyed by the token as
// in verify.cu) and emits the tokens.  Phase 1 does the same for the k mask rows of group i* and
// writes the next candidates (their arg-maxes with P_c = 1, or samples from the filtered rows with
// their probabilities when candidates are sampled); with a commit on board its blocks also move the
// accepted cache rows.  A small batch goes through one launch instead (PHASE_BOTH): every block row is
// searched, and the last block runs both halves on the rows it needs.
//
// SPACE_RESAMPLE_RESIDUAL_DRAFT keeps sampled candidates lossless (Sec. 3.2 claims an unchanged output
// distribution): phase 1 also writes every candidate's filtered distribution D as a list of top_k
// (token, probability) pairs, and phase 0 of the next step, after rejecting candidate i, draws the extra
// token from norm(max(0, Q - D_i)) -- one warp, its 32 lanes holding Q's kept tokens and D_i's entries.
//
// Top-k selection, per block and segment (a few sweeps of 256 threads x four 16-byte vectors): one pass
// keeps every thread's maximum; the maxima of 128 groups of two threads are ranked against each other; the
// top_k-th of them is a bound tau that at least top_k logits reach and, for rows in no particular order,
// only about top_k do (128 groups of which top_k hold a larger logit: 10 for top_k = 10, 37 for 32).  Only
// groups whose maximum reaches tau can hold such a logit, so at most top_k groups' worth are collected
// whatever the row looks like; their threads read again the vector that has their maximum and, only where the
// second largest of their vectors reaches tau too, the others (reading all of them again in an unrolled loop took
// 95 us per call on 64 x 4 rows of 128256 logits, top-10, and 13.6 on 4 x 3 rows of 3000, where it is code size; this
// way 72 and 12.6).
// The collected keys are ranked together with the list of the segments before by counting.
// (Inserting logit by logit into warp lists, with a ballot and shuffles each, took 47 us per launch on
// 24 x 3 rows of 128256 logits and 65 us on ten rows of 32000 with top_k = 32.)
// Keys are 64-bit words whose unsigned order is "larger logit, then lower token", so exact ties go to
// the lower token everywhere.  Block lists go to a scratch array, and an arrival counter picks the block
// that finishes a sequence; it merges the lists of a row with one warp.
#include "common.cuh"
#include <math_constants.h>

namespace {

constexpr int FILT_THREADS = 256;
constexpr int FILT_MAX_CHUNKS = 16;
constexpr int FILT_MAX_K = 32;
constexpr int FILT_GROUP = 2;                            // threads per group whose maximum is ranked
constexpr int FILT_GROUPS = FILT_THREADS / FILT_GROUP;
constexpr int FILT_U = 4;                                // vectors per thread and sweep
constexpr int FILT_BUF = 4096;                           // keys a segment may collect
// Which calls take one launch over all block rows: what it saves is a launch and a second search in a chain, what it
// costs is reading the rows that two launches skip, and more blocks than fit at once.  So: few bytes of logits, or few
// rows and not many bytes.  Measured, us per call (graph replay, other input every call), two launches / one, with 2 heads
// of 64 to commit (32 of 128): few rows: 2 x 25 of 128256 f32 (26 MB, top-30) 29.5 / 23.4 (29.1 / 25.4), 4 x 16 of 128256 bf16
// (16 MB, top-20) 26.6 / 19.1 (27.0 / 21.5), 8 x 9 (18 MB) 23.7 / 18.4 (23.8 / 20.8), 3 x 36 (28 MB) 23.9 / 21.5 (24.4 / 23.8);
// past them: 2 x 64 (33 MB) 24.0 / 27.5, 16 x 9 (37 MB) 25.7 / 27.2, 10 x 16 of 37201 f32 (24 MB) 26.0 / 34.2, 6 x 36 of 50257
// (22 MB) 24.8 / 26.2, but 24 x 9 of 50257 (22 MB) 28.2 / 25.2; few bytes: 4 x 9 of 32000 (2 MB) 17.6 / 12.5, 28 x 9 (16 MB)
// 20.7 / 18.7, 5 x 49 (16 MB) 19.4 / 19.5, 10 x 16 of 50257 (16 MB, top-25) 27.3 / 28.5.
// Not, among the few rows, where one launch has more blocks than fit at once (2 x 36 of 100000 f32, 504 blocks, 24.6 /
// 25.7; 3 x 25, 525 blocks, 23.7 / 25.6; at 448 blocks, 1 x 64, 23.4 / 23.5).  Rows off the 16-byte grid, whose every
// vector is put together from two, have no room for more than three blocks per SM (1 x 64 of 80001 f32, 448 blocks, 25.0 /
// 30.1; 3 x 25 of 70001, 450, 25.9 / 28.8; 1 x 49 of 100001, 441, 25.9 / 24.5), and two sweeps more than both launches take
// together cost more than the launch: two more, 2 x 49 of 50257 f32 22.9 / 25.4, of 128257 bf16 25.6 / 28.6, 3 x 36 of 50257
// f32 22.7 / 25.4, 4 x 25 23.7 / 25.0, 6 x 16 24.1 / 24.4, of 100001 bf16 25.1 / 25.0; one more, 12 x 9 of 50257 f32 27.3 /
// 24.8, of 128257 bf16 29.9 / 27.6; as many, 2 x 25 of 128257 f32 31.0 / 29.1.  On the grid two more gain: 2 x 49 of 128256
// bf16 22.2 / 21.1, of 52000 f32 20.1 / 19.4, 6 x 16 of 50256 f32 21.2 / 18.3.
constexpr int FILT_BOTH_ROWS = 256, FILT_FEW_ROWS = 110;
constexpr int64_t FILT_BOTH_BYTES = 16ll << 20, FILT_FEW_ROWS_BYTES = 30ll << 20;
enum { PHASE_TARGETS = 0, PHASE_MASKS = 1, PHASE_BOTH = 2 };

struct FiltParams {
  int B, k, V, n_q, n_chunks, chunk, top_k, phase;
  int resample, eos_id;
  float top_p, c_t;                    // c_t = log2(e) / T
  uint32_t key0, key1;
  const void* logits; int64_t row_stride;
  const int32_t* cand; const float* cand_prob; const uint32_t* seq_id; const int32_t* kv_len;
  int32_t* n_accept; int32_t* out_tokens; int32_t* n_out; int32_t* next_cand; float* next_cand_prob;
  uint8_t* finished; int32_t* status;
  const int32_t* draft_tok; const float* draft_prob;      // [B, k, list_stride] or NULL (no lists)
  int32_t* next_draft_tok; float* next_draft_prob;        // [B, k, list_stride]
  int list_stride;
  unsigned long long* part;            // [B][rows of the phase][FILT_MAX_CHUNKS][32]
  int* counter;                        // [B], self-resetting
  int do_commit;                       // phase 1 / one launch: the accepted cache rows move as well
  CommitParams cm;
};

__device__ __forceinline__ float fexp2(float x) { float y; asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x)); return y; }

__device__ __forceinline__ unsigned long long make_key(float v, int idx) {
  uint32_t u = __float_as_uint(v + 0.f);                  // (-0 counts as 0)
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)idx);
}
__device__ __forceinline__ void split_key(unsigned long long key, float& v, int& idx) {
  uint32_t u = (uint32_t)(key >> 32);
  u = (u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u;
  v = __uint_as_float(u);
  idx = (int)(0xFFFFFFFFu - (uint32_t)key);
}
__device__ __forceinline__ unsigned long long shfl_xor64(unsigned long long x, int o) {
  const uint32_t lo = __shfl_xor_sync(0xFFFFFFFFu, (uint32_t)x, o), hi = __shfl_xor_sync(0xFFFFFFFFu, (uint32_t)(x >> 32), o);
  return ((unsigned long long)hi << 32) | lo;
}
__device__ __forceinline__ float ld_logit(const float* p) { return *p; }
__device__ __forceinline__ float ld_logit(const __nv_bfloat16* p) { return __bfloat162float(*p); }

// 16 bytes of logits as floats
__device__ __forceinline__ void unpack16(const uint4& v, float (&f)[4], const float*) {
  f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y); f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
}
__device__ __forceinline__ void unpack16(const uint4& v, float (&f)[8], const __nv_bfloat16*) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) { f[2 * i] = __uint_as_float(w[i] << 16); f[2 * i + 1] = __uint_as_float(w[i] & 0xFFFF0000u); }
}

struct FiltShared {
  unsigned long long group_max[FILT_GROUPS];
  unsigned long long run[2][FILT_MAX_K];                  // sorted top_k so far (two copies: one is read, one written)
  unsigned long long tau;
  int count, last, bits, i_star;
  int ok[SPACE_MAX_K + 1];
  unsigned long long buf[FILT_BUF];    // collected keys of a segment, later those of the rows the last block works on
  unsigned long long top[FILT_THREADS / 32][FILT_MAX_K];
};
static_assert(FILT_BUF >= FILT_MAX_K * FILT_GROUP * FILT_U * 8, "one sweep's keys of the longest list must fit");
static_assert(FILT_BUF >= (SPACE_MAX_K + 1) * FILT_MAX_CHUNKS * FILT_MAX_K, "the chunk lists of k+1 rows must fit");

// The N logits at x of a row whose chunk ends at `end` (-inf past it).
template <typename T, bool ALIGNED, int N>
__device__ __forceinline__ void whole_vector(const Piece2& raw, const T* row, int x, int end, float (&f)[N]) {
  if (x + N <= end) unpack16(ALIGNED ? raw.a : shift_pieces(raw, row), f, (const T*)nullptr);
  else
#pragma unroll
    for (int i = 0; i < N; ++i) f[i] = x + i < end ? ld_logit(row + x + i) : -CUDART_INF_F;
}
template <typename T, bool ALIGNED>
__device__ __forceinline__ Piece2 request_vector(const T* row, int x, int end) {
  Piece2 raw;
  raw.a = raw.b = make_uint4(0, 0, 0, 0);
  if (x + 16 / (int)sizeof(T) <= end) {
    if (ALIGNED) raw.a = __ldg(reinterpret_cast<const uint4*>(row + x));
    else raw = load_pieces(row, x);
  }
  return raw;
}

// Top K of logits [begin, end) of a row as a sorted list in sh.run[returned copy].  ALIGNED: the row is
// 16-byte aligned (else see load_pieces).
template <typename T, bool ALIGNED>
__device__ int chunk_top_k(const T* row, int begin, int end, int K, FiltShared& sh) {
  constexpr int N = 16 / (int)sizeof(T), U = FILT_U;
  constexpr int stride = FILT_THREADS * N;
  const int tid = threadIdx.x;
  // sweeps per segment: as many as the buffer can hold the collected keys of (K groups' worth)
  const int sweeps = max(1, FILT_BUF / (K * FILT_GROUP * U * N));
  int cur = 0;
  if (tid < FILT_MAX_K) sh.run[0][tid] = 0ull;
  for (int s0 = begin; s0 < end; s0 += sweeps * U * stride) {
    const int s1 = min(end, s0 + sweeps * U * stride);
    // ---- this thread's largest logit of the segment: value, the vector that has it first, and the largest
    // of its other vectors
    float m = -CUDART_INF_F, m2 = -CUDART_INF_F;
    int at = -1;
    for (int x = s0 + tid * N; x < s1; x += U * stride) {
      Piece2 raw[U];
#pragma unroll
      for (int u = 0; u < U; ++u) raw[u] = request_vector<T, ALIGNED>(row, x + u * stride, s1);
      float vm[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        float a[N];
        whole_vector<T, ALIGNED, N>(raw[u], row, x + u * stride, s1, a);
#pragma unroll
        for (int w = N / 2; w > 0; w >>= 1)
#pragma unroll
          for (int i = 0; i < w; ++i) a[i] = fmaxf(a[i], a[i + w]);
        vm[u] = a[0];
      }
      float sm = vm[0], sm2 = -CUDART_INF_F;
#pragma unroll
      for (int u = 1; u < U; ++u) { sm2 = fmaxf(sm2, fminf(sm, vm[u])); sm = fmaxf(sm, vm[u]); }
      m2 = fmaxf(fmaxf(m2, sm2), fminf(m, sm));
      if (sm > m || at < 0) {
        m = sm;
#pragma unroll
        for (int u = U - 1; u >= 0; --u) if (vm[u] == sm) at = x + u * stride;
      }
    }
    unsigned long long mine = 0ull;                       // (0: no logit)
    if (at >= 0) {
      float f[N];
      whole_vector<T, ALIGNED, N>(request_vector<T, ALIGNED>(row, at, s1), row, at, s1, f);
      int off = 0;
#pragma unroll
      for (int i = N - 1; i >= 0; --i) if (f[i] == m) off = i;
      mine = make_key(m, at + off);
    }
    unsigned long long g = mine;
#pragma unroll
    for (int o = 1; o < FILT_GROUP; o <<= 1) { const unsigned long long other = shfl_xor64(g, o); g = other > g ? other : g; }
    if ((tid & (FILT_GROUP - 1)) == 0) sh.group_max[tid / FILT_GROUP] = g;
    if (tid == 0) { sh.count = 0; sh.tau = 1ull; }        // fewer than K groups with a logit: take them all
    // (the K-th key of the list so far: a later segment's logit counts only if it is larger)
    const unsigned long long kth = s0 == begin ? 0ull : sh.run[cur][K - 1];
    if (!__syncthreads_or(mine > kth)) continue;
    // ---- tau: the K-th largest group maximum
    if (tid < FILT_GROUPS) {
      const unsigned long long x = sh.group_max[tid];
      int above = 0;
#pragma unroll 16
      for (int j = 0; j < FILT_GROUPS; ++j) above += sh.group_max[j] > x;
      if (x != 0ull && above == K - 1) sh.tau = x;
    }
    __syncthreads();
    const unsigned long long tau = sh.tau > kth ? sh.tau : kth;
    // ---- collect the logits that reach it: the few threads that hold one look at their largest vector again, or,
    // where another of theirs holds one as well, at all of them, the next one on its way (L1, L2)
    if (mine >= tau) {
      float tv; int ti;
      split_key(tau, tv, ti);
      const bool one = m2 < tv;
      const int step = one ? s1 : stride;
      int x = one ? at : s0 + tid * N;
      Piece2 raw = request_vector<T, ALIGNED>(row, x, s1);
#pragma unroll 1
      for (; x < s1; x += step) {
        const Piece2 next = request_vector<T, ALIGNED>(row, min(x + step, s1), s1);
        float v[N];
        whole_vector<T, ALIGNED, N>(raw, row, x, s1, v);
        raw = next;
        float vm = v[0];
#pragma unroll
        for (int i = 1; i < N; ++i) vm = fmaxf(vm, v[i]);
        if (vm < tv) continue;
#pragma unroll
        for (int i = 0; i < N; ++i) {
          if (!(v[i] < tv) && x + i < s1) {
            const unsigned long long key = make_key(v[i], x + i);
            if (key >= tau) sh.buf[atomicAdd(&sh.count, 1)] = key;
          }
        }
      }
    }
    if (tid < FILT_MAX_K) sh.run[cur ^ 1][tid] = 0ull;
    __syncthreads();
    // ---- rank them together with the list so far
    const int n = sh.count, total = n + (s0 == begin ? 0 : K);
    for (int i = tid; i < total; i += FILT_THREADS) {
      const unsigned long long x = i < n ? sh.buf[i] : sh.run[cur][i - n];
      int rank = 0;
      for (int j = 0; j < n; ++j) rank += sh.buf[j] > x;
      if (s0 != begin)
        for (int j = 0; j < K; ++j) rank += sh.run[cur][j] > x;
      if (x != 0ull && rank < K) sh.run[cur ^ 1][rank] = x;
    }
    cur ^= 1;
    __syncthreads();
  }
  return cur;
}

__device__ __forceinline__ unsigned long long shfl64(unsigned long long x, int src) {
  const uint32_t lo = __shfl_sync(0xFFFFFFFFu, (uint32_t)x, src), hi = __shfl_sync(0xFFFFFFFFu, (uint32_t)(x >> 32), src);
  return ((unsigned long long)hi << 32) | lo;
}
// Sorted top K of a row from its chunks' sorted lists in L2 (lists[c * 32 + j]), lane j holding the j-th largest:
// all lists are fetched at once, a bound that at least K keys reach leaves a few more than K of them (the largest
// K-th key of a list, or the smallest key at the place that K / n_chunks keys of every list reach), and those are
// ranked by counting in shared memory (tmp: n_chunks * K keys, out: K keys, the warp's own).  (K rounds of a
// warp-wide maximum over the lists' heads took 3 us for ten keys, 7 for 23.)
__device__ unsigned long long merge_lists(const unsigned long long* lists, int n_chunks, int K, int lane,
                                          unsigned long long* tmp, unsigned long long* out) {
  unsigned long long v[FILT_MAX_CHUNKS];
#pragma unroll
  for (int c = 0; c < FILT_MAX_CHUNKS; ++c)
    v[c] = c < n_chunks && lane < K ? __ldcg(lists + c * FILT_MAX_K + lane) : 0ull;
  unsigned long long lo = ~0ull, hi = 0ull;
#pragma unroll
  for (int c = 0; c < FILT_MAX_CHUNKS; ++c) {
    if (c < n_chunks && v[c] < lo) lo = v[c];
    if (v[c] > hi) hi = v[c];
  }
  lo = shfl64(lo, (K + n_chunks - 1) / n_chunks - 1);
  hi = shfl64(hi, K - 1);
  const unsigned long long tau = lo > hi ? lo : hi;
  int n = 0;
#pragma unroll
  for (int c = 0; c < FILT_MAX_CHUNKS; ++c) {
    const bool keep = v[c] != 0ull && v[c] >= tau;
    const unsigned who = __ballot_sync(0xFFFFFFFFu, keep);
    if (keep) tmp[n + __popc(who & ((1u << lane) - 1u))] = v[c];
    n += __popc(who);
  }
  out[lane] = 0ull;
  __syncwarp();
  for (int i = lane; i < n; i += 64) {                      // two keys per lane and pass
    const unsigned long long a = tmp[i], b = i + 32 < n ? tmp[i + 32] : 0ull;
    int ra = 0, rb = 0;
#pragma unroll 8
    for (int j = 0; j < n; ++j) { const unsigned long long x = tmp[j]; ra += x > a; rb += x > b; }
    if (ra < K) out[ra] = a;
    if (b != 0ull && rb < K) out[rb] = b;
  }
  __syncwarp();
  return out[lane];
}

template <typename T, bool ALIGNED>
__global__ void __launch_bounds__(FILT_THREADS) verify_filter_kernel(const FiltParams p) {
  __shared__ FiltShared sh;
  pdl_launch_dependents();
  const int b = blockIdx.z, r = blockIdx.y, ch = blockIdx.x;
  const int k1 = p.k + 1, K = p.top_k;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n_rows = gridDim.y;
  const int begin = ch * p.chunk, end = min(p.V, begin + p.chunk);
  if (p.phase != PHASE_MASKS)                              // (which mask rows are read is not known yet)
    prefetch_chunk<T>(reinterpret_cast<const T*>(p.logits) + ((int64_t)b * p.n_q + (p.phase == PHASE_TARGETS ? r * k1 : r)) * p.row_stride,
                      begin, end);
  pdl_wait();
  const int i_star0 = p.phase == PHASE_MASKS ? max(0, min(p.n_accept[b], p.k)) : 0;
  // target row r, mask row (i*, r+1), or block row r
  const int brow = p.phase == PHASE_TARGETS ? r * k1 : p.phase == PHASE_MASKS ? i_star0 * k1 + r + 1 : r;
  const T* row = reinterpret_cast<const T*>(p.logits) + ((int64_t)b * p.n_q + brow) * p.row_stride;
  // what the block that finishes the sequence needs besides the lists, in flight during the search (lane j holds
  // candidate c_{j+1})
  const int my_cand = lane < p.k ? p.cand[b * p.k + lane] : -1;
  const float my_prob = lane < p.k ? p.cand_prob[b * p.k + lane] : 0.f;
  const uint32_t seq = p.seq_id ? p.seq_id[b] : (uint32_t)b;
  const int L = p.kv_len ? p.kv_len[b] : 0;
  int Lc = 0;
  if (p.do_commit) {                                        // (phase 1: i* is known, every block moves its slice)
    Lc = p.cm.kv_len[b];
    if (p.phase == PHASE_MASKS && commit_fits(p.cm, Lc))
      commit_rows_any(p.cm, b, Lc, i_star0, r * p.n_chunks + ch, n_rows * p.n_chunks, threadIdx.x, FILT_THREADS);
  }
  const int cur = chunk_top_k<T, ALIGNED>(row, begin, end, K, sh);
  unsigned long long* part = p.part + (int64_t)b * n_rows * FILT_MAX_CHUNKS * FILT_MAX_K;
  // ---- the chunk's list, then arrival: the last block of the sequence finishes it (warp 0 publishes and counts)
  if (warp == 0) {
    if (lane < K) __stcg(part + ((int64_t)r * FILT_MAX_CHUNKS + ch) * FILT_MAX_K + lane, sh.run[cur][lane]);
    __threadfence();
    __syncwarp();
    if (lane == 0) {
      const int prev = atomicAdd(p.counter + b, 1);
      sh.last = prev == n_rows * p.n_chunks - 1;
      if (sh.last) p.counter[b] = 0;
      sh.bits = 0;
    }
  }
  __syncthreads();                                          // (also: every thread's read of the old length precedes the arrival)
  if (!sh.last) return;
  __threadfence();

  const bool with_lists = p.resample == SPACE_RESAMPLE_RESIDUAL_DRAFT;
  const bool literal = p.resample == SPACE_RESAMPLE_PAPER_LITERAL || with_lists;   // candidates are sampled
  float z = 0.f, q = 0.f; int idx = -1; bool keep = false;
  // ---- filtered distribution of row list_row(w) by warp w < count
  auto build = [&](int count, int first, int step) {
    z = 0.f; q = 0.f; idx = -1; keep = false;
    if (warp >= count) return;
    const unsigned long long lst = merge_lists(part + (int64_t)(first + warp * step) * FILT_MAX_CHUNKS * FILT_MAX_K, p.n_chunks, K, lane,
                                               sh.buf + warp * FILT_MAX_CHUNKS * FILT_MAX_K, sh.top[warp]);
    const bool valid = lst != 0ull;
    if (valid) split_key(lst, z, idx);
    // temperature, then softmax over the top-k, then the shortest prefix that reaches top_p
    const float s = z * p.c_t;
    const float s0 = __shfl_sync(0xFFFFFFFFu, s, 0);
    float pj = valid ? fexp2(s - s0) : 0.f;
    float tot = pj;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) tot += __shfl_xor_sync(0xFFFFFFFFu, tot, o);
    pj /= tot;
    float cum = pj;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const float up = __shfl_up_sync(0xFFFFFFFFu, cum, o);
      if (lane >= o) cum += up;
    }
    float before = __shfl_up_sync(0xFFFFFFFFu, cum, 1);     // probability of the tokens before this one
    if (lane == 0) before = 0.f;
    keep = valid && (lane == 0 || p.top_p >= 1.f || before < p.top_p);   // top_p = 1: no nucleus cut
    float ksum = keep ? pj : 0.f;
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) ksum += __shfl_xor_sync(0xFFFFFFFFu, ksum, o);
    q = keep ? pj / ksum : 0.f;
  };

  int i_star = i_star0;
  if (p.phase != PHASE_MASKS) {
    build(k1, 0, p.phase == PHASE_BOTH ? k1 : 1);
    // acceptance test of candidate c_{t+1} against the filtered law of target row t (warp t)
    if (warp < p.k) {
      const int c = __shfl_sync(0xFFFFFFFFu, my_cand, warp);
      const float pc = __shfl_sync(0xFFFFFFFFu, my_prob, warp);
      const bool in_range = c >= 0 && c < p.V;
      const unsigned hit = __ballot_sync(0xFFFFFFFFu, keep && idx == c);
      const float qc = hit ? __shfl_sync(0xFFFFFFFFu, q, __ffs(hit) - 1) : 0.f;
      if (lane == 0) {
        if (!in_range) atomicOr(&sh.bits, SPACE_ST_BAD_CANDIDATE);
        const Philox4 w = philox4x32_10(0u, PURPOSE_ACCEPT, seq, (uint32_t)(L + warp + 1), p.key0, p.key1);
        sh.ok[warp] = in_range && pc > 0.f && uniform_open(w.x) * pc <= qc;   // r <= Q'/P_c  <=>  r P_c <= Q'
      }
    }
    __syncthreads();
    while (i_star < p.k && sh.ok[i_star]) ++i_star;
    if (warp == i_star) {
      // extra token: Gumbel arg-max over the kept tokens of row i*, the rejected point-mass candidate left out
      int exclude = -1;
      {
        const float pc = __shfl_sync(0xFFFFFFFFu, my_prob, min(i_star, p.k - 1));
        const int c = __shfl_sync(0xFFFFFFFFu, my_cand, min(i_star, p.k - 1));
        if (!literal && i_star < p.k && pc == 1.0f) exclude = c;
      }
      float sc = -CUDART_INF_F;
      // compact draft distribution of the rejected candidate: the weight of a kept token is
      // max(0, Q - D); Q itself when nothing was rejected, there are no lists, or nothing is left
      float wq = q;
      bool residual = false;
      if (with_lists && i_star < p.k && p.draft_tok) {
        int dt = -1; float dp = 0.f;
        if (lane < p.list_stride) {
          dt = p.draft_tok[((int64_t)b * p.k + i_star) * p.list_stride + lane];
          dp = p.draft_prob[((int64_t)b * p.k + i_star) * p.list_stride + lane];
          if (dt < 0 || dt >= p.V || !(dp > 0.f) || !(dp < CUDART_INF_F)) { dt = -1; dp = 0.f; }
        }
        float d = 0.f;
        for (int j = 0; j < p.list_stride; ++j) {
          const int tj = __shfl_sync(0xFFFFFFFFu, dt, j);
          const float pj2 = __shfl_sync(0xFFFFFFFFu, dp, j);
          if (tj == idx) d += pj2;
        }
        const float res = keep ? fmaxf(q - d, 0.f) : 0.f;
        residual = __any_sync(0xFFFFFFFFu, res > 0.f);
        if (residual) wq = res;
      }
      if (keep && idx != exclude && (!residual || wq > 0.f)) {
        const Philox4 ph = philox4x32_10((uint32_t)(idx >> 2), PURPOSE_TOKEN, seq, (uint32_t)(L + i_star + 1), p.key0, p.key1);
        const uint32_t w4[4] = {ph.x, ph.y, ph.z, ph.w};
        const float g = gumbel2_from_uniform(uniform_open(w4[idx & 3]));
        sc = with_lists ? fast_log2(wq) + g : fmaf(z, p.c_t, g);
      }
      int bi = keep ? idx : 0x7FFFFFFF;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float os = __shfl_xor_sync(0xFFFFFFFFu, sc, o);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
        if (os > sc || (os == sc && oi < bi)) { sc = os; bi = oi; }
      }
      const int bonus = bi;
      const int j = lane;
      const int tok = (j < i_star) ? my_cand : (j == i_star ? bonus : -1);
      const bool is_eos = p.eos_id >= 0 && j <= i_star && tok == p.eos_id;
      const unsigned eos_mask = __ballot_sync(0xFFFFFFFFu, is_eos && j < k1);
      const int n_out = eos_mask ? __ffs(eos_mask) - 1 : i_star + 1;
      if (j < k1) p.out_tokens[b * k1 + j] = (j < n_out) ? tok : -1;
      if (j == 0) {
        p.n_accept[b] = i_star;
        p.n_out[b] = n_out;
        p.finished[b] = (uint8_t)(eos_mask != 0);
        if (p.status && sh.bits) atomicOr(p.status + b, sh.bits);
      }
    }
  }
  if (p.phase == PHASE_TARGETS) return;
  // (one launch: the whole move falls to this block, i* has only just become known)
  if (p.do_commit && p.phase == PHASE_BOTH && commit_fits(p.cm, Lc))
    commit_rows_any(p.cm, b, Lc, i_star, 0, 1, threadIdx.x, FILT_THREADS);
  if (p.phase == PHASE_BOTH) build(p.k, i_star * k1 + 1, 1);
  else build(p.k, 0, 1);
  // every thread of the sequence's blocks has read the old length by now
  if (p.do_commit && threadIdx.x == 0) commit_tables(p.cm, b, Lc, i_star, commit_fits(p.cm, Lc));
  if (warp < p.k) {
    // next candidate o = warp + 1 from mask row (i*, o)
    int tok; float pr;
    if (!literal) {                                         // point-mass draft: the row's arg-max, P_c = 1
      tok = __shfl_sync(0xFFFFFFFFu, idx, 0); pr = 1.f;
    } else {
      float sc = -CUDART_INF_F;
      if (keep) {
        const Philox4 ph = philox4x32_10((uint32_t)(idx >> 2), PURPOSE_DRAFT, seq, (uint32_t)(L + i_star + 1 + warp + 1),
                                         p.key0, p.key1);
        const uint32_t w4[4] = {ph.x, ph.y, ph.z, ph.w};
        sc = fmaf(z, p.c_t, gumbel2_from_uniform(uniform_open(w4[idx & 3])));
      }
      int bi = keep ? idx : 0x7FFFFFFF; float bq = q;
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const float os = __shfl_xor_sync(0xFFFFFFFFu, sc, o);
        const int oi = __shfl_xor_sync(0xFFFFFFFFu, bi, o);
        const float oq = __shfl_xor_sync(0xFFFFFFFFu, bq, o);
        if (os > sc || (os == sc && oi < bi)) { sc = os; bi = oi; bq = oq; }
      }
      tok = bi; pr = bq;
    }
    if (lane == 0) { p.next_cand[b * p.k + warp] = tok; p.next_cand_prob[b * p.k + warp] = pr; }
    if (with_lists && lane < p.list_stride) {               // the row's filtered distribution, descending
      p.next_draft_tok[((int64_t)b * p.k + warp) * p.list_stride + lane] = keep ? idx : -1;
      p.next_draft_prob[((int64_t)b * p.k + warp) * p.list_stride + lane] = keep ? q : 0.f;
    }
  }
}

}  // namespace

// lists of the k+1 target rows of every sequence, or of all block rows of a small batch
size_t verify_filter_scratch_bytes(int max_batch, int k_max) {
  const int rows = max_batch * (k_max + 1);
  return (size_t)(rows > FILT_BOTH_ROWS ? rows : FILT_BOTH_ROWS) * FILT_MAX_CHUNKS * FILT_MAX_K * sizeof(unsigned long long);
}

// cm != nullptr: the commit rides along
int launch_verify_filtered(space_ctx* ctx, const space_verify_args* a, const space_commit_args* cm, cudaStream_t st) {
  if (a->top_k < 1 || a->top_k > FILT_MAX_K || !(a->top_p > 0.f) || a->top_p > 1.f) return SPACE_E_INVALID_ARG;
  FiltParams p;
  memset(&p, 0, sizeof(p));
  p.B = a->batch; p.k = a->k; p.V = a->vocab; p.n_q = (a->k + 1) * (a->k + 1);
  p.top_k = a->top_k < a->vocab ? a->top_k : a->vocab; p.top_p = a->top_p;
  p.resample = a->resample; p.eos_id = a->eos_id;
  p.c_t = 1.4426950408889634f / a->temperature;
  p.key0 = (uint32_t)(a->seed & 0xFFFFFFFFull); p.key1 = (uint32_t)(a->seed >> 32);
  p.logits = a->logits; p.row_stride = a->logits_row_stride;
  p.cand = a->cand; p.cand_prob = a->cand_prob; p.seq_id = a->seq_id; p.kv_len = a->kv_len;
  p.n_accept = a->n_accept; p.out_tokens = a->out_tokens; p.n_out = a->n_out; p.next_cand = a->next_cand;
  p.next_cand_prob = a->next_cand_prob; p.finished = a->finished; p.status = a->status;
  p.draft_tok = a->draft_tok; p.draft_prob = a->draft_prob;
  p.next_draft_tok = a->next_draft_tok; p.next_draft_prob = a->next_draft_prob; p.list_stride = a->top_k;
  p.part = reinterpret_cast<unsigned long long*>(ctx->vtopk);
  const int esz = a->logits_dtype == SPACE_DTYPE_F32 ? 4 : 2;
  const bool aligned = ((uintptr_t)a->logits % 16 == 0) && ((a->logits_row_stride * esz) % 16 == 0);
  if (cm) fill_commit_params(ctx, cm, &p.cm);
  const int64_t block_rows = (int64_t)a->batch * p.n_q;
  const int64_t row_bytes = (int64_t)a->vocab * esz;
  bool both = block_rows <= FILT_BOTH_ROWS && block_rows * row_bytes <= FILT_BOTH_BYTES;
  if (!both && block_rows <= FILT_FEW_ROWS && block_rows * row_bytes <= FILT_FEW_ROWS_BYTES) {
    const int vec = 16 / esz;
    auto sweeps = [&](int64_t rows, int64_t* blocks) {     // that a block takes over its chunk in a launch of so many rows
      int chunk;
      *blocks = rows * row_chunks(a->vocab, (int)rows, vec, ctx->sm_count, FILT_MAX_CHUNKS, &chunk);
      return (chunk + FILT_THREADS * vec * FILT_U - 1) / (FILT_THREADS * vec * FILT_U);
    };
    int64_t blocks, unused;
    const int one = sweeps(block_rows, &blocks);
    const int two = sweeps((int64_t)a->batch * (a->k + 1), &unused) + sweeps((int64_t)a->batch * a->k, &unused);
    both = aligned ? blocks <= row_chunk_slots(ctx->sm_count) : blocks <= 3 * (int64_t)ctx->sm_count && one <= two + 1;
  }
  // the commit rides along, except where one block would have more than 32 KB of rows to move: a launch of its
  // own is faster then (two sequences, one launch; us per step, riding / own: 16 KB 22.1 / 23.7, 32 KB 25.8 / 26.1,
  // 57 KB 29.8 / 28.5)
  const bool carry = cm && !(both && (int64_t)a->k * p.cm.H_kv * p.cm.d * 4 > (32 << 10));
  for (int phase = both ? PHASE_BOTH : PHASE_TARGETS; phase <= (both ? PHASE_BOTH : PHASE_MASKS); ++phase) {
    p.phase = phase;
    p.do_commit = carry && phase != PHASE_TARGETS;
    p.counter = ctx->counters + (phase == PHASE_MASKS ? ctx->cfg.max_batch : 0);
    const int rows = phase == PHASE_TARGETS ? a->k + 1 : phase == PHASE_MASKS ? a->k : p.n_q;
    p.n_chunks = row_chunks(a->vocab, a->batch * rows, 16 / esz, ctx->sm_count, FILT_MAX_CHUNKS, &p.chunk);
    const dim3 grid(p.n_chunks, rows, a->batch);
    ProfScope ps(ctx, phase == PHASE_MASKS ? SPACE_K_VERIFY_EMIT : SPACE_K_VERIFY_TARGET, st);
    if (a->logits_dtype == SPACE_DTYPE_F32) {
      if (aligned) launch_pdl(verify_filter_kernel<float, true>, grid, dim3(FILT_THREADS), 0, st, p);
      else launch_pdl(verify_filter_kernel<float, false>, grid, dim3(FILT_THREADS), 0, st, p);
    } else {
      if (aligned) launch_pdl(verify_filter_kernel<__nv_bfloat16, true>, grid, dim3(FILT_THREADS), 0, st, p);
      else launch_pdl(verify_filter_kernel<__nv_bfloat16, false>, grid, dim3(FILT_THREADS), 0, st, p);
    }
    ctx->launches += 1;
  }
  if (cm && !carry) return launch_commit(ctx, cm, st);
  return cuda_ok(cudaGetLastError());
}
