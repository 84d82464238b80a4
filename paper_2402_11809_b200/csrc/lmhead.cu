// Output projection fused with verification, greedy or sampling (Algorithm 1: the end of the
// model call P = M(I) and the loop after it).
//
// logits[r, x] = <h_r, W_x> for the (k+1)^2 block rows of every sequence and the
// whole vocabulary, but the logits never reach memory: the products run on the
// tensor cores into fp32 accumulators in TMEM.  Two orientations, by the number of rows
// (launch_group has the rule and what was measured):
//   rows on M    A = hidden rows, B = up to 256 rows of W; lane = block row, column = token.
//                Four epilogue threads share one block row (two beyond 128 rows).
//   tokens on M  A = 128 rows of W (two accumulators per box), B = hidden rows; lane = token,
//                column = block row.  The epilogue turns eight rows of a warp's 32 tokens at
//                a time through shared memory and folds them with four lanes per row.
// Either way an epilogue thread folds its tokens of a row into (max, lowest arg-max,
// sum exp(z - max)) in registers, and a row's threads meet once, at the end of the
// block's range.  The last thread block to finish combines the vocabulary ranges and runs the acceptance scan, the extra
// token, the <EOS> cut and the next candidates.
//
// The output embedding is streamed exactly once (the step's HBM roof) for up to 256 block rows, by phase beyond
// (the target rows of every sequence, then the mask rows of its group i*); the hidden rows are re-read from L2
// by every thread block.
//
// Vocabulary ranges: thread block c owns rows [V*c/G, V*(c+1)/G) and covers them
// with boxes of n_box rows (256, or the longest range rounded up to 16 when that
// is shorter); the last box of a range is loaded through a second tensor map
// whose box holds only the rows a range's tail can have, so a range reads at
// most 15 rows of its neighbour.
//
// Warps: 0 TMA producer, 1 TMEM owner and MMA issuer, 2..17 epilogue (four per TMEM
// lane quarter).  With at most 128 block rows two accumulators alternate
// between boxes so that the epilogue of one box runs under the products of the
// next.  Every wait is bounded; an expired wait sets SPACE_ST_TIMEOUT, the block
// drains and exits.
#include "common.cuh"
#include "tc_common.cuh"
#include <cuda.h>
#include <math_constants.h>

namespace {

constexpr int LM_EPI = 16;                  // epilogue warps: four per TMEM lane quarter
constexpr int LM_EPI_T = 32 * LM_EPI;
constexpr int LM_THREADS = 64 + LM_EPI_T;
constexpr int LM_M = 128;                   // block rows per accumulator (MMA M)
constexpr int LM_MAX_BOX = 256;             // vocabulary rows per box (MMA N), at most
constexpr int LM_KB = 64;                   // hidden elements per slice (128 bytes: one swizzle row)
constexpr int LM_MAX_STAGES = 10;
constexpr int LM_L2_AHEAD = 8;              // slices of W a block asks L2 for before its dependency wait (4: two thirds of the gain)
constexpr float LM_NEG = -3.0e38f;          // "no logit yet": finite, so that differences never give NaN
constexpr int LM_MAX_N = 256;               // block rows of the whole batch, padded to 16
constexpr int LM_TOK = 128;                 // tokens per accumulator with the tokens on M
constexpr int LM_XP_PITCH = 36;             // floats per row of a warp's transposing buffer (8 rows of 32 tokens)
// Which block rows a launch projects: all of them, the target rows of every sequence that decide on its candidates (row
// b n + t: n = k+1 greedy, whose extra token is row i*'s arg-max; n = k in sampling mode, where nothing asks for row k), or
// the mask rows of every sequence's group i* (row bk+o-1; i* is the launch before's result) and, in sampling mode, target
// row i* of every sequence once more (row Bk+b): the extra token is drawn there, so that only one target row per
// sequence needs noise, not every one that could turn out to be row i*.
enum { LM_ALL = 0, LM_TARGETS = 1, LM_MASKS = 2 };
// rows gathered for the second phase: all that an accumulator holds, up to D = 16384 (fewer sequences at a time beyond).
// Of half the size it cut sampling batches beyond D = 8192 into more groups, two passes over the embedding each, with k + 1
// rows of a sequence than with k (12 sequences, k = 5, D = 16384, V = 16000: 368 us in bursts in two groups, 200 in one).
constexpr int64_t LM_GATHER_ELEMS = 128 * 16384;
constexpr uint64_t LM_WAIT_NS = 1000000000ull;
constexpr float LOG2E = 1.4426950408889634f;

struct LmPartial { float m, s; int idx, pad; };   // 16 bytes
struct LmNoisy { float gs, gz; int gidx, pad; };   // best noisy score of a range, the logit that has it, its token

struct LmParams {
  CUtensorMap tm_w, tm_wt, tm_h;   // W in boxes of n_box rows, W in boxes of tail_rows rows, hidden rows
  int B, k, V, D, n_q;
  int phase;                  // LM_*
  int n_rows;                 // rows of the launch (B * n_q when it takes all)
  int n_pad;                  // n_rows rounded up to 16: rows of the hidden-state tile
  int n_mt;                   // accumulators of 128 block rows (1 or 2)
  int stages;
  int n_box;                  // rows of the first tensor map's box (N of its products)
  int tail_rows;              // rows of the second tensor map's box
  int kbs;                    // 64-element slices of the hidden dimension per stage
  int backwards;              // a box's stages are taken from the hidden dimension's end (see launch_group)
  int targets;                // rows of a sequence in a launch over the target rows
  int h_bytes;                // of the hidden rows' box per 64-element slice
  int sums;                   // whether any row's sum of exponentials is asked for
  int n_noisy, noise_tok;     // sampling: rows that draw a token, tokens of a box whose noise is tabulated (a multiple of 16)
  int eos_id;
  int mode, resample;         // SPACE_MODE_*, SPACE_RESAMPLE_*
  float c_t;                  // log2(e) / T: exponent scale of the sums and of the noisy scores (sampling)
  uint32_t key0, key1;        // Philox key
  uint32_t seq_base;          // sequence id of the group's first sequence when seq_id is NULL
  const float* cand_prob; const uint32_t* seq_id; const int32_t* kv_len;
  LmNoisy* gpart;             // [n_rows][gridDim.x] (sampling)
  float* zc;                  // [n_rows] logit of the candidate a target row scores, written by the block that owns the token
  const int32_t* cand;
  int32_t* n_accept; int32_t* out_tokens; int32_t* n_out; int32_t* next_cand;
  float* next_cand_prob; uint8_t* finished; int32_t* status;
  float* row_max; int32_t* row_argmax;
  LmPartial* part;            // [n_rows][gridDim.x]
  unsigned long long* keys;   // [n_rows] arg-max keys, combined with atomicMax; zero between launches
  int* counter;               // arrival counter (self-resetting)
  int* err;
};

// PTX helpers: tc_common.cuh.  Every wait of this kernel is bounded by LM_WAIT_NS.
// `backoff`: sleep between polls (the epilogue warps, which wait for a whole group of products).
using namespace tc;
__device__ __noinline__ bool mbar_wait_long(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err, int site,
                                            bool backoff) {
  return mbar_wait_bounded(bar, parity, abort_flag, err, site, LM_WAIT_NS, backoff ? 128u : 0u);
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err, int site,
                                          bool backoff = false) {
  return mbar_try(bar, parity) || mbar_wait_long(bar, parity, abort_flag, err, site, backoff);   // (see mbar_wait_bounded)
}
__device__ __noinline__ void mbar_drain(uint32_t bar, uint32_t parity) { mbar_drain_bounded(bar, parity, LM_WAIT_NS); }
// Shared-memory matrix descriptor: K-major rows of 128 bytes, 128-byte swizzle
// (groups of 8 rows 1024 bytes apart), descriptor version of sm_100.
__device__ __forceinline__ uint64_t smem_desc_k128(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((16u >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((1024u >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
// Instruction descriptor: bf16 x bf16 -> f32, M = 128, N = n, both operands K-major.
__device__ __forceinline__ uint32_t instr_desc(int n) {                  // (M = 128 either way)
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(LM_M >> 4) << 24);
}
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_ld8(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr) : "memory");
}
__device__ __forceinline__ void epi_sync() { asm volatile("bar.sync 1, %0;" ::"n"(LM_EPI_T) : "memory"); }

// (maximum, lowest token) of a row as one 64-bit key whose unsigned order is "larger logit
// first, then lower token": the ranges of all thread blocks combine with one atomicMax each.
// 0 is below every key of a real logit.
__device__ __forceinline__ unsigned long long argmax_key(float m, int idx) {
  uint32_t u = __float_as_uint(m);
  u = (u & 0x80000000u) ? ~u : (u | 0x80000000u);
  return ((unsigned long long)u << 32) | (unsigned long long)(0xFFFFFFFFu - (uint32_t)idx);
}
__device__ __forceinline__ void argmax_unkey(unsigned long long key, float& m, int& idx) {
  uint32_t u = (uint32_t)(key >> 32);
  u = (u & 0x80000000u) ? (u & 0x7FFFFFFFu) : ~u;
  m = __uint_as_float(u);
  idx = (int)(0xFFFFFFFFu - (uint32_t)key);
}

// Fold N consecutive tokens x0 .. x0+N-1 (the first nv of them valid, at least one) into a row's statistics: sums of
// exp2((z - max) c).
template <int N>
__device__ __forceinline__ void fold(float& m, float& s, int& idx, const float (&z)[N], int x0, float c) {
  float cm = z[0];
#pragma unroll
  for (int j = 1; j < N; ++j) cm = fmaxf(cm, z[j]);
  if (cm > m) {                                           // strictly larger: an earlier token keeps a tie
    int at = N - 1;
#pragma unroll
    for (int j = N - 2; j >= 0; --j) at = (z[j] == cm) ? j : at;
    idx = x0 + at;
    s *= fast_exp2((m - cm) * c);
    m = cm;
  }
  const float ms = -m * c;
  float a0 = 0.f, a1 = 0.f, a2 = 0.f, a3 = 0.f;
#pragma unroll
  for (int j = 0; j < N; j += 4) {
    a0 += fast_exp2(fmaf(z[j], c, ms));
    a1 += fast_exp2(fmaf(z[j + 1], c, ms));
    a2 += fast_exp2(fmaf(z[j + 2], c, ms));
    a3 += fast_exp2(fmaf(z[j + 3], c, ms));
  }
  s += (a0 + a1) + (a2 + a3);
}

template <int N>
__device__ __forceinline__ void fold_max(float& m, int& idx, const float (&z)[N], int x0) {
  float cm = z[0];
#pragma unroll
  for (int j = 1; j < N; ++j) cm = fmaxf(cm, z[j]);
  if (cm > m) {
    int at = N - 1;
#pragma unroll
    for (int j = N - 2; j >= 0; --j) at = (z[j] == cm) ? j : at;
    idx = x0 + at;
    m = cm;
  }
}

// What an epilogue thread keeps of one block row in sampling mode, and what it has to know of the row.
struct RowNoisy {
  float gs, gz; int gidx;     // best noisy score so far, the logit that has it, its token
  float zc;                   // logit of the candidate this (target) row scores
};
struct RowConst {
  int cand_tok;               // that candidate, or -1
  int exclude;                // token left out of the draw (the rejected point-mass candidate), or -1
  uint32_t purpose, seq, pos; // Philox counter words of this row's noise
  int noisy;                  // this row's place among the rows that draw a token at all, or -1
  int pad[2];
};

// Noise of the four tokens of Philox block `block`: that of token x is lane x & 3 of the block with counter word
// x >> 2, as in the verification kernels.
__device__ __forceinline__ float4 noise4(uint32_t block, const RowConst& rc, uint32_t key0, uint32_t key1) {
  const Philox4 ph = philox4x32_10(block, rc.purpose, rc.seq, rc.pos, key0, key1);
  return make_float4(gumbel2_from_uniform(uniform_open(ph.x)), gumbel2_from_uniform(uniform_open(ph.y)),
                     gumbel2_from_uniform(uniform_open(ph.z)), gumbel2_from_uniform(uniform_open(ph.w)));
}

// What sampling keeps of N consecutive tokens x0 .. x0+N-1 (x0 a multiple of 4, the first nv valid) besides: the
// candidate's own logit when it lies here, and the best Gumbel-perturbed score z c + noise(token), with the noise from
// `table` or (nullptr) worked out here.  One branch for all N of them: with one per Philox block their chains did not
// run under one another (us per call in bursts, V = 128256, D = 2048, every row drawing, so that most of the noise is
// worked out here: 7 x 36 rows 173.5 / 167.2, 9 x 25 rows 173.0 / 166.7, 4 x 64 rows 170.8 / 164.6; V = 50257, D = 1024,
// 7 x 36 rows 68.7 / 66.1; one row in k + 1 drawing, 60 x 4 rows of V = 128256 167.4 / 162.4).
template <int N>
__device__ __forceinline__ void fold_noisy(RowNoisy& r, const RowConst& rc, const float (&z)[N], int x0, int nv, float c,
                                           uint32_t key0, uint32_t key1, const float* table) {
  if ((unsigned)(rc.cand_tok - x0) < (unsigned)N) {
#pragma unroll
    for (int j = 0; j < N; ++j) if (x0 + j == rc.cand_tok) r.zc = z[j];
  }
  if (rc.noisy < 0) return;
  auto score = [&](int i, const float4& g) {               // tokens 4i .. 4i+3
    const float gg[4] = {g.x, g.y, g.z, g.w};
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int j = 4 * i + l;
      const float sc = fmaf(z[j], c, gg[l]);
      if (j < nv && x0 + j != rc.exclude && sc > r.gs) { r.gs = sc; r.gidx = x0 + j; r.gz = z[j]; }
    }
  };
  if (table) {
#pragma unroll
    for (int i = 0; i < N / 4; ++i) score(i, reinterpret_cast<const float4*>(table)[i]);
  } else {
#pragma unroll
    for (int i = 0; i < N / 4; ++i) score(i, noise4((uint32_t)((x0 >> 2) + i), rc, key0, key1));
  }
}

// Row `row` of a launch: target row t (o = 0) or mask row (t, o) of sequence b.  False: padding.
__device__ __forceinline__ bool row_place(const LmParams& p, int row, int& b, int& t, int& o) {
  if (row >= p.n_rows) return false;
  const int k1 = p.k + 1;
  if (p.phase == LM_ALL) {
    b = row / p.n_q;
    const int i = row - b * p.n_q;
    t = i / k1; o = i - t * k1;
    return true;
  }
  if (p.phase == LM_TARGETS) { b = row / p.targets; t = row - b * p.targets; o = 0; return true; }
  if (row < p.B * p.k) { b = row / p.k; o = row - b * p.k + 1; }
  else { b = row - p.B * p.k; o = 0; }
  t = max(0, min(p.n_accept[b], p.k));                      // (a first pass that gave up has left it as it was)
  return true;
}

// Per-row constants of the sampling mode; target rows score candidate c_{t+1} and draw the extra token of the
// case i* = t at position L+t+1 (by phase, the first pass scores and the second draws, from row i* alone); mask rows (t, o) draw candidate o of that case at position
// L+t+1+o when candidates are sampled (Algorithm 1 as printed).
__device__ __forceinline__ RowConst row_const(const LmParams& p, int row) {
  RowConst r{-1, -1, 0u, 0u, 0u, -1, {0, 0}};
  int b, t, o;
  if (!row_place(p, row, b, t, o)) return r;
  const bool literal = p.resample == SPACE_RESAMPLE_PAPER_LITERAL;
  r.seq = p.seq_id ? p.seq_id[b] : p.seq_base + (uint32_t)b;
  const int L = p.kv_len ? p.kv_len[b] : 0;
  if (o == 0) {
    r.purpose = PURPOSE_TOKEN; r.pos = (uint32_t)(L + t + 1);
    if (p.phase != LM_TARGETS) r.noisy = literal ? row : p.phase == LM_MASKS ? b : b * (p.k + 1) + t;
    if (t < p.k) {
      const int tok = p.cand[b * p.k + t];
      if (p.phase != LM_MASKS) r.cand_tok = tok;
      if (!literal && p.cand_prob[b * p.k + t] == 1.0f) r.exclude = tok;          // residual of a point mass
    }
  } else if (literal) {
    r.purpose = PURPOSE_DRAFT; r.pos = (uint32_t)(L + t + 1 + o);
    r.noisy = row;
  }
  return r;
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xFFFFFFFFu, v, off);
  return v;
}

// Shared-memory plan (dynamic, 1024-byte aligned base):
//   [stages]{ [kbs] hidden tiles of n_pad*128 bytes, [kbs] W tiles of n_box*128 bytes } | pad |
//   (tokens on M: the epilogue warps' transposing buffers) | (sampling: the rows' constants, the noise table) |
//   barriers | row results [n_pad] x 2 | candidates | misc
// A product reads 128 rows of its first operand whatever the tile holds: the rows past the
// tile are whatever follows in shared memory (other tiles, then `pad`) and only reach
// accumulator lanes nobody reads.  `pad` keeps that read inside the allocation.
struct LmSmem {
  uint32_t a_bytes, b_bytes, b_in_stage, stage_bytes, xp_off, rowc_off, noise_off, bar_off, row_off, cand_off, misc_off, total;
  __host__ __device__ LmSmem(bool tokens_on_m, bool sample, int n_noisy, int noise_tok, int n_pad, int n_box, int stages, int kbs) {
    a_bytes = (uint32_t)n_pad * LM_KB * 2;
    b_bytes = (uint32_t)n_box * LM_KB * 2;
    b_in_stage = (uint32_t)kbs * a_bytes;
    stage_bytes = b_in_stage + (uint32_t)kbs * b_bytes;
    // bytes the products read from the last tile of their first operand, and bytes that follow its start
    const uint32_t reach = 16384u * (tokens_on_m ? (n_box > LM_TOK ? 2u : 1u) : (n_pad > LM_M ? 2u : 1u));
    const uint32_t have = tokens_on_m ? b_bytes : a_bytes + (uint32_t)kbs * b_bytes;
    const uint32_t pad = reach > have ? (reach - have + 1023u) / 1024u * 1024u : 0u;
    xp_off = (uint32_t)stages * stage_bytes + pad;
    rowc_off = xp_off + (tokens_on_m ? LM_EPI * 8u * LM_XP_PITCH * 4u : 0u);
    noise_off = rowc_off + (sample ? (uint32_t)n_pad * (uint32_t)sizeof(RowConst) : 0u);
    bar_off = noise_off + (sample && noise_tok ? (uint32_t)n_noisy * (uint32_t)(noise_tok + 4) * 4u : 0u);
    row_off = bar_off + 8u * (2 * LM_MAX_STAGES + 4);
    cand_off = row_off + 2u * 4u * (uint32_t)n_pad;                      // candidates of the batch: fewer than n_pad
    misc_off = cand_off + 4u * (uint32_t)n_pad;
    total = misc_off + 64u;
  }
};

// TM: tokens on the M extent, block rows on N, greedy calls only (see the file header and launch_group's rule).
template <bool TM, bool SAMPLE>
__global__ void __launch_bounds__(LM_THREADS, 1) lmhead_verify_kernel(const __grid_constant__ LmParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  const uint32_t sm_base = smem_u32(smem_raw);
  const LmSmem L(TM, SAMPLE, p.n_noisy, p.noise_tok, p.n_pad, p.n_box, p.stages, p.kbs);
  static_assert(!TM || !SAMPLE, "sampling keeps the rows on M");
  constexpr bool sample = SAMPLE;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int S = p.stages;
  const uint32_t bar0 = sm_base + L.bar_off;
#define LBAR(i) (bar0 + 8u * (uint32_t)(i))
  const int B_FULL = 0, B_EMPTY = LM_MAX_STAGES, B_ACCFULL = 2 * LM_MAX_STAGES, B_ACCEMPTY = 2 * LM_MAX_STAGES + 2;
  float* row_s = reinterpret_cast<float*>(smem_raw + L.row_off);           // [n_pad]
  int* row_i = reinterpret_cast<int*>(row_s + p.n_pad);
  int* cand_s = reinterpret_cast<int*>(smem_raw + L.cand_off);            // [B * k]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(smem_raw + L.misc_off);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(smem_raw + L.misc_off + 4);
  int* last_flag = reinterpret_cast<int*>(smem_raw + L.misc_off + 8);

  pdl_launch_dependents();
  if (threadIdx.x == 0) {
    *abort_flag = (sm_base & 1023u) ? 1 : 0;               // swizzled tiles need a 1024-byte aligned base
    for (int s = 0; s < S; ++s) { mbar_init(LBAR(B_FULL + s), 1); mbar_init(LBAR(B_EMPTY + s), 1); }
    for (int a = 0; a < 2; ++a) { mbar_init(LBAR(B_ACCFULL + a), 1); mbar_init(LBAR(B_ACCEMPTY + a), LM_EPI); }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp == 0 && lane == 0) {
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.tm_w) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.tm_wt) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.tm_h) : "memory");
  }
  if (warp == 0 && lane == 0) {
    // With a programmatic launch the block is resident before its dependency wait returns: ask L2 for its
    // first slices of W meanwhile (a request to the point of coherence, so whatever the kernel before still
    // writes is what the loads will see).  V = 32000, D = 4096, 36 rows: 51.3 -> 49.8 us per call in bursts, 53.5 ->
    // 53.2 in a steady loop, where the power cap sets the pace.
    // (Backwards, the launch before has just read the first slices.)
    const int first = (int)(((long long)p.V * blockIdx.x) / gridDim.x) & ~15;
    const uint64_t pol = l2_evict_first_policy();
    for (int kb = 0; !p.backwards && kb < min(LM_L2_AHEAD, (p.D + LM_KB - 1) / LM_KB); ++kb)
      tma_prefetch_l2_4d(&p.tm_w, kb * LM_KB, first, 0, 0, pol);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();                                              // global memory from here on

  // this thread block's vocabulary range and its boxes
  const int G = gridDim.x, c = blockIdx.x;
  // (range boundaries are multiples of 16 tokens, so that a group of 16 accumulator columns
  // always starts on a Philox block)
  const int r0 = (int)(((long long)p.V * c) / G) & ~15;
  const int r1 = (c == G - 1) ? p.V : ((int)(((long long)p.V * (c + 1)) / G) & ~15);
  const int nb = (r1 - r0 + p.n_box - 1) / p.n_box;
  const int KB = (p.D + LM_KB - 1) / LM_KB;
  const int kbs = p.kbs;
  const int KI = (KB + kbs - 1) / kbs;                     // stages per box
  auto first_slice = [&](int ki) { return (p.backwards ? KI - 1 - ki : ki) * kbs; };   // of a box's ki-th stage
  const int n_bufs = p.n_mt == 1 ? 2 : 1;                  // accumulator buffers of n_mt x 256 columns
  const int acc_cols = TM ? p.n_mt * LM_TOK : 0;           // (tokens on M: columns of one of a buffer's two accumulators)

  if (warp == 0) {
    // ================= producer ==============================================
    if (elect_one()) {
      bool ok = !*abort_flag;
      // (the ring's place is kept as a stage and a phase bit: divisions by the run-time stage count took
      // longer than the requests they were for, on the one thread every stage waits for)
      uint32_t it = 0, s = 0, empty_phase = 1;               // the first pass over the ring finds it free
      for (int box = 0; box < nb && ok; ++box) {
        const int row0 = r0 + box * p.n_box;
        const bool tail = r1 - row0 <= p.tail_rows;          // the remaining rows fit the small box
        const CUtensorMap* tm = tail ? &p.tm_wt : &p.tm_w;
        const uint32_t slice_bytes = (uint32_t)(tail ? p.tail_rows : p.n_box) * LM_KB * 2 + (uint32_t)p.h_bytes;
        for (int ki = 0; ki < KI; ++ki, ++it) {
          const int kb0 = first_slice(ki);
          // stage `it`: the W tiles and the hidden tiles of its slices
          if (it >= (uint32_t)S) ok = mbar_wait(LBAR(B_EMPTY + s), empty_phase, abort_flag, p.err, 1);
          if (!ok) break;
          const int nk = min(kbs, KB - kb0);
          const uint32_t st_base = sm_base + s * L.stage_bytes;
          mbar_expect_tx(LBAR(B_FULL + s), (uint32_t)nk * slice_bytes);
          for (int j = 0; j < nk; ++j)
            tma_load_4d(st_base + L.b_in_stage + (uint32_t)j * L.b_bytes, tm, LBAR(B_FULL + s), (kb0 + j) * LM_KB, row0, 0, 0);
          for (int j = 0; j < nk; ++j)
            tma_load_4d(st_base + (uint32_t)j * L.a_bytes, &p.tm_h, LBAR(B_FULL + s), (kb0 + j) * LM_KB, 0, 0, 0);
          if (++s == (uint32_t)S) { s = 0; empty_phase ^= 1; }
        }
      }
      if (!ok) {
        // copies already requested still land: wait for them (bounded) before the block exits
        const uint32_t first = it > (uint32_t)S ? it - S : 0;
        for (uint32_t j = first; j < it; ++j) mbar_drain(LBAR(B_FULL + j % S), (j / S) & 1);
      }
    }
  } else if (warp == 1) {
    // ================= MMA issuer =============================================
    if (elect_one()) {
      const uint64_t desc0 = smem_desc_k128(sm_base);
      uint32_t s = 0, full_phase = 0;
      int buf = 0;
      bool ok = !*abort_flag;
      for (int box = 0; box < nb && ok; ++box) {
        const int row0 = r0 + box * p.n_box;
        const uint32_t idesc = instr_desc(TM ? p.n_pad : (r1 - row0 <= p.tail_rows) ? p.tail_rows : p.n_box);
        const int n_tt = (min(r1 - row0, p.n_box) + LM_TOK - 1) / LM_TOK;   // (tokens on M: accumulators of this box)
        // (the buffer's user before this one: box - n_bufs)
        if (box >= n_bufs) ok = mbar_wait(LBAR(B_ACCEMPTY + buf), (n_bufs == 2 ? (box >> 1) - 1 : box - 1) & 1, abort_flag, p.err, 2);
        if (!ok) break;
        tc_fence_after();
        for (int ki = 0; ki < KI; ++ki) {
          const int kb0 = first_slice(ki);
          const int nk = min(kbs, KB - kb0);
          ok = mbar_wait(LBAR(B_FULL + s), full_phase, abort_flag, p.err, 3);
          if (!ok) break;
          tc_fence_after();
          const uint32_t st_off = s * L.stage_bytes;
          for (int j = 0; j < nk; ++j) {
            const uint64_t wd = desc0 + (uint64_t)((st_off + L.b_in_stage + (uint32_t)j * L.b_bytes) >> 4);
            if (TM) {
              const uint64_t hd = desc0 + (uint64_t)((st_off + (uint32_t)j * L.a_bytes) >> 4);
              for (int tt = 0; tt < n_tt; ++tt) {
                const uint32_t acc = tmem + (uint32_t)((buf * 2 + tt) * acc_cols);
#pragma unroll
                for (int kk = 0; kk < LM_KB / 16; ++kk)
                  mma_ss(acc, wd + (uint64_t)(tt * (16384 >> 4) + kk * 2), hd + (uint64_t)(kk * 2), idesc, (ki | j | kk) ? 1u : 0u);
              }
            } else {
              for (int mt = 0; mt < p.n_mt; ++mt) {
                // block rows 128*mt .. of the hidden tile (8-row groups are contiguous: 16 KB further on)
                const uint64_t hd = desc0 + (uint64_t)((st_off + (uint32_t)j * L.a_bytes + (uint32_t)mt * 16384u) >> 4);
                const uint32_t acc = tmem + (uint32_t)((buf * p.n_mt + mt) * LM_MAX_BOX);
#pragma unroll
                for (int kk = 0; kk < LM_KB / 16; ++kk)    // 32 bytes per 16 elements inside the swizzled row
                  mma_ss(acc, hd + (uint64_t)(kk * 2), wd + (uint64_t)(kk * 2), idesc, (ki | j | kk) ? 1u : 0u);
              }
            }
          }
          tc_commit(LBAR(B_EMPTY + s));
          if (++s == (uint32_t)S) { s = 0; full_phase ^= 1; }
        }
        if (ok) tc_commit(LBAR(B_ACCFULL + buf));
        buf = n_bufs == 2 ? buf ^ 1 : 0;
      }
    }
  } else {
    // ================= epilogue ================================================
    const int quarter = warp & 3;                          // TMEM lanes 32*quarter .. +31
    const int ew = warp - 2;
    // the candidates are an input: fetched now, so that the last block's scan does not wait for them
    for (int t = threadIdx.x - 64; t < p.B * p.k; t += LM_EPI_T) cand_s[t] = p.cand[t];
    // Sampling: the noise does not depend on the logits, and while the products run the epilogue warps have nothing
    // else to do.  So they work it out for a box before they wait for its accumulators, spread over all threads,
    // where the folds would do it for 32 rows in step although only every (k+1)-th of them draws a token, after
    // the last product, with the whole chip waiting.  D = 4096, bursts, in the folds / tabulated: one sequence of 36 rows,
    // V = 32000, 56.9 / 52.9 us, V = 128256 (D = 2048) 92.7 / 87.3, 144 rows of V = 32000 69.9 / 66.2, of V = 20000 (D = 2048)
    // 37.7 / 33.2.  (A launch whose rows draw nothing, as the first of two by phase, has no table; what the stages leave no
    // room for, up to all of it, the folds work out.)
    RowConst* rowc = reinterpret_cast<RowConst*>(smem_raw + L.rowc_off);
    float* noise = reinterpret_cast<float*>(smem_raw + L.noise_off);       // [n_noisy][noise_tok + 4]
    const int noise_pitch = p.noise_tok + 4;
    if (sample) {
      for (int row = threadIdx.x - 64; row < p.n_pad; row += LM_EPI_T) rowc[row] = row_const(p, row);
      epi_sync();
    }
    auto fill_noise = [&](int row0, int n_valid) {
      if (p.noise_tok == 0) return;
      epi_sync();                                            // (the table of the box before has been read)
      const int n4 = min(p.noise_tok, (n_valid + 15) & ~15) >> 2;
      for (int at = threadIdx.x - 64; at < p.n_noisy * n4; at += LM_EPI_T) {
        const int y = at / n4, q = at - y * n4;
        // row of the y-th noisy one (row_const says which those are)
        const int k1 = p.k + 1;
        const int row = p.resample == SPACE_RESAMPLE_PAPER_LITERAL ? y : p.phase == LM_MASKS ? p.B * p.k + y : y / k1 * p.n_q + y % k1 * k1;
        reinterpret_cast<float4*>(noise + y * noise_pitch)[q] = noise4((uint32_t)(row0 >> 2) + q, rowc[row], p.key0, p.key1);
      }
      epi_sync();
    };
    // statistics of other tokens of a row join (m0, s0, i0)
    auto join = [&](float& m0, float& s0, int& i0, float m2, float s2, int i2) {
      if (m2 > m0 || (m2 == m0 && i2 < i0)) i0 = i2;
      const float e = fast_exp2(-fabsf(m0 - m2) * p.c_t);    // (one of the two exponentials is exp(0))
      s0 = (m0 >= m2) ? fmaf(s2, e, s0) : fmaf(s0, e, s2);
      m0 = fmaxf(m0, m2);
    };
    if (TM) {
      // ---- tokens on M: lane = token, column = block row.  A warp reads 8 rows of its 32 tokens, turns them through
      // its shared-memory buffer and folds them with four lanes per row, eight tokens each.  The four warps of a lane
      // quarter take the groups of eight rows in turn, both accumulators of a box one after the other; what a lane
      // keeps of its up to eight rows stays in registers until the end of the range.
      constexpr int GP = LM_MAX_N / 8 / 4;
      const int part = ew >> 2, n_grp = p.n_pad >> 3;
      const int rl = lane & 7, tl = (lane >> 3) * 8;         // this lane's row of a group, its first token of the 32
      float* xp = reinterpret_cast<float*>(smem_raw + L.xp_off) + ew * (8 * LM_XP_PITCH);
      float m[GP], sm[GP];
      int id[GP];
#pragma unroll
      for (int i = 0; i < GP; ++i) { m[i] = LM_NEG; sm[i] = 0.f; id[i] = 0x7FFFFFFF; }
      bool ok = true;
      for (int box = 0; box < nb; ++box) {
        const int buf = n_bufs == 2 ? box & 1 : 0;
        ok = ok && mbar_wait(LBAR(B_ACCFULL + buf), (n_bufs == 2 ? box >> 1 : box) & 1, abort_flag, p.err, 4, true);
        ok = __all_sync(0xFFFFFFFFu, ok);
        if (!ok) break;
        tc_fence_after();
        const int row0 = r0 + box * p.n_box, n_valid = min(r1 - row0, p.n_box);
        const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(buf * 2 * acc_cols);
#pragma unroll
        for (int i = 0; i < GP; ++i) {
          const int g = part + 4 * i;
          if (g < n_grp) {
            uint32_t v[2][8];                                // (a second accumulator that the box does not use: never read on)
            tmem_ld8(acc + (uint32_t)(g * 8), v[0]);
            tmem_ld8(acc + (uint32_t)(acc_cols + g * 8), v[1]);
            tmem_wait_ld();
#pragma unroll
            for (int tt = 0; tt < 2; ++tt) {
              const int tok = tt * LM_TOK + quarter * 32;    // first token of this warp's lanes within the box
              if (tok >= n_valid) break;
#pragma unroll
              for (int j = 0; j < 8; ++j) xp[j * LM_XP_PITCH + lane] = __uint_as_float(v[tt][j]);
              __syncwarp();
              float z[8];
              *reinterpret_cast<float4*>(z) = *reinterpret_cast<const float4*>(xp + rl * LM_XP_PITCH + tl);
              *reinterpret_cast<float4*>(z + 4) = *reinterpret_cast<const float4*>(xp + rl * LM_XP_PITCH + tl + 4);
              __syncwarp();
              const int nv = n_valid - tok - tl, x0 = row0 + tok + tl;
              if (nv > 0) {
#pragma unroll
                for (int j = 1; j < 8; ++j) z[j] = (j < nv) ? z[j] : LM_NEG;
                fold(m[i], sm[i], id[i], z, x0, p.c_t);
              }
            }
          }
        }
        // this accumulator buffer may be overwritten by the products of the next box that uses it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(LBAR(B_ACCEMPTY + buf));
      }
      // ---- the four lanes of a row meet, then (through the idle stages: every product is done) the four quarters
      float* x = reinterpret_cast<float*>(smem_raw);         // [4][3][LM_MAX_N]
#pragma unroll
      for (int i = 0; i < GP; ++i) {
        const int g = part + 4 * i;
        if (g < n_grp) {
#pragma unroll
          for (int o = 8; o <= 16; o <<= 1)
            join(m[i], sm[i], id[i], __shfl_xor_sync(0xFFFFFFFFu, m[i], o), __shfl_xor_sync(0xFFFFFFFFu, sm[i], o),
                 __shfl_xor_sync(0xFFFFFFFFu, id[i], o));
          if (lane < 8) {
            float* y = x + quarter * 3 * LM_MAX_N + g * 8 + lane;
            y[0] = m[i]; y[LM_MAX_N] = sm[i]; y[2 * LM_MAX_N] = __int_as_float(id[i]);
          }
        }
      }
      epi_sync();
      // publish this block's statistics of every block row
      const int row = threadIdx.x - 64;
      if (row < p.n_rows) {
        float v[4][3];
#pragma unroll
        for (int q = 0; q < 4; ++q)
#pragma unroll
          for (int f = 0; f < 3; ++f) v[q][f] = x[(q * 3 + f) * LM_MAX_N + row];
        int i0 = __float_as_int(v[0][2]);
#pragma unroll
        for (int q = 1; q < 4; ++q) join(v[0][0], v[0][1], i0, v[q][0], v[q][1], __float_as_int(v[q][2]));
        LmPartial out; out.m = v[0][0]; out.s = v[0][1]; out.idx = i0; out.pad = 0;
        *reinterpret_cast<int4*>(p.part + (size_t)row * G + c) = *reinterpret_cast<const int4*>(&out);
        atomicMax(p.keys + row, argmax_key(v[0][0], i0));
      }
    } else {
      // The warps of a lane quarter share the accumulators, and take an accumulator's column groups in turn;
      // they meet at the end (with one warp per quarter its scan was what a call ended on, and what a sampling
      // call waited for all along).
      const int mt = (ew >> 2) % p.n_mt, n_parts = LM_EPI / 4 / p.n_mt, part = (ew >> 2) / p.n_mt;
      const int row = mt * LM_M + quarter * 32 + lane;       // this thread's block row
      float m0 = LM_NEG, s0 = 0.f;
      int i0 = 0x7FFFFFFF;
      RowNoisy n0{-CUDART_INF_F, 0.f, 0x7FFFFFFF, LM_NEG};
      RowConst rc{-1, -1, 0u, 0u, 0u, -1, {0, 0}};
      if (sample && row < p.n_pad) rc = rowc[row];
      // a warp whose 32 lanes hold no block row only takes part in the hand-shakes
      const bool has_rows = row - lane < p.n_rows;
      bool ok = true;
      for (int box = 0; box < nb; ++box) {
        const int buf = n_bufs == 2 ? box & 1 : 0;
        if (sample) fill_noise(r0 + box * p.n_box, min(r1 - r0 - box * p.n_box, p.n_box));
        ok = ok && mbar_wait(LBAR(B_ACCFULL + buf), (n_bufs == 2 ? box >> 1 : box) & 1, abort_flag, p.err, 4, true);
        ok = __all_sync(0xFFFFFFFFu, ok);
        tc_fence_after();
        const int row0 = r0 + box * p.n_box;
        const int n_valid = ok ? min(r1 - row0, (r1 - row0 <= p.tail_rows) ? p.tail_rows : p.n_box) : 0;
        const uint32_t acc = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)((buf * p.n_mt + mt) * LM_MAX_BOX);
        if (has_rows) {
          for (int c0 = 16 * part; c0 < n_valid; c0 += 16 * n_parts) {
            uint32_t v[16];
            tmem_ld16(acc + (uint32_t)c0, v);
            tmem_wait_ld();
            const int nv = n_valid - c0;
            float z[16];
#pragma unroll
            for (int j = 0; j < 16; ++j) z[j] = (j < nv) ? __uint_as_float(v[j]) : LM_NEG;
            if (!sample || p.sums) fold(m0, s0, i0, z, row0 + c0, p.c_t);
            else fold_max(m0, i0, z, row0 + c0);
            if (sample)
              fold_noisy(n0, rc, z, row0 + c0, nv, p.c_t, p.key0, p.key1,
                         c0 < p.noise_tok ? noise + rc.noisy * noise_pitch + c0 : nullptr);   // (both multiples of 16)
          }
        }
        // this accumulator buffer may be overwritten by the products of the next box that uses it
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(LBAR(B_ACCEMPTY + buf));
      }
      {
        // the other parts' columns join the first's (the pipeline stages are idle: every product is done)
        float* x = reinterpret_cast<float*>(smem_raw) + row;   // [n_parts - 1][7][2 LM_M]
        constexpr int W = 2 * LM_M;
        if (part > 0 && has_rows) {
          float* y = x + (part - 1) * 7 * W;
          y[0] = m0; y[W] = s0; y[2 * W] = __int_as_float(i0);
          if (sample) { y[3 * W] = n0.gs; y[4 * W] = n0.gz; y[5 * W] = __int_as_float(n0.gidx); y[6 * W] = n0.zc; }
        }
        epi_sync();
        if (part == 0 && has_rows) {
          for (int o = 1; o < n_parts; ++o) {
            const float* y = x + (o - 1) * 7 * W;
            join(m0, s0, i0, y[0], y[W], __float_as_int(y[2 * W]));
            if (sample) {
              const float g2 = y[3 * W];
              const int gi2 = __float_as_int(y[5 * W]);
              if (g2 > n0.gs || (g2 == n0.gs && gi2 < n0.gidx)) { n0.gs = g2; n0.gz = y[4 * W]; n0.gidx = gi2; }
              n0.zc = fmaxf(n0.zc, y[6 * W]);
            }
          }
        }
      }
      // publish this block's statistics of every block row
      if (row < p.n_rows && part == 0) {
        LmPartial out; out.m = m0; out.s = s0; out.idx = i0; out.pad = 0;
        *reinterpret_cast<int4*>(p.part + (size_t)row * G + c) = *reinterpret_cast<const int4*>(&out);
        atomicMax(p.keys + row, argmax_key(m0, i0));
        if (sample) {
          if (p.n_noisy) {
            LmNoisy g; g.gs = n0.gs; g.gz = n0.gz; g.gidx = n0.gidx; g.pad = 0;
            *reinterpret_cast<int4*>(p.gpart + (size_t)row * G + c) = *reinterpret_cast<const int4*>(&g);
          }
          if ((unsigned)(rc.cand_tok - r0) < (unsigned)(r1 - r0)) p.zc[row] = n0.zc;   // this block owns the candidate's token
        }
      }
    }
    epi_sync();
    const int et = threadIdx.x - 64;                       // 0 .. LM_EPI_T-1
    if (et == 0) {
      __threadfence();                                      // (the barrier ordered every thread's stores before this)
      const int prev = atomicAdd(p.counter, 1);
      const int last = prev == G - 1;
      if (last) { *p.counter = 0; __threadfence(); }       // ready for the next launch
      *last_flag = last;
    }
    epi_sync();
    if (*last_flag) {
      // ---- last thread block.  Every row's (maximum, arg-max) is already combined in its key;
      // only the k mask rows of group i* of every sequence need their sums, so only those rows'
      // per-range partials are read, all of them at once over the threads.
      const int k1 = p.k + 1;
      // the launch's rows of target t and of mask row (i*, j+1) of sequence b
      const bool with_targets = p.phase != LM_MASKS, with_masks = p.phase != LM_TARGETS;
      auto target_row = [&](int b, int t) { return p.phase == LM_ALL ? b * p.n_q + t * k1 : b * p.targets + t; };
      auto mask_row = [&](int b, int i_star, int j) { return p.phase == LM_ALL ? b * p.n_q + i_star * k1 + j + 1 : b * p.k + j; };
      float* row_m = row_s;                                // [n_rows] maxima (row_s is reused: sums come later)
      int* istar = reinterpret_cast<int*>(smem_raw);       // [B] (the pipeline stages are idle now)
      float* terms = reinterpret_cast<float*>(smem_raw) + LM_MAX_N;   // [B * k][G] scaled sums of the ranges
      for (int r = et; r < p.n_rows; r += LM_EPI_T) {
        const unsigned long long key = atomicExch(p.keys + r, 0ull);      // read, and ready for the next launch
        float m; int idx;
        argmax_unkey(key, m, idx);
        row_m[r] = m; row_i[r] = idx;
        if (p.row_max) p.row_max[r] = m;
        if (p.row_argmax) p.row_argmax[r] = idx;
      }
      epi_sync();
      if (sample) {
        // ---- sampling mode (Algorithm 1 with r <= Q/P_c; see verify.cu for the same steps on
        // stored logits).  tsum: sums of exp2((z - max) c) of the rows named by row_of(b, j),
        // j = 0..k-1, combined from the ranges' partials in a fixed order.
        const float cT = p.c_t;
        float* tsum = reinterpret_cast<float*>(smem_raw) + LM_MAX_N;        // [B * k]
        float* terms2 = tsum + LM_MAX_N;                                    // [B * k][G]
        const bool literal = p.resample == SPACE_RESAMPLE_PAPER_LITERAL;
        auto sum_rows = [&](bool mask_rows) {
          const int total = p.B * p.k * G;
          for (int i0 = et; i0 < total; i0 += LM_EPI_T * 8) {
            int4 v[8]; float mx[8];
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int at = i0 + u * LM_EPI_T;
              v[u] = make_int4(0, 0, 0, 0); mx[u] = 0.f;
              if (at < total) {
                const int g = at % G, bj = at / G;
                const int b = bj / p.k, jj = bj - b * p.k;
                const int row = mask_rows ? mask_row(b, istar[b], jj) : target_row(b, jj);
                mx[u] = row_m[row];
                v[u] = __ldcg(reinterpret_cast<const int4*>(p.part + (size_t)row * G + g));
              }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const int at = i0 + u * LM_EPI_T;
              if (at < total) terms2[at] = __int_as_float(v[u].y) * fast_exp2((__int_as_float(v[u].x) - mx[u]) * cT);
            }
          }
          epi_sync();
          for (int bj = ew; bj < p.B * p.k; bj += LM_EPI) {
            float sv = 0.f;
            for (int g = lane; g < G; g += 32) sv += terms2[bj * G + g];
            sv = warp_sum(sv);
            if (lane == 0) tsum[bj] = sv;
          }
          epi_sync();
        };
        // best noisy score of a row over the ranges: larger score, then lower token; every lane gets it
        auto best_noisy = [&](int row, float& gz_out) -> int {
          float gs = -CUDART_INF_F, gz = 0.f; int gi = 0x7FFFFFFF;
          for (int g = lane; g < G; g += 32) {
            const int4 v = __ldcg(reinterpret_cast<const int4*>(p.gpart + (size_t)row * G + g));
            const float s2 = __int_as_float(v.x);
            if (s2 > gs || (s2 == gs && v.z < gi)) { gs = s2; gz = __int_as_float(v.y); gi = v.z; }
          }
#pragma unroll
          for (int off = 16; off > 0; off >>= 1) {
            const float os = __shfl_xor_sync(0xFFFFFFFFu, gs, off);
            const float oz = __shfl_xor_sync(0xFFFFFFFFu, gz, off);
            const int oi = __shfl_xor_sync(0xFFFFFFFFu, gi, off);
            if (os > gs || (os == gs && oi < gi)) { gs = os; gz = oz; gi = oi; }
          }
          gz_out = gz;
          return gi;
        };
        // emitted tokens of a sequence (one warp): the candidates before i*, then the draw of row i*
        auto emit = [&](int b, int i_star, int cv) {
          float gz_unused;
          const int bonus = best_noisy(p.phase == LM_ALL ? target_row(b, i_star) : p.B * p.k + b, gz_unused);
          const int j = lane;
          const int c_j = __shfl_sync(0xFFFFFFFFu, cv, min(j, p.k - 1));
          const int tok = (j < i_star) ? c_j : (j == i_star ? bonus : -1);
          const bool is_eos = p.eos_id >= 0 && j <= i_star && tok == p.eos_id;
          const unsigned eos_mask = __ballot_sync(0xFFFFFFFFu, is_eos && j < k1);
          const int n_out = eos_mask ? __ffs(eos_mask) - 1 : i_star + 1;
          if (j < k1) p.out_tokens[b * k1 + j] = (j < n_out) ? tok : -1;
          if (j == 0) { p.n_out[b] = n_out; p.finished[b] = (uint8_t)(eos_mask != 0); }
        };
        if (with_targets) {
        sum_rows(false);                                   // target rows t = 0..k-1 of every sequence
        for (int b = ew; b < p.B; b += LM_EPI) {
          const int t = lane;
          const int cv = (t < p.k) ? cand_s[b * p.k + t] : -1;
          const bool in_range = cv >= 0 && cv < p.V;
          const unsigned bad = __ballot_sync(0xFFFFFFFFu, t < p.k && !in_range);
          bool okc = false;
          const uint32_t seq = p.seq_id ? p.seq_id[b] : p.seq_base + (uint32_t)b;
          const int Lb = p.kv_len ? p.kv_len[b] : 0;
          if (t < p.k && in_range) {
            const int row = target_row(b, t);
            const float zc = __ldcg(p.zc + row);
            const float q = fast_exp2((zc - row_m[row]) * cT) / tsum[b * p.k + t];
            const Philox4 w = philox4x32_10(0u, PURPOSE_ACCEPT, seq, (uint32_t)(Lb + t + 1), p.key0, p.key1);
            const float pc = p.cand_prob[b * p.k + t];
            okc = pc > 0.f && uniform_open(w.x) * pc <= q;  // r <= Q/P_c  <=>  r P_c <= Q
          }
          const unsigned acc_mask = __ballot_sync(0xFFFFFFFFu, okc);
          const int i_star = __ffs(~acc_mask) - 1;          // first candidate that is not accepted (k when all are)
          if (p.phase == LM_ALL) emit(b, i_star, cv);
          if (lane == 0) {
            istar[b] = i_star;
            p.n_accept[b] = i_star;
            if (p.status && bad) atomicOr(p.status + b, SPACE_ST_BAD_CANDIDATE);
          }
        }
        } else {
          for (int b = et; b < p.B; b += LM_EPI_T) istar[b] = max(0, min(p.n_accept[b], p.k));
          for (int b = ew; b < p.B; b += LM_EPI) emit(b, max(0, min(p.n_accept[b], p.k)), lane < p.k ? cand_s[b * p.k + lane] : -1);
        }
        epi_sync();
        if (with_masks && !literal) {                      // point-mass drafts: arg-max of mask row (i*, j+1), P_c = 1
          for (int bj = et; bj < p.B * p.k; bj += LM_EPI_T) {
            const int b = bj / p.k, j = bj - b * p.k;
            p.next_cand[bj] = row_i[mask_row(b, istar[b], j)];
            p.next_cand_prob[bj] = 1.f;
          }
        } else if (with_masks) {
          // candidates sampled from the mask rows of group i*, with their probabilities
          sum_rows(true);
          for (int bj = ew; bj < p.B * p.k; bj += LM_EPI) {
            const int b = bj / p.k, jj = bj - b * p.k;
            const int row = mask_row(b, istar[b], jj);
            float gz;
            const int tok = best_noisy(row, gz);
            if (lane == 0) {
              p.next_cand[bj] = tok;
              p.next_cand_prob[bj] = fast_exp2((gz - row_m[row]) * cT) / tsum[bj];
            }
          }
        }
      } else {
      // acceptance scan and emitted tokens: one warp per sequence
      for (int b = ew; b < p.B && with_targets; b += LM_EPI) {
        const int cv = (lane < p.k) ? cand_s[b * p.k + lane] : -1;
        const bool in_range = cv >= 0 && cv < p.V;
        const unsigned bad = __ballot_sync(0xFFFFFFFFu, lane < p.k && !in_range);
        const bool match = lane < p.k && in_range && cv == row_i[target_row(b, lane)];
        const unsigned acc_mask = __ballot_sync(0xFFFFFFFFu, match);
        const int i_star = __ffs(~acc_mask) - 1;            // first candidate that does not match (k when all do)
        const int j = lane;
        const int c_j = __shfl_sync(0xFFFFFFFFu, cv, min(j, p.k - 1));
        const int tok = (j < i_star) ? c_j : (j == i_star ? row_i[target_row(b, i_star)] : -1);
        const bool is_eos = p.eos_id >= 0 && j <= i_star && tok == p.eos_id;
        const unsigned eos_mask = __ballot_sync(0xFFFFFFFFu, is_eos && j < k1);
        const int n_out = eos_mask ? __ffs(eos_mask) - 1 : i_star + 1;
        if (j < k1) p.out_tokens[b * k1 + j] = (j < n_out) ? tok : -1;
        if (j == 0) {
          istar[b] = i_star;
          p.n_accept[b] = i_star;
          p.n_out[b] = n_out;
          p.finished[b] = (uint8_t)(eos_mask != 0);
          if (p.status && bad) atomicOr(p.status + b, SPACE_ST_BAD_CANDIDATE);
        }
      }
      if (!with_targets) for (int b = et; b < p.B; b += LM_EPI_T) istar[b] = max(0, min(p.n_accept[b], p.k));
      epi_sync();
      // sums of the mask rows of group i*: (sequence, mask row, range) triples spread over the threads
      const int total = with_masks ? p.B * p.k * G : 0;
      for (int i0 = et; i0 < total; i0 += LM_EPI_T * 8) {
        int4 v[8]; float mx[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int at = i0 + u * LM_EPI_T;
          v[u] = make_int4(0, 0, 0, 0); mx[u] = 0.f;
          if (at < total) {
            const int g = at % G, bj = at / G;
            const int b = bj / p.k, jj = bj - b * p.k;
            const int row = mask_row(b, istar[b], jj);
            mx[u] = row_m[row];
            v[u] = __ldcg(reinterpret_cast<const int4*>(p.part + (size_t)row * G + g));
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          const int at = i0 + u * LM_EPI_T;
          if (at < total) terms[at] = __int_as_float(v[u].y) * fast_exp2((__int_as_float(v[u].x) - mx[u]) * LOG2E);
        }
      }
      epi_sync();
      // fixed summation order: the result does not depend on which block came last or on timing
      for (int bj = ew; bj < p.B * p.k && with_masks; bj += LM_EPI) {
        float sv = 0.f;
        for (int g = lane; g < G; g += 32) sv += terms[bj * G + g];
        sv = warp_sum(sv);
        if (lane == 0) {
          const int b = bj / p.k;
          p.next_cand[bj] = row_i[mask_row(b, istar[b], bj - b * p.k)];
          p.next_cand_prob[bj] = 1.f / sv;                 // softmax at T = 1 of its own maximum
        }
      }
      }
    }
  }
#undef LBAR
  // ---- exit: every role is done (or has given up); free TMEM
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (*abort_flag && threadIdx.x == 0 && p.status) atomicOr(p.status, SPACE_ST_TIMEOUT);
  if (warp == 1)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
}

// [rows, D] bf16 matrix with `ld` elements between rows, boxes of box_rows x 64
int lm_make_map(CUtensorMap* tm, const void* base, int64_t rows, int64_t D, int64_t ld, int box_rows) {
  const cuuint64_t dims[4] = {(cuuint64_t)D, (cuuint64_t)rows, 1, 1};
  const cuuint64_t strides[3] = {(cuuint64_t)ld * 2, (cuuint64_t)ld * 2 * (cuuint64_t)rows, (cuuint64_t)ld * 2 * (cuuint64_t)rows};
  const cuuint32_t box[4] = {(cuuint32_t)LM_KB, (cuuint32_t)box_rows, 1, 1};
  return make_map(tm, base, dims, strides, box);
}

}  // namespace

size_t lmhead_gather_bytes() { return LM_GATHER_ELEMS * sizeof(__nv_bfloat16); }
size_t lmhead_partial_bytes(int sm_count) {
  return (size_t)LM_MAX_N * sm_count * (sizeof(LmPartial) + sizeof(LmNoisy));
}

namespace {

// Mask rows (i*, 1..k) of every sequence, then target row i* of every one where the grid asks for it, one thread block per
// row, next to one another for the second phase's box.  (Fetching them by a box per sequence instead, eight rows of 128 bytes each, paced the whole phase:
// 406 us under ncu for 16 sequences, D = 4096, V = 128256.)
__global__ void __launch_bounds__(256) lm_gather_kernel(const uint4* hidden, int64_t row_stride, int n_q, int k, int n_masks, int vecs,
                                                        const int32_t* n_accept, uint4* dst) {
  pdl_launch_dependents();
  pdl_wait();
  const int r = blockIdx.x, b = r < n_masks ? r / k : r - n_masks, o = r < n_masks ? r - b * k + 1 : 0;
  const uint4* src = hidden + ((int64_t)b * n_q + max(0, min(n_accept[b], k)) * (k + 1) + o) * row_stride;
  for (int i = threadIdx.x; i < vecs; i += blockDim.x) dst[(int64_t)blockIdx.x * vecs + i] = src[i];
}

// One launch: the rows that `phase` names of the sequences of `a` (at most LM_MAX_N); seq_base = index of the first
// of them in the caller's batch.
int launch_group(space_ctx* ctx, const space_lmhead_args* a, uint32_t seq_base, int phase, cudaStream_t st) {
  LmParams p;
  memset(&p, 0, sizeof(p));
  p.B = a->batch; p.k = a->k; p.V = a->vocab; p.D = a->hidden_dim;
  p.n_q = (a->k + 1) * (a->k + 1);
  p.phase = phase;
  const bool sampling = a->mode == SPACE_MODE_SAMPLE, literal = a->resample == SPACE_RESAMPLE_PAPER_LITERAL;
  // Sampling: target row k scores no candidate and draws nothing in the first pass, and row i* comes once more in the
  // second.  k+1 rows / k rows, us per call in a loop, V = 32000, D = 4096 (the draws all in the first pass, before the second
  // had row i*, in brackets): k = 1, 128 sequences 253.5 / 243.9 (247.6), 70 229.4 / 225.1 (228.1), k = 2, 32 121.7 / 118.7
  // (121.9), k = 3, 20 120.0 / 115.7 (120.8); 16 x 36 rows of V = 128256 394.7 / 392.3 (399.8).
  p.targets = sampling ? a->k : a->k + 1;
  p.n_rows = p.B * (phase == LM_ALL ? p.n_q : phase == LM_TARGETS ? p.targets : sampling ? a->k + 1 : a->k);
  p.sums = !(sampling && phase == LM_MASKS && !literal);    // (point-mass drafts: arg-maxes and the draw alone)
  p.n_pad = (p.n_rows + 15) / 16 * 16;
  if (p.n_pad > LM_MAX_N) return SPACE_E_UNSUPPORTED;
  p.n_mt = p.n_pad > LM_M ? 2 : 1;                         // (tokens on M: accumulators of 256 columns instead of 128)
  int grid = ctx->sm_count;
  const int max_useful = (a->vocab + 31) / 32;             // at least 32 tokens per thread block
  if (grid > max_useful) grid = max_useful;
  if (grid < 1) grid = 1;
  const int max_len = (a->vocab + grid - 1) / grid + 15;   // the longest vocabulary range (boundaries are multiples of 16)
  p.n_box = max_len >= LM_MAX_BOX ? LM_MAX_BOX : (max_len + 15) / 16 * 16;
  p.tail_rows = (((max_len - 1) % p.n_box) + 1 + 15) / 16 * 16;
  // Slices per stage: one (finer hand-over, more W in flight: with 144 block rows of V = 32000 two would leave
  // two stages, a fifth slower), except where a slice's products take less time than its hand-over, that is
  // with few tokens per thread block (us per call, graph replay, for one / two / four: 64 rows of V = 2091
  // 23.6 / 18.5 / 16.4, 25 rows of V = 5000 25.0 / 20.6 / 18.4, 36 rows of V = 12000 28.2 / 26.9 / 26.9, of
  // V = 32000 53.2 / 53.5 / -).  As many stages as fit, at most LM_MAX_STAGES.
  // Which operand is the block rows'.  Rows on M: an instruction of 128 rows and N tokens takes 43 + N/2 cycles (one per
  // 128 rows), however few of the 128 are real, and their energy with it, which under the power cap is time.  Tokens
  // on M: 43 + rows/2 for 128 tokens.  So tokens on M for few rows (energy) and where the rows would take two
  // instructions for little more than one's worth, as long as the 128-token accumulators are filled; up to about 80
  // rows and from 200 the time of the products is even, in between it is the other's.  Measured with D = 4096,
  // us per call in a steady loop (bursts), rows on M / tokens on M: greedy, V = 32000: 9 rows 53.2 (48.3) / 48.5 (48.1),
  // 36 rows 54.1 (48.8) / 51.1 (49.5), 49 rows 54.7 (49.6) / 52.7 (50.3), 72 rows 55.4 (50.4) / 55.6 (52.6), 108 rows
  // 57.9 (52.7) / 59.4 (54.1), 144 rows 72.9 (61.2) / 63.0 (56.4), 176 rows 75.8 (62.5) / 72.3 (62.0), 192 rows 75.8 (62.7) /
  // 74.0 (63.4), 252 rows 79.5 (67.9) / 84.9 (72.6); V = 128256: 36 rows 191 (167) / 171 (161); accumulators half empty,
  // V = 20000, D = 2048, 36 rows 22.3 (21.4) / 23.1 (23.9).  Sampling keeps the rows on M: with seven values per row the
  // epilogue of the other form is the longer one (measured when both had it, V = 32000: 36 rows 55.7 (52.9) / 56.8 (57.3),
  // 144 rows 77.2 (66.1) / 75.6 (73.1), 176 rows 82.2 (71.3) / 87.4 (85.7)).
  // (At 1965 MHz that is 1.4 % given away at 36 to 49 rows of V = 32000, D = 4096, for 5 % under the cap.)  Accumulators
  // less than three quarters full are the exception: a range of 257 to 288 tokens takes a third one for a few of them.
  // Bursts (loop), rows on M / tokens on M: V = 37800 (271 tokens), D = 1024 25 rows 22.2 (21.9) / 23.4 (23.2), 64 rows
  // 22.9 (22.5) / 24.1 (23.6), 160 rows 34.1 (33.6) / 35.7 (35.2), 175 rows 34.3 (33.6) / 36.7 (36.3); D = 2048 64 rows 38.2
  // (39.0) / 39.8 (39.6), 175 rows 51.7 (53.2) / 55.5 (54.9); D = 3072 25 rows 51.7 (53.5) / 53.1 (52.7), 160 rows 68.6 (73.7) /
  // 71.7 (71.4), 175 rows 71.0 (73.1) / 74.4 (74.8); V = 40000 (286 tokens), D = 1024 25 rows 22.9 (22.8) / 24.1 (23.6), D = 2048
  // 37.6 (39.8) / 38.2 (37.9).  So rows on M there for short products, and from 161 rows for all; 144 rows keep the tokens
  // there (V = 37800, D = 512 25.3 (24.7) before this form / 23.3 (22.9) with it, D = 4096 87.2 (93.4) / 83.1 (84.3)).
  const int in_acc = (max_len + LM_TOK - 1) / LM_TOK * LM_TOK;            // tokens that a range's accumulators have room for
  const bool filled = 4 * max_len > 3 * in_acc;
  const bool tokens_on_m = !sampling && p.n_box > 192 && (p.n_pad <= (filled || p.D > 1536 ? 64 : 16) ||
                                                          (p.n_pad > LM_M && p.n_pad <= (filled ? 176 : p.D > 1536 ? 160 : 144)));
  // (all that a block may have: with 96 rows it holds five stages, with 220 KB four; 16 x 36 rows of V = 128256, greedy,
  // 350 -> 343 us in bursts, 112 rows of V = 32000 52.8 -> 51.4, 144 sampling 66.7 -> 64.3, 72 of V = 5000 17.8 -> 16.8)
  const size_t budget = 227 * 1024;
  if (sampling) {
    // rows that draw a token (row_const), and as many tokens' noise as the table has room for
    p.n_noisy = phase == LM_TARGETS ? 0 : literal ? p.n_rows : p.B * (phase == LM_ALL ? a->k + 1 : 1);
    if (p.n_noisy) {
      // The table may take what a pipeline of a few stages leaves: five up to 80 rows (96 by phase, where only every
      // (k+1)-th draws a token unless drafts are sampled too), four up to 128 rows, three where the rows need two
      // accumulators and a stage is large.  24 KB / this, us per call in bursts: D = 2048, V = 128256, 160 rows 146.7 / 134.9;
      // D = 4096, V = 32000, 160 rows 71.1 / 68.0, 208 rows 74.1 / 71.0.  Other numbers of stages: 208 rows, two 88.4; 80
      // rows of V = 128256 (D = 2048), four / five 94.5 / 92.5; 16 x 36 rows, 96 of them at a time, four / five
      // 343.6 / 340.8; 108 rows of V = 32000, four / five 56.5 / 58.7.
      const int keep = p.n_pad > LM_M ? 3 : (p.n_pad <= 80 || (p.n_pad <= 96 && phase != LM_ALL)) ? 5 : 4;
      int64_t rest = (int64_t)budget - 1024 - LmSmem(false, true, 0, 0, p.n_pad, p.n_box, keep, 1).total;
      if (p.n_box <= 128 && rest > 24 * 1024) rest = 24 * 1024;        // (stages of several slices, see below)
      const int64_t room = rest / 4 / p.n_noisy - 4;
      p.noise_tok = room < 16 ? 0 : (int)(room < p.n_box ? room : p.n_box) & ~15;
    }
  }
  // Where a range is one box, the mask rows' pass takes the slices from the end: those of the target rows' pass that are
  // still in L2 (us per call in bursts (steady loop), forwards / backwards: 16 x 36 rows, V = 32000, D = 4096 107.8 (116.8) /
  // 104.9 (112.7), D = 2048, sampling, 76.2 (77.5) / 72.9 (73.0)).  With more boxes the stream itself is slower that way
  // (V = 128256, D = 4096 359 / 375), and the last box alone first gains nothing that lasts (359 / 360; V = 64000 186.5 / 184.3,
  // V = 80000, D = 2048 130.3 / 132.7).
  p.backwards = phase == LM_MASKS && max_len <= p.n_box;
  int stages = 0;
  for (p.kbs = p.n_box <= 128 ? 4 : 1; p.kbs >= 1; p.kbs /= 2) {
    stages = LM_MAX_STAGES;
    while (stages > 1 && LmSmem(tokens_on_m, sampling, p.n_noisy, p.noise_tok, p.n_pad, p.n_box, stages, p.kbs).total + 1024 > budget) --stages;
    if (stages >= (p.kbs > 1 ? 3 : 2)) break;
  }
  if (stages < 2) return SPACE_E_UNSUPPORTED;
  p.stages = stages;
  const LmSmem L(tokens_on_m, sampling, p.n_noisy, p.noise_tok, p.n_pad, p.n_box, stages, p.kbs);
  if (L.total + 1024 > budget) return SPACE_E_UNSUPPORTED;
  p.eos_id = a->eos_id;
  p.mode = a->mode; p.resample = a->resample;
  p.c_t = LOG2E / (a->mode == SPACE_MODE_SAMPLE ? a->temperature : 1.0f);
  p.key0 = (uint32_t)(a->seed & 0xFFFFFFFFull); p.key1 = (uint32_t)(a->seed >> 32);
  p.seq_base = seq_base;
  p.cand_prob = a->cand_prob; p.seq_id = a->seq_id; p.kv_len = a->kv_len;
  p.gpart = reinterpret_cast<LmNoisy*>(ctx->lm_part + (size_t)LM_MAX_N * ctx->sm_count * sizeof(LmPartial));
  p.zc = reinterpret_cast<float*>(reinterpret_cast<char*>(ctx->lm_counter) + 256 + LM_MAX_N * sizeof(unsigned long long));
  p.cand = a->cand;
  p.n_accept = a->n_accept; p.out_tokens = a->out_tokens; p.n_out = a->n_out; p.next_cand = a->next_cand;
  p.next_cand_prob = a->next_cand_prob; p.finished = a->finished; p.status = a->status;
  p.row_max = a->row_max; p.row_argmax = a->row_argmax;
  p.part = reinterpret_cast<LmPartial*>(ctx->lm_part);
  p.counter = ctx->lm_counter;
  p.keys = reinterpret_cast<unsigned long long*>(ctx->lm_counter + 64);
  p.err = ctx->lm_counter + 1;
  int rc = lm_make_map(&p.tm_w, a->weight, a->vocab, a->hidden_dim, a->weight_row_stride, p.n_box);
  if (rc == SPACE_OK) rc = lm_make_map(&p.tm_wt, a->weight, a->vocab, a->hidden_dim, a->weight_row_stride, p.tail_rows);
  // hidden rows in one box: all of them, every (k+1)-th (the target rows lie k+1 rows apart, across
  // sequences too), the first k of those of every sequence (sampling; no rows of zeros up to n_pad follow them: what lies
  // there only reaches accumulator lanes nobody reads), or the gathered rows
  const bool first_k = sampling && phase == LM_TARGETS;
  p.h_bytes = (first_k ? p.n_rows : p.n_pad) * LM_KB * 2;
  if (rc == SPACE_OK && first_k) {
    const cuuint64_t ld = (cuuint64_t)a->hidden_row_stride * 2;
    const cuuint64_t dims[4] = {(cuuint64_t)p.D, (cuuint64_t)p.k, (cuuint64_t)p.B, 1};
    const cuuint64_t strides[3] = {ld * (p.k + 1), ld * p.n_q, ld * p.n_q * p.B};
    const cuuint32_t box[4] = {(cuuint32_t)LM_KB, (cuuint32_t)p.k, (cuuint32_t)p.B, 1};
    rc = make_map(&p.tm_h, a->hidden, dims, strides, box);
  } else if (rc == SPACE_OK) {
    rc = phase == LM_MASKS ? lm_make_map(&p.tm_h, ctx->lm_gather, p.n_rows, a->hidden_dim, a->hidden_dim, p.n_pad)
                           : lm_make_map(&p.tm_h, a->hidden, p.n_rows, a->hidden_dim,
                                         a->hidden_row_stride * (phase == LM_TARGETS ? a->k + 1 : 1), p.n_pad);
  }
  if (rc != SPACE_OK) return rc;
  const size_t sm = L.total + 1024;
  auto kernel = tokens_on_m ? lmhead_verify_kernel<true, false> : sampling ? lmhead_verify_kernel<false, true> : lmhead_verify_kernel<false, false>;
  // (all that a block may have, whatever this call needs: the limit is the kernel's, and a thread with a context of its
  // own must not find it lowered between this and its launch)
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)budget);
  {
    ProfScope ps(ctx, SPACE_K_LMHEAD, st);
    launch_pdl(kernel, dim3(grid), dim3(LM_THREADS), sm, st, p);
  }
  ctx->launches += 1;
  return cuda_ok(cudaGetLastError());
}

}  // namespace

// Which launches a batch takes.  Up to 256 block rows: one launch over all of them, one pass over the output
// embedding.  More: the step decides on 2k+1 rows of every sequence only, so the target rows go first and the
// mask rows of the groups they select second (sampling: with target row i* once more, which draws the extra token; the
// noise of every target row, of which k in k+1 was for nothing, before: 16 x 36 rows of V = 128256 376 -> 370 us in a loop, of
// V = 32000 119.0 -> 115.1, 16 x 64 rows of V = 60000, D = 1024 76.6 -> 72.7, drafts sampled 16 x 36 of V = 32000 88.3 -> 85.5) -- two passes over the embedding, each near the pace of its
// stream, instead of one per 256 rows at the pace of the product.  Calls that ask for every row's maximum
// keep to the full rows.
// Measured, us per call, D = 4096, sampling, steady loop (bursts), over all rows / by phase: 16 x 36 rows of
// V = 128256 832 (722) / 370 (341); 4 x 36 rows of V = 32000 80 (71) / 115 (109); 16 x 16 rows of V = 50257
// 140 (125) / 182 (169).
int launch_lmhead_verify(space_ctx* ctx, const space_lmhead_args* a, cudaStream_t st) {
  const int n_q = (a->k + 1) * (a->k + 1), k1 = a->k + 1;
  const int rows = a->batch * n_q;
  const int second = a->mode == SPACE_MODE_SAMPLE ? k1 : a->k;             // rows of a sequence in the second phase
  const int64_t fit = LM_GATHER_ELEMS / ((int64_t)second * a->hidden_dim);  // sequences whose rows can be gathered
  const int per_phase = fit < LM_M / k1 ? (int)fit : LM_M / k1, per_all = LM_MAX_N / n_q;
  bool by_phase = per_phase > 0 && !a->row_max && !a->row_argmax && rows > LM_MAX_N;
  // a small embedding (under about 10 us of stream) is paced by launches instead: as few of them as can be
  if (by_phase && (int64_t)a->vocab * a->hidden_dim < (32ll << 20))
    by_phase = 2 * ((a->batch + per_phase - 1) / per_phase) < (a->batch + per_all - 1) / per_all;
  const int per_group = by_phase ? per_phase : per_all;
  if (per_group < 1) return SPACE_E_UNSUPPORTED;
  for (int b0 = 0; b0 < a->batch; b0 += per_group) {
    space_lmhead_args g = *a;
    g.batch = a->batch - b0 < per_group ? a->batch - b0 : per_group;
    g.hidden = static_cast<const __nv_bfloat16*>(a->hidden) + (int64_t)b0 * n_q * a->hidden_row_stride;
    g.cand = a->cand + (int64_t)b0 * a->k;
    if (a->cand_prob) g.cand_prob = a->cand_prob + (int64_t)b0 * a->k;
    if (a->seq_id) g.seq_id = a->seq_id + b0;
    if (a->kv_len) g.kv_len = a->kv_len + b0;
    g.n_accept = a->n_accept + b0; g.out_tokens = a->out_tokens + (int64_t)b0 * k1; g.n_out = a->n_out + b0;
    g.next_cand = a->next_cand + (int64_t)b0 * a->k; g.next_cand_prob = a->next_cand_prob + (int64_t)b0 * a->k;
    g.finished = a->finished + b0;
    if (a->status) g.status = a->status + b0;
    if (a->row_max) g.row_max = a->row_max + (int64_t)b0 * n_q;
    if (a->row_argmax) g.row_argmax = a->row_argmax + (int64_t)b0 * n_q;
    int rc = launch_group(ctx, &g, (uint32_t)b0, by_phase ? LM_TARGETS : LM_ALL, st);
    if (rc == SPACE_OK && by_phase) {
      launch_pdl(lm_gather_kernel, dim3(g.batch * second), dim3(256), 0, st, static_cast<const uint4*>(g.hidden),
                 a->hidden_row_stride / 8, n_q, a->k, g.batch * a->k, a->hidden_dim / 8, (const int32_t*)g.n_accept, (uint4*)ctx->lm_gather);
      ctx->launches += 1;
      rc = launch_group(ctx, &g, (uint32_t)b0, LM_MASKS, st);
    }
    if (rc != SPACE_OK) return rc;
  }
  return SPACE_OK;
}
