// Tensor-core attention of the block rows over cache + block (Eq. 5) for sm_100a,
// row orientation: used when the query block of one kv head has more than 64
// rows (block rows times GQA group), where a full 128-row MMA tile is well
// filled.  Narrower blocks go to the transposed kernel of attn_tc.cu, which
// this file mirrors in structure (clustered cut or flat tile list, split partials, merge).
//
// Here the query rows are the MMA M extent and the 128 keys of a tile the N
// extent: S = Q K^T (128 x 128) into one of three TMEM buffers, P overwrites S in
// TMEM as two bf16 terms, O += (P_hi + P_lo) V with P read back from TMEM.
// Inside a block (12 warps): warps 0 and 2 stream K (and the query rows) and V tiles
// with TMA, warps 1 and 3 issue the S and the O products, warps 4-11 are two threads
// per query row (64 keys of the tile each) with a running row maximum and lazy
// rescaling of O.  Every wait is bounded; an expired wait sets SPACE_ST_TIMEOUT
// and the block drains and exits.
#include "common.cuh"
#include "tc_common.cuh"
#include "attn_common.cuh"
#include <cuda.h>
#include <math_constants.h>

namespace {

constexpr int TILE_N = 128;            // keys per tile
constexpr int THREADS = 384;            // K (+Q), S-issuer, V, O-issuer warps + 8 softmax warps
constexpr uint64_t WAIT_NS = 1000000000ull;   // one second per wait
constexpr float RESCALE_THRESHOLD = 8.f;
// Starting a share (query load, pipeline refill, epilogue) costs about as much as
// this many tiles; the flat list carries that many extra entries per (sequence, head).
constexpr int SHARE_COST = 4;

struct AttnParams {
  CUtensorMap tm_q, tm_k, tm_v;
  int B, n_q, H_q, H_kv, G;
  int n_mblocks, rows_per_mb;          // query-row blocks per kv head; block rows i per block
  int n_groups;                        // thread-block groups (grid = n_groups * n_mblocks)
  int pieces;                          // > 0: the grid is cut into clusters of pieces * n_mblocks blocks, one per (sequence, head)
  int out_dtype;
  int64_t s_cap;                       // rows a sequence may hold (paged: pages_per_seq * SPACE_PAGE_SIZE)
  // Paged cache (page_table != nullptr): tm_k / tm_v describe a pool [n_pages][H_kv][TILE_N][d] and tile t
  // of sequence b is the whole page page_table[b * pages_per_seq + t]; no tile is shifted back, the
  // rows of the last page past the last key are masked (S) and cleared in shared memory (V).
  const int32_t* page_table; int pages_per_seq, n_pages;
  float scale_log2;                    // scale * log2(e)
  const int32_t* kv_len;
  void* out; float* lse; int32_t* status;
  float* part;                         // [slots][ROWS*(DH+2)]
  int* err;                            // one word: first timeout site
  int2* desc;                          // [B*H_kv*n_mblocks] {first group, number of groups} of each cut
  int4* owner;                         // [grid] the cut whose last piece this thread block computed: {(sequence, kv head) or -1,
                                       // its descriptor}
  int merge_by_owner;                  // the merge grid is indexed by attention thread block, not by (sequence, head)
  int* arrived;                        // [B*H_kv*n_mblocks] pieces of a cut whose partial is stored (self-resetting)
  uint64_t mask[SPACE_MAX_ROWS];
};

// One share: tiles t0, t0 + step, ... (n of them) of the T tiles of (sequence b, kv head h).
struct Seg { int b, h, t0, n, step, T, L; };
// How a share's (sequence, head) was cut: {first group, number of groups}.
__host__ __device__ __forceinline__ int2 share_cut(const int* prefix, int B, int n_groups, const Seg& sg, int group) {
  return sg.n == sg.T ? make_int2(group, 1) : attn::list_cut(prefix, B, n_groups, SHARE_COST, sg.b, sg.h, sg.T);
}

// PTX helpers: tc_common.cuh.  Every wait of this kernel is bounded by WAIT_NS.
using namespace tc;
using namespace attn;
__device__ __noinline__ bool mbar_wait_long(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err, int site) {
  return mbar_wait_bounded(bar, parity, abort_flag, err, site, WAIT_NS, 0);
}
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int* err, int site) {
  return mbar_try(bar, parity) || mbar_wait_long(bar, parity, abort_flag, err, site);   // (see mbar_wait_bounded)
}
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity) { mbar_drain_bounded(bar, parity, WAIT_NS); }
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* r) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
        "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
        "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr) : "memory");
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t* r) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
        "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]),
        "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]),
        "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
// Instruction descriptor: bf16 x bf16 -> f32, M = 128.
__host__ __device__ constexpr uint32_t instr_desc(int n, int b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)b_mn_major << 16) |
         ((uint32_t)(n >> 3) << 17) | ((uint32_t)(ROWS >> 4) << 24);
}

// ------------------------------------------------------------ work partition
// Flat tile index space: sequence-major, then kv head, then tile.  Group g of
// n_groups owns flat tiles [W*g/n_groups, W*(g+1)/n_groups).
struct Partition {
  const int* seq_len;    // [B]   verified length, or -1 for a sequence that does not fit
  const int* prefix;     // [B+1] flat offset of sequence b
  int B, H_kv, n_q;
  long long cur, end;
  int b;
  const int* one;        // clustered cut: {b, h, t0, n, T, L, step}, this block's only share
  __device__ void init_one(const int* share) { one = share; cur = 0; end = share[3] > 0 ? 1 : 0; }
  // Only min(n_groups, W) groups take part, so every taking-part group owns at
  // least one tile and the groups of one (sequence, head) are consecutive.
  __host__ __device__ void init(const int* sl, const int* pf, int B_, int H, int nq, int group, int n_groups) {
    seq_len = sl; prefix = pf; B = B_; H_kv = H; n_q = nq; b = 0; one = nullptr;
    const long long W = pf[B_];
    const long long NG = W < n_groups ? W : n_groups;
    if (group >= NG) { cur = end = 0; return; }
    cur = muldiv(W, group, NG);
    end = muldiv(W, group + 1, NG);
  }
  __host__ __device__ bool next(Seg& s) {
    if (one) {
      if (cur >= end) return false;
      ++cur;
      const int4 u = reinterpret_cast<const int4*>(one)[0], v = reinterpret_cast<const int4*>(one)[1];
      s.b = u.x; s.h = u.y; s.t0 = u.z; s.n = u.w; s.T = v.x; s.L = v.y; s.step = v.z;
      return true;
    }
    // The list holds T + SHARE_COST entries per (sequence, head); the first
    // SHARE_COST stand for the fixed cost of starting a share there, so that
    // equal list shares are shares of about equal time.
    for (;;) {
      if (cur >= end) return false;
      while (prefix[b + 1] <= cur) ++b;
      const int L = seq_len[b];
      const int T = (L + n_q + TILE_N - 1) / TILE_N;
      const int Tv = T + SHARE_COST;
      const int rem = (int)(cur - prefix[b]);
      const int h = rem / Tv, r0 = rem - h * Tv;
      long long n = Tv - r0;
      if (n > end - cur) n = end - cur;
      cur += n;
      const int t0 = max(r0 - SHARE_COST, 0), t1 = max(r0 + (int)n - SHARE_COST, 0);
      if (t1 <= t0) continue;                               // only cost entries here: no tiles
      s.b = b; s.h = h; s.t0 = t0; s.n = t1 - t0; s.step = 1; s.T = T; s.L = L;
      return true;
    }
  }
};

template <int DH>
struct Smem {
  static constexpr int HALVES = DH / 64;
  static constexpr int TILE_BYTES = TILE_N * DH * 2;         // one K or V tile
  static constexpr int Q_BYTES = ROWS * DH * 2;
  static constexpr int K_STAGES = (DH == 128) ? 2 : 3;
  static constexpr int V_STAGES = (DH == 128) ? 2 : 4;
  static constexpr int Q_OFF = 0;
  static constexpr int K_OFF = Q_BYTES;
  static constexpr int V_OFF = K_OFF + K_STAGES * TILE_BYTES;
  static constexpr int BAR_OFF = V_OFF + V_STAGES * TILE_BYTES;
  static constexpr int S_BUFS = 3;                           // S / P buffers in TMEM (3 x 128 columns, O at 384)
  // q_full, q_empty, k_full[], k_empty[], v_full[], v_empty[], s_full[3], p_ready[3], pv_done[3], drain
  static constexpr int N_BARS = 2 + 2 * K_STAGES + 2 * V_STAGES + 3 * S_BUFS + 1;
  static constexpr int MISC_OFF = BAR_OFF + (N_BARS * 8 + 15) / 16 * 16;   // tmem base, abort flag
  static constexpr int SEG0_OFF = MISC_OFF + 16;             // the only share of a clustered cut (8 ints)
  static constexpr int XMAX_OFF = MISC_OFF + 48;             // [2 parities][2 halves][ROWS] float
  static constexpr int XSUM_OFF = XMAX_OFF + 2 * 2 * ROWS * 4;   // [2 halves][ROWS] float
  static constexpr int EPI_PITCH = 36;                       // floats per staged row: 32 columns + 4 (16-byte aligned, conflict-free)
  static constexpr int EPI_OFF = XSUM_OFF + 2 * ROWS * 4;    // [8 warps][32 rows][EPI_PITCH] float: epilogue transpose
  // a piece's partial for the cluster, in the slot format of global memory: over the K (and V) stages, all
  // consumed by then
  static constexpr int PART_OFF = K_OFF;
  static_assert(PART_OFF + ROWS * (DH + 2) * 4 <= BAR_OFF, "a partial must fit the K and V stages");
  static constexpr int TABLE_OFF = EPI_OFF + 8 * 32 * EPI_PITCH * 4;   // seq_len[max_batch], prefix[max_batch+1]
};


// The two softmax warps that share a TMEM lane quarter meet here (ids 1..4).
__device__ __forceinline__ void pair_sync(int quarter) {
  asm volatile("bar.sync %0, 64;" ::"r"(quarter + 1) : "memory");
}

// Warp roles
constexpr int WARP_K = 0, WARP_MMA = 1, WARP_V = 2, WARP_PV = 3, WARP_SOFTMAX0 = 4;

template <int DH>
__global__ void __launch_bounds__(THREADS, 1) attn_rows_kernel(const __grid_constant__ AttnParams p,
                                                             int max_batch) {
  using S = Smem<DH>;
  extern __shared__ __align__(1024) unsigned char sm[];
  const uint32_t sm_base = smem_u32(sm);
  const uint32_t bar0 = sm_base + S::BAR_OFF;
  auto BAR = [&](int i) { return bar0 + 8u * i; };
  constexpr int B_QFULL = 0, B_QEMPTY = 1, B_KFULL = 2, B_KEMPTY = B_KFULL + S::K_STAGES,
                B_VFULL = B_KEMPTY + S::K_STAGES, B_VEMPTY = B_VFULL + S::V_STAGES,
                B_SFULL = B_VEMPTY + S::V_STAGES, B_PREADY = B_SFULL + S::S_BUFS,
                B_PVDONE = B_SFULL + 2 * S::S_BUFS, B_DRAIN = B_SFULL + 3 * S::S_BUFS;
  constexpr uint32_t NS = S::S_BUFS;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(sm + S::MISC_OFF);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(sm + S::MISC_OFF + 4);
  float* xmax = reinterpret_cast<float*>(sm + S::XMAX_OFF);
  float* xsum = reinterpret_cast<float*>(sm + S::XSUM_OFF);
  int* seq_len = reinterpret_cast<int*>(sm + S::TABLE_OFF);
  int* prefix = seq_len + max_batch;
  int* seg0 = reinterpret_cast<int*>(sm + S::SEG0_OFF);
  int4* duties = reinterpret_cast<int4*>(seg0);            // (where there is no clustered cut: see note_if_last)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = blockIdx.x / p.n_mblocks, mb = blockIdx.x % p.n_mblocks;
  const int i0 = mb * p.rows_per_mb;                       // first block row of this query-row block
  // MMA rows that carry a real (block row, head) pair are 0 .. m_valid-1
  const int m_valid = min(p.rows_per_mb, p.n_q - i0) * p.G;
  const int n_quarters = (m_valid + 31) >> 5;              // TMEM lane quarters with live rows
  const int n_soft = 64 * n_quarters;                      // softmax threads that take part

  // the query rows' box holds rows_per_mb block rows; the rows after them in shared memory stay zero
  const int q_rows = p.rows_per_mb * p.G;
  const uint32_t q_bytes = (uint32_t)q_rows * DH * 2;

  // ---- set-up ------------------------------------------------------------
  pdl_launch_dependents();
  for (int x = q_rows * 8 + threadIdx.x; x < ROWS * 8; x += THREADS)      // 16-byte pieces of 128-byte rows
#pragma unroll
    for (int hf = 0; hf < S::HALVES; ++hf)
      asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(sm_base + S::Q_OFF + hf * (ROWS * 128) + x * 16), "r"(0u) : "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  if (threadIdx.x == 0) {
    for (int e = 0; e < MAX_DUTIES; ++e) duties[e].x = -1;
    *abort_flag = (sm_base & 1023u) ? 1 : 0;               // swizzled tiles need a 1024-byte aligned base
    mbar_init(BAR(B_QFULL), 1);
    mbar_init(BAR(B_QEMPTY), 1);
    for (int s = 0; s < S::K_STAGES; ++s) { mbar_init(BAR(B_KFULL + s), 1); mbar_init(BAR(B_KEMPTY + s), 1); }
    for (int s = 0; s < S::V_STAGES; ++s) { mbar_init(BAR(B_VFULL + s), 1); mbar_init(BAR(B_VEMPTY + s), 1); }
    for (int i = 0; i < S::S_BUFS; ++i) {
      mbar_init(BAR(B_SFULL + i), 1);
      mbar_init(BAR(B_PREADY + i), n_soft);
      mbar_init(BAR(B_PVDONE + i), 1);
    }
    mbar_init(BAR(B_DRAIN), 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == WARP_MMA) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                 ::"r"(smem_u32(tmem_slot)), "r"(512u) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  if (warp == WARP_K && lane == 0)
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.tm_k) : "memory");
  if (warp == WARP_V && lane == 0)
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.tm_v) : "memory");
  if (warp == WARP_MMA && lane == 0)
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&p.tm_q) : "memory");
  // Clustered cut (see attn_tc.cu): piece cl_piece of pair cl_pair, tiles cl_piece, cl_piece + pieces, ...
  const int cl_pair = p.pieces ? group / p.pieces : 0, cl_piece = p.pieces ? group - cl_pair * p.pieces : 0;
  const bool cl_mine = p.pieces && cl_pair < p.B * p.H_kv;
  const int cl_b = cl_pair / p.H_kv, cl_h = cl_pair - cl_b * p.H_kv;
  // barriers and the TMEM allocation are visible to every warp before the first global access (with a
  // programmatic launch this part runs under the previous kernel)
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_wait();                                              // global memory from here on
  if (cl_mine && warp == WARP_K && lane == 0 && !*abort_flag) {
    // the query rows and the first K tile, before any length is read (should the length turn out too short for
    // that tile, or the cut not be taken, the S issuer lets both buffers go unused)
    mbar_expect_tx(BAR(B_QFULL), q_bytes);
#pragma unroll
    for (int hf = 0; hf < S::HALVES; ++hf)
      tma_load_4d(sm_base + S::Q_OFF + hf * (ROWS * 128), &p.tm_q, BAR(B_QFULL), hf * 64, cl_h * p.G, i0, cl_b);
    mbar_expect_tx(BAR(B_KFULL), S::TILE_BYTES);
#pragma unroll
    for (int hf = 0; hf < S::HALVES; ++hf)
      tma_load_4d(sm_base + S::K_OFF + hf * (TILE_N * 128), &p.tm_k, BAR(B_KFULL), hf * 64,
                  p.page_table ? 0 : cl_piece * TILE_N, cl_h, p.page_table ? page_of(p, cl_b, cl_piece, false) : cl_b);
  }
  bool clustered = false, spec_ok = false;                 // spec_ok: the early requests serve this block's share
  int cl_n = 0;                                            // pieces of this block's pair that have tiles
  if (p.pieces) {
    // every warp works the same things out for itself: nothing has to be handed over
    auto tiles_of = [&](int L) { return (L >= 0 && (int64_t)L + p.n_q <= p.s_cap) ? (L + p.n_q + TILE_N - 1) / TILE_N : 0; };
    const int L0 = cl_mine ? p.kv_len[cl_b] : -1;
    clustered = cluster_fits(p, lane, tiles_of);
    if (clustered) {
      const int T = tiles_of(L0), L = T ? L0 : -1;
      if (cl_mine && !T && cl_piece == 0 && cl_h == 0 && mb == 0 && threadIdx.x == 0 && p.status)
        atomicOr(p.status + cl_b, SPACE_ST_CAPACITY);
      const int n_mine = cl_piece < T ? (T - cl_piece + p.pieces - 1) / p.pieces : 0;
      cl_n = min(p.pieces, T);
      spec_ok = n_mine > 0 && (p.page_table || (cl_piece + 1) * TILE_N <= L + p.n_q);
      if (p.page_table && spec_ok && warp == WARP_K && lane == 0) (void)page_of(p, cl_b, cl_piece);   // flags a bad entry
      // (identical values by every thread, each reads back what it wrote)
      reinterpret_cast<int4*>(seg0)[0] = make_int4(cl_b, cl_h, cl_piece, n_mine);
      reinterpret_cast<int4*>(seg0)[1] = make_int4(T, L, p.pieces, 0);
    }
  }
  if (!clustered) {
  if (warp == WARP_SOFTMAX0) {
    // per-sequence tile counts and their running sum, 32 sequences per round
    int carry = 0;
    for (int b0 = 0; b0 < p.B; b0 += 32) {
      const int b = b0 + lane;
      int L = -1, tiles = 0;
      if (b < p.B) {
        L = p.kv_len[b];
        const bool ok = L >= 0 && (int64_t)L + p.n_q <= p.s_cap;
        if (!ok && blockIdx.x == 0 && p.status) atomicOr(p.status + b, SPACE_ST_CAPACITY);
        if (!ok) L = -1;
        tiles = ok ? ((L + p.n_q + TILE_N - 1) / TILE_N + SHARE_COST) * p.H_kv : 0;
      }
      int incl = tiles;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xFFFFFFFFu, incl, o);
        if (lane >= o) incl += v;
      }
      if (b < p.B) { seq_len[b] = L; prefix[b] = carry + incl - tiles; }
      carry += __shfl_sync(0xFFFFFFFFu, incl, 31);
    }
    if (lane == 0) prefix[p.B] = carry;
  }
  __syncthreads();                                          // the tables reach every warp
  }
  const uint32_t tmem = *tmem_slot;
  const uint32_t TM_S0 = tmem, TM_O = tmem + S::S_BUFS * TILE_N;   // S buffers at columns 0, 128, 256; O at 384

  Partition part;
  if (clustered) part.init_one(seg0);
  else part.init(seq_len, prefix, p.B, p.H_kv, p.n_q, group, p.n_groups);
  Seg sg;
  const bool dead = *abort_flag != 0;

  if (dead) {
    // nothing was issued; fall through to the teardown
  } else if (warp == WARP_K || warp == WARP_V) {
    // ================= K / V producers ====================================
    if (elect_one()) {
      const bool is_k = warp == WARP_K;
      const int n_st = is_k ? S::K_STAGES : S::V_STAGES;
      const int b_full = is_k ? B_KFULL : B_VFULL, b_empty = is_k ? B_KEMPTY : B_VEMPTY;
      const uint32_t ring = sm_base + (is_k ? S::K_OFF : S::V_OFF);
      const CUtensorMap* tm = is_k ? &p.tm_k : &p.tm_v;
      // gt counts the ring's tiles; early requests that serve no share take the first place of either buffer
      bool pre = is_k && spec_ok;                           // Q and the first K tile of the share are on their way
      uint32_t gt = cl_mine && is_k && !spec_ok ? 1u : 0u, seg = gt;
      bool ok = true;
      while (ok && part.next(sg)) {
        const int n_keys = sg.L + p.n_q;
        if (is_k) {
          // the K producer also loads this share's query rows, once the last S
          // product of the share before has read the buffer
          if (!pre) {
            if (seg > 0) ok = mbar_wait(BAR(B_QEMPTY), (seg - 1) & 1, abort_flag, p.err, 3);
            if (!ok) break;
            mbar_expect_tx(BAR(B_QFULL), q_bytes);
#pragma unroll
            for (int hf = 0; hf < S::HALVES; ++hf)
              tma_load_4d(sm_base + S::Q_OFF + hf * (ROWS * 128), &p.tm_q, BAR(B_QFULL), hf * 64,
                          sg.h * p.G, i0, sg.b);
          }
          ++seg;
        }
        for (int j = 0, t = sg.t0; j < sg.n && ok; ++j, t += sg.step, ++gt) {
          if (pre) { pre = false; continue; }
          const int s = gt % n_st;
          if (gt >= (uint32_t)n_st)
            ok = mbar_wait(BAR(b_empty + s), ((gt / n_st) - 1) & 1, abort_flag, p.err, is_k ? 1 : 2);
          if (!ok) break;
          // the last tile of a sequence is shifted back so that it ends at the
          // last key: rows past the end are never read (they may hold anything)
          // (a paged cache has whole pages for tiles instead; see AttnParams)
          const int kt = p.page_table ? 0 : (((t + 1) * TILE_N <= n_keys) ? t * TILE_N : n_keys - TILE_N);
          const int kb = p.page_table ? page_of(p, sg.b, t) : sg.b;
          const uint32_t dst = ring + s * S::TILE_BYTES;
          mbar_expect_tx(BAR(b_full + s), S::TILE_BYTES);
#pragma unroll
          for (int hf = 0; hf < S::HALVES; ++hf)
            tma_load_4d(dst + hf * (TILE_N * 128), tm, BAR(b_full + s), hf * 64, kt, sg.h, kb);
        }
      }
      // drain: every issued copy must have landed before the block may exit
      const uint32_t first = gt > (uint32_t)n_st ? gt - n_st : 0;
      for (uint32_t g = first; g < gt; ++g) mbar_drain(BAR(b_full + g % n_st), (g / n_st) & 1);
      if (is_k && seg > 0) mbar_drain(BAR(B_QFULL), (seg - 1) & 1);
    }
  } else if (warp == WARP_MMA) {
    // ================= S issuer ============================================
    if (elect_one()) {
      constexpr uint32_t IDESC_QK = instr_desc(TILE_N, 0);
      uint32_t gt = 0, seg = 0, koff = 0;
      bool ok = true;
      if (cl_mine && !spec_ok) {
        // the early requests serve no share: once they have landed their buffers go back unused
        ok = mbar_wait(BAR(B_QFULL), 0, abort_flag, p.err, 15);
        if (ok) ok = mbar_wait(BAR(B_KFULL), 0, abort_flag, p.err, 16);
        mbar_arrive(BAR(B_QEMPTY));
        mbar_arrive(BAR(B_KEMPTY));
        seg = 1; koff = 1;
      }
      while (ok && part.next(sg)) {
        ok = mbar_wait(BAR(B_QFULL), seg & 1, abort_flag, p.err, 6);
        const int n = sg.n;
        for (int j = 0; j < n && ok; ++j, ++gt) {
          const int s = (gt + koff) % S::K_STAGES;
          const uint32_t buf = gt % NS;
          ok = mbar_wait(BAR(B_KFULL + s), ((gt + koff) / S::K_STAGES) & 1, abort_flag, p.err, 7);
          // S buffer `buf` held the P of tile gt - 3, read by that tile's O product
          if (ok && gt >= NS) ok = mbar_wait(BAR(B_PVDONE + buf), ((gt / NS) - 1) & 1, abort_flag, p.err, 8);
          if (!ok) break;
          tc_fence_after();
          const uint32_t qsm = sm_base + S::Q_OFF;
          const uint32_t ksm = sm_base + S::K_OFF + s * S::TILE_BYTES;
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk) {
            const uint32_t off = (kk >> 2) * (ROWS * 128) + (kk & 3) * 32;   // 64-wide half, then 32 B per 16 elements
            mma_ss(TM_S0 + buf * TILE_N, smem_desc(qsm + off, 16, 1024), smem_desc(ksm + off, 16, 1024),
                   IDESC_QK, kk > 0 ? 1u : 0u);
          }
          tc_commit(BAR(B_SFULL + buf));
          tc_commit(BAR(B_KEMPTY + s));
          if (j == n - 1) tc_commit(BAR(B_QEMPTY));
        }
        ++seg;
      }
    }
  } else if (warp == WARP_PV) {
    // ================= O issuer ============================================
    // A thread of its own: the S products of later tiles need not queue behind
    // the sixteen instructions of an O product or wait for its operands.
    if (elect_one()) {
      constexpr uint32_t IDESC_PV = instr_desc(DH, 1);
      uint32_t g = 0;
      bool ok = true;
      while (ok && part.next(sg)) {
        for (int j = 0; j < sg.n && ok; ++j, ++g) {
          // O += (P_hi + P_lo) V; the first product of a share overwrites O
          const int s = g % S::V_STAGES;
          const uint32_t buf = g % NS;
          ok = mbar_wait(BAR(B_VFULL + s), (g / S::V_STAGES) & 1, abort_flag, p.err, 4);
          if (ok) ok = mbar_wait(BAR(B_PREADY + buf), (g / NS) & 1, abort_flag, p.err, 5);
          if (!ok) break;
          tc_fence_after();
          const uint32_t vsm = sm_base + S::V_OFF + s * S::TILE_BYTES;
          const uint32_t ptm = TM_S0 + buf * TILE_N;
#pragma unroll
          for (int part_i = 0; part_i < 2; ++part_i) {        // P_hi, then P_lo
#pragma unroll
            for (int kk = 0; kk < TILE_N / 16; ++kk) {
              // V tile is MN-major: 64-wide d blocks TILE_N*128 bytes apart, 8-key groups 1024 bytes apart
              const uint64_t bd = smem_desc(vsm + kk * 2048, TILE_N * 128, 1024);
              mma_ts(TM_O, ptm + part_i * (TILE_N / 2) + kk * 8, bd, IDESC_PV,
                     (j == 0 && kk == 0 && part_i == 0) ? 0u : 1u);
            }
          }
          tc_commit(BAR(B_VEMPTY + s));
          tc_commit(BAR(B_PVDONE + buf));
        }
      }
      // all tensor work done before TMEM is released (every S product was read by
      // the softmax before the O product that follows it was issued)
      tc_commit(BAR(B_DRAIN));
      mbar_drain(BAR(B_DRAIN), 0);
    }
  } else if ((warp & 3) < n_quarters) {
    // ================= softmax / epilogue ==================================
    // Two threads per query row: `half` picks which 64 keys of a tile (and which
    // half of the head dimension in the epilogue) this thread handles.
    const int quarter = warp & 3;                          // TMEM lane quarter this warp may touch
    const int half = (warp - WARP_SOFTMAX0) >> 2;
    const int m = quarter * 32 + lane;                     // MMA row
    const int il = m / p.G, g = m % p.G;
    const int i = i0 + il;                                 // block row
    const bool row_valid = m < m_valid;
    const uint64_t mrow = row_valid ? p.mask[i] : 0ull;
    const uint32_t lane_addr = (uint32_t)(quarter * 32) << 16;
    const int sidx = half * (32 * n_quarters) + m;          // index among the n_soft softmax threads
    const float c = p.scale_log2;
    constexpr int HC = TILE_N / 2;                         // keys per thread and tile
    constexpr int OC = DH / 2;                             // output columns per thread
    uint32_t gt = 0;
    // A failed (expired) wait does not leave the loops: every thread keeps the
    // same control flow so that the pair barriers below always match up; once
    // the abort flag is set all later waits return at once and the block drains.
    bool ok = true;
    int4 own = make_int4(-1, 0, 0, 0);                     // the cut whose last piece this block holds
    while (part.next(sg)) {
      const int n_keys = sg.L + p.n_q;
      float m_ref = -CUDART_INF_F, l_sum = 0.f;
      for (int jt = 0, t = sg.t0; jt < sg.n; ++jt, t += sg.step, ++gt) {
        const uint32_t buf = gt % NS;
        ok &= mbar_wait(BAR(B_SFULL + buf), (gt / NS) & 1, abort_flag, p.err, 9);
        tc_fence_after();
        const uint32_t ts = TM_S0 + buf * TILE_N + lane_addr;
        uint32_t sreg[HC];
#pragma unroll
        for (int cc = 0; cc < HC / 32; ++cc) tmem_ld32(ts + half * HC + cc * 32, sreg + cc * 32);
        tmem_wait_ld();
        const int lo = t * TILE_N;
        const int kt = (p.page_table || (t + 1) * TILE_N <= n_keys) ? lo : n_keys - TILE_N;
        const bool masked = (kt + TILE_N > sg.L) || (kt < lo);   // (rows of a page past the last key: no mask bit names them)
        float tmax = -CUDART_INF_F;
        if (masked) {
          // Visibility of this thread's 64 keys as one 64-bit word (bit c: key k0 + c):
          // keys before `lo` belong to the previous tile; cached keys (< L) are seen by
          // every row; block keys by the Eq. 5 mask row of this query row.
          const int k0 = kt + half * HC;
          const int sh = sg.L - k0;                         // first block key sits at bit `sh`
          uint64_t vis;
          if (sh >= 64) vis = ~0ull;
          else if (sh > 0) vis = ((1ull << sh) - 1ull) | (mrow << sh);
          else if (sh > -64) vis = mrow >> (-sh);
          else vis = 0ull;
          const int below = lo - k0;                        // keys k0 .. lo-1 are not this tile's
          if (below >= 64) vis = 0ull;
          else if (below > 0) vis &= ~0ull << below;
          const uint32_t v0 = (uint32_t)vis, v1 = (uint32_t)(vis >> 32);
#pragma unroll
          for (int cidx = 0; cidx < HC; ++cidx) {
            const uint32_t w = cidx < 32 ? v0 : v1;
            const float v = ((w >> (cidx & 31)) & 1u) ? __uint_as_float(sreg[cidx]) : -CUDART_INF_F;
            sreg[cidx] = __float_as_uint(v);
          }
        }
        {
          // four independent running maxima: one chain over 64 values would cost 64 dependent steps
          float t4[4] = {-CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F, -CUDART_INF_F};
#pragma unroll
          for (int cidx = 0; cidx < HC; cidx += 2)
            t4[(cidx >> 1) & 3] = max3(t4[(cidx >> 1) & 3], __uint_as_float(sreg[cidx]), __uint_as_float(sreg[cidx + 1]));
          tmax = fmaxf(fmaxf(t4[0], t4[1]), fmaxf(t4[2], t4[3]));
        }
        // the row maximum needs the other half's keys; the pair barrier also orders
        // both threads' reads of S before either overwrites it with P
        float* xm = xmax + (gt & 1) * (2 * ROWS);
        xm[half * ROWS + m] = tmax;
        pair_sync(quarter);
        tmax = fmaxf(tmax, xm[(half ^ 1) * ROWS + m]);
        tmax *= c;                                         // c > 0
        if (!(tmax > -CUDART_INF_F)) tmax = -CUDART_INF_F; // also catches NaN
        const bool first = (jt == 0);
        const bool need = !first && (tmax > m_ref + RESCALE_THRESHOLD);
        if (first) m_ref = tmax;
        if (__any_sync(0xFFFFFFFFu, need)) {
          // lazy rescale of this row's accumulator; PV of the previous tile must be done
          ok &= mbar_wait(BAR(B_PVDONE + (gt - 1) % NS), ((gt - 1) / NS) & 1, abort_flag, p.err, 10);
          tc_fence_after();
          const float m_new = fmaxf(m_ref, tmax);
          const float f = (m_ref > -CUDART_INF_F) ? fast_exp2(m_ref - m_new) : 0.f;
          l_sum *= f;
          m_ref = m_new;
#pragma unroll 1
          for (int cc = 0; cc < OC / 32; ++cc) {
            uint32_t o[32];
            const uint32_t ta = TM_O + lane_addr + half * OC + cc * 32;
            tmem_ld32(ta, o);
            tmem_wait_ld();
#pragma unroll
            for (int x = 0; x < 32; ++x) o[x] = __float_as_uint(__uint_as_float(o[x]) * f);
            tmem_st32(ta, o);
          }
          tmem_wait_st();
        }
        // (rows past the last one are kept at zero, in Q and in P: under the power cap a product's energy is time,
        // and zeros cost little of it)
        const float m_use = !row_valid ? CUDART_INF_F : (m_ref > -CUDART_INF_F) ? m_ref : 0.f;
        // P = P_hi + P_lo, two bf16 terms: bf16 alone (8 significant bits) leaves
        // an output error near 1e-2 of the output RMS.  P_hi occupies columns
        // 0..63 of the S buffer, P_lo columns 64..127 (two keys per column).
        uint32_t lreg[HC / 2];
        const uint64_t cc = pack2(c, c), mm = pack2(-m_use, -m_use);
        uint64_t sum[2] = {0ull, 0ull};
#pragma unroll
        for (int x = 0; x < HC / 2; ++x) {
          float e0, e1;
          unpack2(fma2(pack2(__uint_as_float(sreg[2 * x]), __uint_as_float(sreg[2 * x + 1])), cc, mm), e0, e1);
          const float p0 = fast_exp2(e0), p1 = fast_exp2(e1);
          const uint64_t pp = pack2(p0, p1);
          sum[x & 1] = add2(sum[x & 1], pp);
          const __nv_bfloat162 hi = __floats2bfloat162_rn(p0, p1);   // .x (low half) = even key
          sreg[x] = *reinterpret_cast<const uint32_t*>(&hi);
          float l0, l1;
          low_terms(sreg[x], p0, p1, l0, l1);
          const __nv_bfloat162 lw = __floats2bfloat162_rn(l0, l1);
          lreg[x] = *reinterpret_cast<const uint32_t*>(&lw);
        }
        {
          float a0, a1;
          unpack2(add2(sum[0], sum[1]), a0, a1);
          l_sum += a0 + a1;
        }
        tmem_st32(ts + half * (HC / 2), sreg);
        tmem_st32(ts + TILE_N / 2 + half * (HC / 2), lreg);
        tmem_wait_st();
        if (p.page_table && kt + TILE_N > n_keys) {
          // Paged cache, last tile: the page's rows past the last key may hold anything, and 0 * NaN
          // would reach the output.  Once the V tile has landed the softmax threads clear those rows
          // (128 contiguous bytes per row and 64-wide half of d, whatever the swizzle inside them).
          // The softmax may run up to NS tiles ahead of the O product: where the V ring has fewer stages,
          // first make sure that the stage's previous tile has been consumed, so that the wait below
          // looks at the barrier phase of THIS tile and the stores cannot hit the tile before it.  (With
          // more stages than NS this tile's S product has waited for that already, and the barrier's
          // phase may be two further on: a wait for it would not return.)
          const uint32_t vs = gt % S::V_STAGES;
          if ((uint32_t)S::V_STAGES < NS && gt >= (uint32_t)S::V_STAGES) {
            const uint32_t pg = gt - S::V_STAGES;
            ok &= mbar_wait(BAR(B_PVDONE + pg % NS), (pg / NS) & 1, abort_flag, p.err, 18);
          }
          ok &= mbar_wait(BAR(B_VFULL + vs), (gt / S::V_STAGES) & 1, abort_flag, p.err, 17);
          const int first_bad = n_keys - kt;
          for (int it = first_bad * S::HALVES + sidx; it < TILE_N * S::HALVES; it += n_soft) {
            const int r = it / S::HALVES, hf = it % S::HALVES;
            const uint32_t vrow = sm_base + S::V_OFF + vs * S::TILE_BYTES + hf * (TILE_N * 128) + r * 128;
#pragma unroll
            for (int x = 0; x < 8; ++x)
              asm volatile("st.shared.v4.b32 [%0], {%1, %1, %1, %1};" ::"r"(vrow + x * 16), "r"(0u) : "memory");
          }
          asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        }
        tc_fence_before();
        mbar_arrive(BAR(B_PREADY + buf));
      }
      // ---- end of share: final output or partial ---------------------------
      ok &= mbar_wait(BAR(B_PVDONE + (gt - 1) % NS), ((gt - 1) / NS) & 1, abort_flag, p.err, 11);
      tc_fence_after();
      xsum[half * ROWS + m] = l_sum;
      pair_sync(quarter);
      const float l_tot = l_sum + xsum[(half ^ 1) * ROWS + m];
      const bool whole = sg.n == sg.T, to_smem = clustered && !whole;
      const int hq = sg.h * p.G + g;
      const int item = sg.b * p.H_kv + sg.h;
      float* pslot = to_smem ? reinterpret_cast<float*>(sm + S::PART_OFF)
                             : p.part + ((size_t)(item + group) * p.n_mblocks + mb) * (ROWS * (DH + 2));
      const float inv = (l_tot > 0.f) ? 1.f / l_tot : 0.f;
      // how this (sequence, head) was cut is read by attn_rows_merge_kernel (every group of the cut writes the same pair)
      int2 cut_d = make_int2(0, 0);
      if (sidx == 0 && !clustered) {
        cut_d = share_cut(prefix, p.B, p.n_groups, sg, group);
        if (!p.pieces && !p.merge_by_owner) p.desc[(size_t)item * p.n_mblocks + mb] = cut_d;
        // at most one per block: only its first share can start late
        if (sg.t0 > 0 && sg.t0 + sg.n == sg.T) own = make_int4(item, cut_d.x, cut_d.y, 0);
      }
      // A partial goes to the cluster's shared memory over the K stages: every softmax thread is past the last O
      // product by now, so all products of this block (its only share) have read them.
      // O leaves TMEM with one row per lane; written like that, a store instruction
      // would touch 32 different lines.  Each warp turns its 32 x 32 block through
      // shared memory so that eight lanes write 128 contiguous bytes of one row.
      float* stg = reinterpret_cast<float*>(sm + S::EPI_OFF) + (warp - WARP_SOFTMAX0) * (32 * S::EPI_PITCH);
      const int gsh = __ffs(p.G) - 1;                       // G is a power of two
      const float scale_o = whole ? inv : 1.f;
#pragma unroll 1
      for (int cc = 0; cc < OC / 32; ++cc) {
        uint32_t o[32];
        const int col = half * OC + cc * 32;
        tmem_ld32(TM_O + lane_addr + col, o);
        tmem_wait_ld();
#pragma unroll
        for (int x = 0; x < 8; ++x)
          *reinterpret_cast<float4*>(stg + lane * S::EPI_PITCH + 4 * x) =
              make_float4(__uint_as_float(o[4 * x]) * scale_o, __uint_as_float(o[4 * x + 1]) * scale_o,
                          __uint_as_float(o[4 * x + 2]) * scale_o, __uint_as_float(o[4 * x + 3]) * scale_o);
        __syncwarp();
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          const int rl = it * 4 + (lane >> 3), c4 = (lane & 7) * 4;   // row within the warp's block, first of 4 columns
          const int mr = quarter * 32 + rl;
          const float4 v = *reinterpret_cast<const float4*>(stg + rl * S::EPI_PITCH + c4);
          if (mr >= m_valid || !ok) continue;
          if (whole) {
            const int ir = i0 + (mr >> gsh), hr = sg.h * p.G + (mr & (p.G - 1));
            const size_t off = (((size_t)sg.b * p.n_q + ir) * p.H_q + hr) * DH + col + c4;
            if (p.out_dtype == SPACE_DTYPE_F32) {
              *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + off) = v;
            } else {
              const __nv_bfloat162 a0 = __floats2bfloat162_rn(v.x, v.y), a1 = __floats2bfloat162_rn(v.z, v.w);
              *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + off) =
                  make_uint2(*reinterpret_cast<const uint32_t*>(&a0), *reinterpret_cast<const uint32_t*>(&a1));
            }
          } else {
            *reinterpret_cast<float4*>(pslot + (size_t)mr * DH + col + c4) = v;
          }
        }
        __syncwarp();                                       // the block is rewritten by the next chunk
      }
      tc_fence_before();
      if (row_valid && half == 0 && ok) {
        if (whole) {
          if (p.lse)
            p.lse[((size_t)sg.b * p.H_q + hq) * p.n_q + i] = (m_ref + log2f(l_tot)) * 0.6931471805599453f;
        } else {
          pslot[ROWS * DH + m] = m_ref;
          pslot[ROWS * DH + ROWS + m] = l_tot;
        }
      }
      if (p.pieces && !clustered && !whole) {
        asm volatile("bar.sync 5, %0;" ::"r"(n_soft) : "memory");   // every thread's stores
        cut_d.x += item;                                    // slots are numbered by item + group
        if (sidx == 0) note_if_last(p, item, cut_d, p.arrived + (size_t)item * p.n_mblocks + mb, duties);
      }
    }
    if (p.merge_by_owner && sidx == 0) p.owner[blockIdx.x] = own;
  }
  if (clustered && cl_n > 1) {
    const uint32_t at = sm_base + S::PART_OFF;
    cluster_merge<DH>(p, cl_b, cl_h, i0, m_valid, cl_piece, p.pieces, cl_n, mb, at, at + ROWS * DH * 4, at + (ROWS * DH + ROWS) * 4,
                      abort_flag);
  }
  const bool fell_back = p.pieces && !clustered;            // (the same in every block of the grid)
  if (fell_back) cluster_duties<DH>(p, duties, abort_flag);

  // ---- teardown -----------------------------------------------------------
  tc_fence_before();
  __syncthreads();
  if (warp == WARP_MMA) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512u) : "memory");
  }
  if (threadIdx.x == 0 && *abort_flag && p.status) {
    for (int b = 0; b < p.B; ++b) atomicOr(p.status + b, SPACE_ST_TIMEOUT);
  }
  if ((clustered && cl_n > 1) || fell_back) cluster_leave();
}

// Combine the partials of every (sequence, kv head, query-row block) that was
// cut over several groups: one thread per 16 output bytes, all loads of a
// thread independent, running maximum / denominator / accumulator in one pass.
// grid = (B*H_kv*n_mblocks, ceil(rows*DH/4 / 128)), 128 threads.
template <int DH>
__global__ void __launch_bounds__(128) attn_rows_merge_kernel(const AttnParams p) {
  pdl_launch_dependents();
  pdl_wait();
  constexpr int C4 = DH / 4;
  // Large batches: one grid column per attention thread block (each holds the last
  // piece of at most one cut); small ones: one per (sequence, head, row block).
  int item = blockIdx.x / p.n_mblocks, b, h, n;
  const int mb = blockIdx.x % p.n_mblocks;
  int2 d;
  if (p.merge_by_owner) {
    // (one round trip to the partials' place; with the block's cut looked up by number in the descriptors it was two:
    // sixteen ragged sequences 130.2 -> 129.2, 24 short paged ones 89.4 -> 89.1 us a step)
    const int4 o = __ldcg(p.owner + blockIdx.x);
    if (o.x < 0) return;
    item = o.x; b = item / p.H_kv; h = item % p.H_kv; d = make_int2(o.y, o.z);
    n = d.y;
  } else {
    b = item / p.H_kv; h = item % p.H_kv;
    // both loads are issued before either is tested: one round trip, not two
    const int L = __ldcg(p.kv_len + b);
    d = __ldcg(p.desc + (size_t)item * p.n_mblocks + mb);
    if (L < 0 || (int64_t)L + p.n_q > p.s_cap) return;
    n = d.y;
  }
  if (n <= 1) return;                                       // written directly by the main kernel
  const int i0 = mb * p.rows_per_mb;
  const int m_valid = min(p.rows_per_mb, p.n_q - i0) * p.G;
  const int idx = blockIdx.y * 128 + threadIdx.x;
  if (idx >= m_valid * C4) return;
  const int r = idx / C4, c4 = idx % C4;
  const size_t slot_floats = (size_t)ROWS * (DH + 2);
  const float* ps = p.part + ((size_t)(item + d.x) * p.n_mblocks + mb) * slot_floats;
  const size_t gstride = (size_t)p.n_mblocks * slot_floats;
  MergeAcc acc;
  acc.clear();
#pragma unroll 8
  for (int x = 0; x < n; ++x, ps += gstride)
    acc.add(__ldcg(ps + ROWS * DH + r), __ldcg(ps + ROWS * DH + ROWS + r),
            __ldcg(reinterpret_cast<const float4*>(ps + (size_t)r * DH) + c4));
  acc.template store<DH>(p, b, h, i0, r, c4);
}

// ------------------------------------------------------------------ host side
void plan(const space_config* cfg, int sm_count, int k, AttnPlanHost* pl) {
  const int G = cfg->n_q_heads / cfg->n_kv_heads;
  const int n_q = (k + 1) * (k + 1);
  const int max_rows = ROWS / G;                            // block rows one MMA tile can hold
  pl->n_mblocks = (n_q + max_rows - 1) / max_rows;
  pl->rows_per_mblock = (n_q + pl->n_mblocks - 1) / pl->n_mblocks;
  int groups = sm_count / pl->n_mblocks;
  if (groups < 1) groups = 1;
  pl->n_ctas = groups * pl->n_mblocks;
}

template <int DH>
size_t smem_bytes(int max_batch) {
  return Smem<DH>::TABLE_OFF + (size_t)(2 * max_batch + 2) * sizeof(int);
}

template <int DH>
cudaError_t launch_dim(const AttnParams& p, int n_ctas, int max_batch, int size, cudaStream_t st, int* max_clusters) {
  // the kernel's limits are raised once per device (to the most any batch needs)
  static unsigned long long done_mask = 0;
  int dev = 0;
  cudaGetDevice(&dev);
  if (dev >= 64 || !((done_mask >> dev) & 1ull)) {
    cudaFuncSetAttribute(attn_rows_kernel<DH>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem_bytes<DH>(128));
    cudaFuncSetAttribute(attn_rows_kernel<DH>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (dev < 64) done_mask |= 1ull << dev;
  }
  return launch_clusters(attn_rows_kernel<DH>, n_ctas, THREADS, smem_bytes<DH>(max_batch), size, st, max_clusters, p, max_batch);
}
cudaError_t launch_main(int DH, const AttnParams& p, int n_ctas, int max_batch, int size, cudaStream_t st, int* max_clusters) {
  return DH == 128 ? launch_dim<128>(p, n_ctas, max_batch, size, st, max_clusters)
                   : launch_dim<64>(p, n_ctas, max_batch, size, st, max_clusters);
}

}  // namespace

int launch_attn_rows(space_ctx* ctx, const space_attn_args* a, const uint64_t* mask_rows,
                       cudaStream_t st) {
  const space_config& cfg = ctx->cfg;
  const int DH = cfg.head_dim;
  AttnPlanHost pl;
  plan(&cfg, ctx->sm_count, a->k, &pl);
  AttnParams p;
  memset(&p, 0, sizeof(p));
  p.B = a->batch; p.n_q = (a->k + 1) * (a->k + 1);
  p.H_q = cfg.n_q_heads; p.H_kv = cfg.n_kv_heads; p.G = p.H_q / p.H_kv;
  p.n_mblocks = pl.n_mblocks; p.rows_per_mb = pl.rows_per_mblock;
  p.n_groups = pl.n_ctas / pl.n_mblocks;
  p.out_dtype = a->out_dtype;
  p.s_cap = a->page_table ? (int64_t)a->pages_per_seq * SPACE_PAGE_SIZE : cfg.s_cap;
  p.page_table = a->page_table; p.pages_per_seq = a->pages_per_seq; p.n_pages = a->n_pages;
  p.scale_log2 = a->scale * 1.4426950408889634f;
  p.kv_len = a->kv_len; p.out = a->out; p.lse = a->lse; p.status = a->status;
  p.part = ctx->attn_part; p.err = ctx->counters + 3 * cfg.max_batch;
  p.desc = reinterpret_cast<int2*>(ctx->merge_cnt);
  p.owner = reinterpret_cast<int4*>(ctx->merge_cnt + (size_t)cfg.max_batch * cfg.n_kv_heads * 8 * 2);
  p.merge_by_owner = (a->batch * p.H_kv * p.n_mblocks > pl.n_ctas) ? 1 : 0;
  p.arrived = ctx->arrived;
  for (int i = 0; i < SPACE_MAX_ROWS; ++i) p.mask[i] = mask_rows[i];

  // TMA descriptors, rebuilt only when a base pointer or a stride changes
  const int64_t key[8] = {a->kv_stride_b, a->kv_stride_h, a->kv_stride_s, a->batch, p.n_q, -1,
                          a->page_table ? a->n_pages : 0, 0};
  if (ctx->tm_q_ptr != a->q || ctx->tm_k_ptr != a->k_cache || ctx->tm_v_ptr != a->v_cache ||
      memcmp(key, ctx->tm_key, sizeof(key)) != 0) {
    const cuuint64_t kd[4] = {(cuuint64_t)DH, (cuuint64_t)(a->page_table ? TILE_N : cfg.s_cap), (cuuint64_t)p.H_kv,
                              (cuuint64_t)(a->page_table ? a->n_pages : a->batch)};
    const cuuint64_t ks[3] = {(cuuint64_t)a->kv_stride_s * 2, (cuuint64_t)a->kv_stride_h * 2,
                              (cuuint64_t)a->kv_stride_b * 2};
    const cuuint32_t kb[4] = {64, TILE_N, 1, 1};
    const cuuint64_t qd[4] = {(cuuint64_t)DH, (cuuint64_t)p.H_q, (cuuint64_t)p.n_q, (cuuint64_t)a->batch};
    const cuuint64_t qs[3] = {(cuuint64_t)DH * 2, (cuuint64_t)p.H_q * DH * 2, (cuuint64_t)p.n_q * p.H_q * DH * 2};
    const cuuint32_t qb[4] = {64, (cuuint32_t)p.G, (cuuint32_t)p.rows_per_mb, 1};
    int rc = make_map((CUtensorMap*)ctx->tm_k, a->k_cache, kd, ks, kb);
    if (rc == SPACE_OK) rc = make_map((CUtensorMap*)ctx->tm_v, a->v_cache, kd, ks, kb);
    if (rc == SPACE_OK) rc = make_map((CUtensorMap*)ctx->tm_q, a->q, qd, qs, qb);
    if (rc != SPACE_OK) { ctx->tm_q_ptr = nullptr; return rc; }
    ctx->tm_q_ptr = a->q; ctx->tm_k_ptr = a->k_cache; ctx->tm_v_ptr = a->v_cache;
    memcpy(ctx->tm_key, key, sizeof(key));
  }
  memcpy(&p.tm_q, ctx->tm_q, sizeof(CUtensorMap));
  memcpy(&p.tm_k, ctx->tm_k, sizeof(CUtensorMap));
  memcpy(&p.tm_v, ctx->tm_v, sizeof(CUtensorMap));

  int n_ctas = pl.n_ctas, size = 1, n_clusters = 0;
  p.pieces = plan_clusters(a->batch * p.H_kv, p.n_mblocks, (p.s_cap + TILE_N - 1) / TILE_N, ctx->sm_count, ctx->cluster_fit[1],
                           [&](int sz, int* fit) { return launch_main(DH, p, ctx->sm_count / sz * sz, cfg.max_batch, sz, st, fit); },
                           &n_clusters);
  if (p.pieces) { size = p.pieces * p.n_mblocks; n_ctas = n_clusters * size; }
  p.n_groups = n_ctas / p.n_mblocks;
  {
    ProfScope ps(ctx, SPACE_K_ATTN, st);
    launch_main(DH, p, n_ctas, cfg.max_batch, size, st, nullptr);
    ctx->launches += 1;
  }
  if (!p.pieces) {
    const int m_valid_max = p.rows_per_mb * p.G;
    const dim3 mgrid(p.merge_by_owner ? n_ctas : a->batch * p.H_kv * p.n_mblocks, (m_valid_max * (DH / 4) + 127) / 128);
    ProfScope ps(ctx, SPACE_K_MERGE, st);
    if (DH == 128) launch_pdl(attn_rows_merge_kernel<128>, mgrid, dim3(128), 0, st, p);
    else launch_pdl(attn_rows_merge_kernel<64>, mgrid, dim3(128), 0, st, p);
    ctx->launches += 1;
  }
  return cuda_ok(cudaGetLastError());
}
