// What the two tensor-core attention kernels (attn_tc.cu, attn_rows.cu) share: page look-ups, the arithmetic of the
// flat tile list, and how partial results of a (sequence, kv head, query-row block) that was cut over several
// thread blocks are combined: in the shared memory of a cluster, or from global memory by the cluster of the block that
// stored the last of them (by a merge kernel of its own where no clusters are launched).  `P` is a kernel's parameter struct (G, H_q, n_q, n_mblocks, out_dtype, out, lse, part;
// page_table, pages_per_seq, n_pages, status).
#pragma once
#include "common.cuh"
#include "tc_common.cuh"
#include <math_constants.h>

namespace attn {

constexpr int ROWS = 128;              // query rows of a partial's slot in global memory
constexpr int MAX_CLUSTER = 16;        // blocks per cluster (more than 8 need the opt-in)
// The clustered cut is taken while its longest piece has at most this many tiles more than an even share of
// all tiles: that is about what the cut over the grid costs on top (starting more than one share per block,
// the merge in global memory).
constexpr int CLUSTER_SLACK = 10;

// Shared memory of another block of the cluster.
__device__ __forceinline__ uint32_t map_cluster(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float ld_cluster(uint32_t a) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a) : "memory");
  return v;
}

// Page of tile t of sequence b (paged cache).  An entry outside the pool is flagged and answered
// with a page past the pool's end: the TMA load then fills the tile with zeros.
// (flag = false: a request made before the length is known, for a tile the sequence may not have.)
template <class P>
__device__ __forceinline__ int page_of(const P& p, int b, int t, bool flag = true) {
  const int pg = t < p.pages_per_seq ? p.page_table[(int64_t)b * p.pages_per_seq + t] : -1;
  if (pg >= 0 && pg < p.n_pages) return pg;
  if (flag && p.status) atomicOr(p.status + b, SPACE_ST_BAD_PAGE);
  return p.n_pages;
}

// floor(a * b / c) for a*b that may need 64 bits; 32-bit division when it fits
__host__ __device__ __forceinline__ long long muldiv(long long a, long long b, long long c) {
  const unsigned long long prod = (unsigned long long)a * (unsigned long long)b;
  if ((prod >> 32) == 0) return (long long)((unsigned)prod / (unsigned)c);
  return (long long)(prod / (unsigned long long)c);
}
// group that owns flat tile f (largest g with floor(W*g/NG) <= f)
__host__ __device__ __forceinline__ int group_of(long long f, long long W, long long NG) {
  const unsigned long long num = (unsigned long long)(f + 1) * (unsigned long long)NG - 1ull;
  if ((num >> 32) == 0) return (int)((unsigned)num / (unsigned)W);
  return (int)(num / (unsigned long long)W);
}
// {first group, number of groups} that the list gives the T tiles of (sequence b, kv head h) to.  The lengths alone say
// it, so every piece of a cut comes to the same answer, one whose waits ran out as well: the pieces are counted by it.
__host__ __device__ __forceinline__ int2 list_cut(const int* prefix, int B, int n_groups, int share_cost, int b, int h, int T) {
  const long long W = prefix[B];
  const long long NG = W < n_groups ? W : n_groups;
  const long long f0 = (long long)prefix[b] + (long long)h * (T + share_cost) + share_cost;   // its first tile
  const int g0 = group_of(f0, W, NG);
  return make_int2(g0, group_of(f0 + T - 1, W, NG) - g0 + 1);
}

// Query row r of the row block that starts at block row i0, columns 4 c4 .. of (sequence b, kv head h).
template <int DH, class P>
__device__ __forceinline__ void store_out(const P& p, int b, int h, int i0, int r, int c4, const float4& v) {
  const int gsh = __ffs(p.G) - 1;                           // G is a power of two
  const int ri = i0 + (r >> gsh), hq = h * p.G + (r & (p.G - 1));
  const size_t off = (((size_t)b * p.n_q + ri) * p.H_q + hq) * DH + c4 * 4;
  if (p.out_dtype == SPACE_DTYPE_F32) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p.out) + off) = v;
  } else {
    const __nv_bfloat162 x = __floats2bfloat162_rn(v.x, v.y), y = __floats2bfloat162_rn(v.z, v.w);
    *reinterpret_cast<uint2*>(reinterpret_cast<__nv_bfloat16*>(p.out) + off) =
        make_uint2(*reinterpret_cast<const uint32_t*>(&x), *reinterpret_cast<const uint32_t*>(&y));
  }
}
template <class P>
__device__ __forceinline__ void store_lse(const P& p, int b, int h, int i0, int r, float v) {
  const int gsh = __ffs(p.G) - 1;
  p.lse[((size_t)b * p.H_q + h * p.G + (r & (p.G - 1))) * p.n_q + i0 + (r >> gsh)] = v;
}

// Four output elements of one query row from the partials of a cut: running reference, denominator and
// accumulator.
struct MergeAcc {
  float mx, den;
  float4 a;
  __device__ __forceinline__ void clear() { mx = -CUDART_INF_F; den = 0.f; a = make_float4(0.f, 0.f, 0.f, 0.f); }
  __device__ __forceinline__ void add(float m, float l, const float4& o) {
    const float mn = fmaxf(mx, m);
    if (mn > -CUDART_INF_F) {
      const float e0 = tc::fast_exp2(mx - mn), e1 = tc::fast_exp2(m - mn);
      den = den * e0 + l * e1;
      a.x = a.x * e0 + o.x * e1; a.y = a.y * e0 + o.y * e1;
      a.z = a.z * e0 + o.z * e1; a.w = a.w * e0 + o.w * e1;
    }
    mx = mn;
  }
  // four partials at once (a missing one: m = -inf, l = 0, o = 0): one maximum, independent weights, where one
  // after the other is a chain of two exponentials each (sixteen pieces for each of two sequences of 500..1500 keys,
  // attention call in graph replay: one query head 8.75 -> 8.47 us, eight 12.1 -> 11.5)
  __device__ __forceinline__ void add4(const float (&m)[4], const float (&l)[4], const float4 (&o)[4]) {
    const float mn = fmaxf(fmaxf(fmaxf(mx, m[0]), fmaxf(m[1], m[2])), m[3]);
    if (mn > -CUDART_INF_F) {
      const float e = tc::fast_exp2(mx - mn);
      den *= e; a.x *= e; a.y *= e; a.z *= e; a.w *= e;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float w = tc::fast_exp2(m[j] - mn);
        den += l[j] * w; a.x += o[j].x * w; a.y += o[j].y * w; a.z += o[j].z * w; a.w += o[j].w * w;
      }
    }
    mx = mn;
  }
  template <int DH, class P>
  __device__ __forceinline__ void store(const P& p, int b, int h, int i0, int r, int c4) const {
    const float rd = 1.f / den;
    store_out<DH>(p, b, h, i0, r, c4, make_float4(a.x * rd, a.y * rd, a.z * rd, a.w * rd));
    if (p.lse && c4 == 0) store_lse(p, b, h, i0, r, (mx + log2f(den)) * 0.6931471805599453f);
  }
};

// The pieces of a cluster's pair meet: every block combines its part of the rows from all pieces' shared
// memory (o_at / m_at / l_at: addresses of the accumulators, references and sums, the same in every block).
// All threads of the cluster's blocks take part, those of a piece without tiles too; every wait before this
// is bounded, so all of them arrive.  cluster_leave() must follow before the block exits.
template <int DH, class P>
__device__ __forceinline__ void cluster_merge(const P& p, int b, int h, int i0, int m_valid, int piece, int pieces, int n,
                                              int mb, uint32_t o_at, uint32_t m_at, uint32_t l_at, volatile int* abort_flag) {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  const int stride = pieces * (int)blockDim.x;
  for (int idx = piece * (int)blockDim.x + (int)threadIdx.x; idx < m_valid * (DH / 4) && !*abort_flag; idx += stride) {
    const int r = idx / (DH / 4), c4 = idx % (DH / 4);
    MergeAcc acc;
    acc.clear();
    for (int x0 = 0; x0 < n; x0 += 4) {                     // all loads of a batch are issued before any is used
      float ms[4], ls[4];
      float4 ov[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        ms[j] = -CUDART_INF_F; ls[j] = 0.f; ov[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (x0 + j < n) {
          const uint32_t rank = (uint32_t)((x0 + j) * p.n_mblocks + mb);
          ms[j] = ld_cluster(map_cluster(m_at + r * 4, rank));
          ls[j] = ld_cluster(map_cluster(l_at + r * 4, rank));
          ov[j] = ld_cluster4(map_cluster(o_at + (r * DH + c4 * 4) * 4, rank));
        }
      }
      acc.add4(ms, ls, ov);
    }
    acc.template store<DH>(p, b, h, i0, r, c4);
  }
  // No block leaves while another may still read its shared memory: this half says that this block has read
  // (relaxed: nothing is handed over, so it need not wait for the output's stores).
  __syncwarp();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_leave() {
  __syncwarp();
  asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
}

// Clusters were launched, but the lengths are too unequal for them: each cut's pieces go to global memory, and the piece
// that finds all the others stored notes the cut in its block's shared memory (no merge kernel follows such a launch;
// as the rule for larger batches this was slower, 137 against 130 us per step of sixteen ragged sequences when it was
// tried: every piece waits for its fence and its atomic).  At the end the blocks of a cluster combine together what any
// of them noted.  Called by one thread, after a barrier that orders the stores of all of the block's threads before it,
// for every piece of the cut and with the same cut, also where a wait ran out and nothing was stored: a piece that did
// not count, or counted to another number, would leave the counter off for every later call.
constexpr int MAX_DUTIES = 2;          // a block's share of the list starts and ends inside one cut each, at most
template <class P>
__device__ __forceinline__ void note_if_last(const P& p, int item, int2 cut, int* arrived, int4* duties) {
  __threadfence();
  if (atomicAdd(arrived, 1) != cut.y - 1) return;
  *arrived = 0;                                             // ready for the next launch
  __threadfence();
  duties[duties[0].x < 0 ? 0 : 1] = make_int4(item, cut.x, cut.y, 0);
}
// All threads of the cluster's blocks take part (every wait before this is bounded, so all of them arrive); duties: the
// block's own list, MAX_DUTIES entries, item -1 where there is none.  cluster_leave() must follow before the block exits.
// The last block alone, before: one sequence of 16000 keys with 392 query rows (four cuts over 36 pieces) 60.0 us a
// step, this way 30.1; of 16000 paged keys with 2 x 392 rows of 64 46.5 -> 30.9; nine sequences of 800 to 16384 keys, 4 x 36
// rows, 71.3 -> 62.4.  (Out of line, or with sixteen loads a batch, the kernels' loops were compiled otherwise: the step
// of one 7B-shaped sequence 18.15 -> 18.3 and 19.2.)
template <int DH, class P>
__device__ __forceinline__ void cluster_duties(const P& p, const int4* duties, volatile int* abort_flag) {
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  static_assert(MAX_CLUSTER * MAX_DUTIES <= 32, "a lane per entry");
  const int size = p.pieces * p.n_mblocks, lane = threadIdx.x & 31, threads = size * (int)blockDim.x;
  uint32_t rank;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(rank));
  int4 mine = make_int4(-1, 0, 0, 0);                       // lane e: entry e of the cluster, rank e / MAX_DUTIES
  if (lane < size * MAX_DUTIES) {
    const uint32_t at = map_cluster(tc::smem_u32(duties) + (lane % MAX_DUTIES) * 16, (uint32_t)(lane / MAX_DUTIES));
    asm volatile("ld.shared::cluster.v4.b32 {%0, %1, %2, %3}, [%4];" : "=r"(mine.x), "=r"(mine.y), "=r"(mine.z), "=r"(mine.w) : "r"(at) : "memory");
  }
  const size_t slot_floats = (size_t)ROWS * (DH + 2), gstride = (size_t)p.n_mblocks * slot_floats;
  // the cuts' elements one after another over the cluster's threads: next is this thread's place before the cut's first one
  int next = (int)(rank * blockDim.x + threadIdx.x);
  for (unsigned todo = __ballot_sync(0xFFFFFFFFu, mine.x >= 0); todo && !*abort_flag; todo &= todo - 1) {
    const int e = __ffs(todo) - 1;
    const int item = __shfl_sync(0xFFFFFFFFu, mine.x, e), slot = __shfl_sync(0xFFFFFFFFu, mine.y, e), n = __shfl_sync(0xFFFFFFFFu, mine.z, e);
    // (the cluster's ranks are blocks in order: row block rank % n_mblocks)
    const int b = item / p.H_kv, h = item % p.H_kv, mb = e / MAX_DUTIES % p.n_mblocks;
    const int i0 = mb * p.rows_per_mb, count = min(p.rows_per_mb, p.n_q - i0) * p.G * (DH / 4);
    const float* ps = p.part + ((size_t)slot * p.n_mblocks + mb) * slot_floats;
    int idx = next;
    for (; idx < count; idx += threads) {
      const int r = idx / (DH / 4), c4 = idx % (DH / 4);
      MergeAcc acc;
      acc.clear();
      for (int x0 = 0; x0 < n; x0 += 8) {                  // all loads of a batch are issued before any is used
        float ms[8], ls[8];
        float4 ov[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          ms[j] = -CUDART_INF_F; ls[j] = 0.f; ov[j] = make_float4(0.f, 0.f, 0.f, 0.f);
          if (x0 + j < n) {
            const float* pj = ps + (size_t)(x0 + j) * gstride;
            ms[j] = __ldcg(pj + ROWS * DH + r);
            ls[j] = __ldcg(pj + ROWS * DH + ROWS + r);
            ov[j] = __ldcg(reinterpret_cast<const float4*>(pj + (size_t)r * DH) + c4);
          }
        }
#pragma unroll
        for (int g = 0; g < 8; g += 4) {
          const float m4[4] = {ms[g], ms[g + 1], ms[g + 2], ms[g + 3]}, l4[4] = {ls[g], ls[g + 1], ls[g + 2], ls[g + 3]};
          const float4 o4[4] = {ov[g], ov[g + 1], ov[g + 2], ov[g + 3]};
          acc.add4(m4, l4, o4);
        }
      }
      acc.template store<DH>(p, b, h, i0, r, c4);
    }
    next = idx - count;                                     // (the next cut's elements follow this one's)
  }
  // no block leaves while another may still read its list
  __syncwarp();
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
}

// Whether the clustered cut serves these lengths (all lanes of a warp call this; every warp gets the same
// answer): the longest piece in tiles against an even share.  tiles_of(L): tiles of a sequence of length L.
template <class P, class F>
__device__ __forceinline__ bool cluster_fits(const P& p, int lane, F tiles_of) {
  int Tmax = 0, W = 0;
  if (p.B == 1) {
    Tmax = W = tiles_of(p.kv_len[0]);
  } else {
    for (int b0 = 0; b0 < p.B; b0 += 32) {
      const int T = b0 + lane < p.B ? tiles_of(p.kv_len[b0 + lane]) : 0;
      Tmax = max(Tmax, __reduce_max_sync(0xFFFFFFFFu, T));
      W += __reduce_add_sync(0xFFFFFFFFu, T);
    }
  }
  return (Tmax + p.pieces - 1) / p.pieces <= (W * p.H_kv + p.n_groups - 1) / p.n_groups + CLUSTER_SLACK;
}

// Host side: launch with programmatic serialization and, when size > 1, clusters of `size` blocks; with
// max_clusters, no launch but the number of such clusters that can be resident.
template <typename K, typename... Args>
static inline cudaError_t launch_clusters(K kernel, int n_ctas, int threads, size_t smem, int size, cudaStream_t st,
                                          int* max_clusters, const Args&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(n_ctas); cfg.blockDim = dim3(threads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = size; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  if (max_clusters) {
    cfg.attrs = attr + 1; cfg.numAttrs = 1;
    return cudaOccupancyMaxActiveClusters(max_clusters, kernel, &cfg);
  }
  cfg.attrs = attr; cfg.numAttrs = size > 1 ? 2 : 1;
  return cudaLaunchKernelEx(&cfg, kernel, args...);
}

// The clustered cut of `pairs` (sequence, kv head) pairs: as many pieces as there are SMs for (and tiles a
// sequence may have), in clusters of pieces * n_mblocks blocks that fit next to one another.  fit[size]:
// clusters of that size that can be resident, 0 = not asked yet (ask(size) tells).  Returns the pieces (0: more
// pairs than fit) and the number of clusters to launch.
template <typename Ask>
static inline int plan_clusters(int pairs, int n_mblocks, int64_t cap_tiles, int sm_count, int* fit, Ask ask, int* n_clusters) {
  for (int c = cap_tiles < MAX_CLUSTER / n_mblocks ? (int)cap_tiles : MAX_CLUSTER / n_mblocks; c >= 1; --c) {
    const int size = c * n_mblocks;
    if (pairs * size > sm_count) continue;
    if (fit[size] == 0) {
      if (size == 1) fit[size] = sm_count;
      else if (ask(size, &fit[size]) != cudaSuccess || fit[size] == 0) { cudaGetLastError(); fit[size] = -1; }
    }
    if (fit[size] < pairs) continue;
    // Where no length that fits the cache makes a piece too long for cluster_fits, the cut over the grid will not be
    // needed.  A launch that then leaves half of the chip idle launches no more blocks than it needs, and the next
    // kernel's, or another stream's, start on the rest at once (space_step_host, whose verification runs beside the
    // attention: two sequences of eight heads 127.9 -> 108.7 us, of one head 46.7 -> 43.6; one small step 12.40 -> 12.28).
    // With 120 blocks of 148 it was 17.52 -> 17.91 (odd5): the next kernel's blocks crowd on the few idle SMs.
    *n_clusters = pairs * size <= sm_count / 2 && (cap_tiles + c - 1) / c <= CLUSTER_SLACK ? pairs : fit[size];
    return c;
  }
  return 0;
}

}  // namespace attn
