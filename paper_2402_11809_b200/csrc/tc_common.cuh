// PTX helpers shared by the tensor-core kernels of libspace (attn_tc.cu, attn_rows.cu, lmhead.cu):
// mbarrier handling with bounded waits, TMA tile loads, tcgen05 fences / commits / products and the
// shared-memory matrix descriptor of sm_100, and the host's tensor maps.  One copy, so that the wait protocol that the
// time-out test exercises (space_debug_wait_timeout) is the one every kernel uses.
#pragma once
#include "common.cuh"
#include <cuda.h>
#include <stdint.h>

namespace tc {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.b32 %0, 1, 0, p;\n\t}"
      : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
  return ok != 0;
}
// True in one lane of the (converged) warp.  The roles that issue tensor-core products and TMA requests pick
// their thread with this, not with a comparison of the lane number: the compiler knows that one thread is left
// then and keeps the descriptors in uniform registers.  Picked by lane number every operand of every
// instruction is moved there first; measured, cycles per M = 128, K = 16 product in a row, by lane / elected:
// both operands in shared memory N = 32 108 / 59, N = 64 108 / 75, N = 128 108 / 107, N = 224 155 / 155
// (43 + N/2), first operand in TMEM N = 128 108 / 74 (10 + N/2).
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n\t.reg .pred q;\n\telect.sync _|q, 0xffffffff;\n\tselp.b32 %0, 1, 0, q;\n\t}"
      : "=r"(p));
  return p != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

// Bounded wait on an mbarrier phase: at most `limit_ns` of wall time (%globaltimer, looked at
// every 256 polls).  Returns false when the limit expired or another thread of the block gave up
// before; the first expiry sets the block's abort flag and records `site` in *err (first one wins).
// Once the flag is set every later wait returns at once, so the block drains instead of blocking.
// sleep_ns > 0: sleep between polls (leaves the issue slots to the working warps).
// (Inlined here; the kernels keep one out-of-line copy and try the barrier once before they call it: a wait
// that has nothing to wait for takes 65 cycles that way instead of 166, and a role's loop has two or three of
// them per tile.)
__device__ __forceinline__ bool mbar_wait_bounded(uint32_t bar, uint32_t parity, volatile int* abort_flag,
                                               int* err, int site, uint64_t limit_ns, uint32_t sleep_ns) {
  if (*abort_flag) return mbar_try(bar, parity);            // draining: never block
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try(bar, parity)) return true;
    if (sleep_ns) __nanosleep(sleep_ns);
    if ((it & 255u) == 255u) {
      if (*abort_flag) return false;
      const uint64_t now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) break;
    }
  }
  *abort_flag = 1;
  atomicCAS(err, 0, site);
  return false;
}
// Bounded wait without the abort protocol (used while draining before exit).
__device__ __forceinline__ void mbar_drain_bounded(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  uint64_t t0 = 0;
  for (uint32_t it = 0;; ++it) {
    if (mbar_try(bar, parity)) return;
    if ((it & 255u) == 255u) {
      const uint64_t now = global_ns();
      if (t0 == 0) t0 = now;
      else if (now - t0 > limit_ns) return;
    }
  }
}

// Tiled TMA load of one box of a 4-D tensor map into shared memory, completion on `bar`.
// (No cluster multicast anywhere: every block fetches its own tiles.)
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const CUtensorMap* tm, uint32_t bar,
                                            int c0, int c1, int c2, int c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];"
      ::"r"(dst), "l"((uint64_t)tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3) : "memory");
}
// The same load with an L2 policy word (see l2_evict_first_policy).
__device__ __forceinline__ void tma_load_4d_hint(uint32_t dst, const CUtensorMap* tm, uint32_t bar,
                                                 int c0, int c1, int c2, int c3, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4, %5, %6}], [%2], %7;"
      ::"r"(dst), "l"((uint64_t)tm), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(pol) : "memory");
}
// Asks L2 for one box of a 4-D tensor map without waiting for it and without a destination in
// shared memory.  L2 is the point of coherence for global memory, so the request may be made
// while an earlier kernel can still write the tensor: the later load sees the final bytes.
__device__ __forceinline__ void tma_prefetch_l2_4d(const CUtensorMap* tm, int c0, int c1, int c2, int c3, uint64_t pol) {
  asm volatile(
      "cp.async.bulk.prefetch.tensor.4d.L2.global.tile.L2::cache_hint [%0, {%1, %2, %3, %4}], %5;"
      ::"l"((uint64_t)tm), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "l"(pol) : "memory");
}
// Policy for data that is read once per step: its lines are evicted first and leave the cache to
// what is read again (kernel code, lengths, partials).
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
  uint64_t pol;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
  return pol;
}

__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after()  { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}
// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss(uint32_t d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts(uint32_t d, uint32_t a, uint64_t bdesc, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}"
      ::"r"(d), "r"(a), "l"(bdesc), "r"(idesc), "r"(acc) : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor, 128-byte swizzle, descriptor version of sm_100.
// lbo / sbo (leading / stride byte offsets) in bytes.
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFF);
  d |= (uint64_t)((lbo >> 4) & 0x3FFF) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFF) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Two floats per instruction (64-bit register pairs) and a maximum of three: the softmax loops are bound by
// instruction issue.
__device__ __forceinline__ uint64_t pack2(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// What two floats leave over their bf16 values (the halves of `hi`, p0's in the low one): one mixed-precision
// instruction each, where widening both halves and subtracting takes three for the two.  64 keys of a softmax row
// (scale, exponential, sum, both terms): 407 -> 311 instructions a warp, 1450 -> 1243 cycles with two warps per
// scheduler.  The difference is exact: its bits are the ones of p that bf16 dropped.
__device__ __forceinline__ void low_terms(uint32_t hi, float p0, float p1, float& l0, float& l1) {
  asm("{\n\t.reg .b16 a, b, m;\n\tmov.b32 {a, b}, %4;\n\tmov.b16 m, 0xBF80;\n\t"       // -1
      "fma.rn.f32.bf16 %0, a, m, %2;\n\tfma.rn.f32.bf16 %1, b, m, %3;\n\t}"
      : "=f"(l0), "=f"(l1) : "f"(p0), "f"(p1), "r"(hi));
}

// 2^x by the hardware approximation
__device__ __forceinline__ float fast_exp2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// ---- host side: tensor map of a 4-D bf16 tensor whose boxes are 64 elements (128 bytes, swizzled) wide
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

static inline EncodeTiledFn get_encode() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) != cudaSuccess ||
        qres != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = (EncodeTiledFn)ptr;
  }
  return fn;
}

static inline int make_map(CUtensorMap* tm, const void* base, const cuuint64_t dims[4], const cuuint64_t strides_bytes[3],
                           const cuuint32_t box[4]) {
  EncodeTiledFn enc = get_encode();
  if (!enc) return SPACE_E_CUDA;
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  // (L2 promotion of 128 B, 64 B or none: the projection of 36 rows of 32000 52.4 us per call instead of 49.8)
  const CUresult r = enc(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides_bytes,
                         box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                         CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? SPACE_OK : SPACE_E_CUDA;
}

}  // namespace tc
