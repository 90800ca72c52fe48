// Device-side helpers of libjf: inline PTX for sm_103a (mbarrier, TMA, tcgen05, programmatic
// dependent launch), bounded waits and the shared error flag.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "jf_internal.h"

#define JF_DEV __device__ __forceinline__

typedef __nv_bfloat16 bf16;


JF_DEV void jf_set_error(int* err, int code) {
  if (err) atomicCAS(err, 0, code);
}

JF_DEV uint64_t jf_globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// Kernel ids of the timeline records.
enum TlKernel : unsigned {
  TL_NORM = 1, TL_NORM_ACC = 2, TL_QKV_FINISH = 3, TL_ATTN = 5, TL_GEMM = 10 /* + epilogue kind */,
  TL_EMBED = 20, TL_ACCEPT = 21, TL_COMMIT = 22, TL_ARGMAX = 23
};

// Timeline of the forward's kernels, compiled in only with -DJF_TIMELINE (the default build has
// none of it): thread 0 of every CTA records its kernel id, block, SM, entry time, the time it got
// past its dependency wait and its exit time, into a caller buffer set by jf_tl_enable().
#ifdef JF_TIMELINE
struct TlRec {
  unsigned kid, blk, smid, pad;
  unsigned long long t0, t1, t2;
};
constexpr int kTlMaxRecords = 2000000;
static __device__ TlRec* jf_tl_buf;  // one pair per translation unit, set by its own setter
static __device__ int* jf_tl_idx;
JF_DEV void jf_tl_record(unsigned kid, uint64_t t0, uint64_t t1) {
  if (!jf_tl_buf) return;
  const uint64_t t2 = jf_globaltimer();
  unsigned sm;
  asm volatile("mov.u32 %0, %%smid;" : "=r"(sm));
  const int i = atomicAdd(jf_tl_idx, 1);
  if (i < kTlMaxRecords) jf_tl_buf[i] = TlRec{kid, blockIdx.x, sm, 0u, t0, t1, t2};
}
#define JF_TL_ENTRY()                       \
  const uint64_t jf_tl_t0 = jf_globaltimer(); \
  uint64_t jf_tl_t1 = 0
#define JF_TL_WAITED() (jf_tl_t1 = jf_globaltimer())
#define JF_TL_EXIT(kid)                                               \
  do {                                                                \
    if (threadIdx.x == 0) jf_tl_record((unsigned)(kid), jf_tl_t0, jf_tl_t1); \
  } while (0)
#define JF_TL_SETTER(name)                                                     \
  cudaError_t name(void* records, void* counter) {                             \
    cudaError_t e = cudaMemcpyToSymbol(jf_tl_buf, &records, sizeof(void*));   \
    return e != cudaSuccess ? e : cudaMemcpyToSymbol(jf_tl_idx, &counter, sizeof(void*)); \
  }
#else
#define JF_TL_ENTRY() \
  do {                \
  } while (0)
#define JF_TL_WAITED() \
  do {                 \
  } while (0)
#define JF_TL_EXIT(kid) \
  do {                  \
  } while (0)
#endif

// ------------------------------------------------------------------------------------------
// Programmatic dependent launch. Every kernel of the chain but the forward's first (k_embed, a full
// boundary) calls pdl_wait() before it reads anything an earlier kernel of the chain wrote (and before it
// exits), so completion stays transitive.
// ------------------------------------------------------------------------------------------
JF_DEV void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
JF_DEV void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// ------------------------------------------------------------------------------------------
// Shared-memory addresses, mbarriers
// ------------------------------------------------------------------------------------------
JF_DEV uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

JF_DEV void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}

JF_DEV void fence_mbar_init() { asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory"); }

JF_DEV void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// (predicated off when `on` is false, like the copies below)
JF_DEV void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes, bool on = true) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %2, 0;\n\t"
      "@q mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n\t}" ::"r"(bar),
      "r"(bytes), "r"((int)on)
      : "memory");
}

JF_DEV void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// True once phase `parity` is complete. The thread may be suspended for up to kWaitHintNs meanwhile: a
// wait that polls takes issue slots from the warps that feed it.
constexpr uint32_t kWaitHintNs = 20000u;
JF_DEV bool mbar_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(kWaitHintNs)
      : "memory");
  return ok != 0;
}

// Wait for phase `parity` of an mbarrier, giving up after `limit_ns` nanoseconds.
JF_DEV bool mbar_wait_bounded(uint32_t bar, uint32_t parity, uint64_t limit_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = jf_globaltimer();
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if (jf_globaltimer() - t0 > limit_ns) return false;
  }
}

// Barrier ID of N threads (whole warps, in any convergence); true when every thread's `ok` is. A wait's outcome
// may differ from thread to thread when its phase completes near the limit: threads that meet at barriers or in
// warp-wide instructions afterwards agree on it first, and leave together.
template <int ID, int N>
JF_DEV bool sync_and(bool ok) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((int)ok), "n"(ID), "n"(N)
      : "memory");
  return r != 0;
}

// ------------------------------------------------------------------------------------------
// Thread-block clusters: ranks, cluster-wide barrier
// ------------------------------------------------------------------------------------------
JF_DEV uint32_t cluster_rank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of shared-memory address `a` in the cluster's CTA `rank`
JF_DEV uint32_t map_to_rank(uint32_t a, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
  return r;
}
JF_DEV void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
JF_DEV void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// ------------------------------------------------------------------------------------------
// TMA (cp.async.bulk.tensor) loads with an L2 cache-policy hint
// ------------------------------------------------------------------------------------------
JF_DEV uint64_t l2_policy_evict_first() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(p));
  return p;
}

JF_DEV uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// 2-D tiled load: box at coordinates (c0 = innermost, c1) into shared memory, completing
// `bytes` on mbarrier `bar`. The innermost coordinate is always a multiple of 64 elements
// (128 bytes) here, which keeps every copy on a 16-byte boundary.
JF_DEV void tma_load_2d(uint32_t smem_dst, const void* tmap, uint32_t bar, int c0, int c1, uint64_t policy, bool on) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %6, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;\n\t}" ::"r"(smem_dst),
      "l"(tmap), "r"(c0), "r"(c1), "r"(bar), "l"(policy), "r"((int)on)
      : "memory");
}

// Contiguous copy (both addresses and the size multiples of 16 bytes) and 3-D tiled load, without a
// cache-policy hint.
JF_DEV void bulk_load(uint32_t smem_dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
JF_DEV void tma_load_3d_plain(uint32_t smem_dst, const void* tmap, uint32_t bar, int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(
          smem_dst),
      "l"(tmap), "r"(c0), "r"(c1), "r"(c2), "r"(bar)
      : "memory");
}

// 2-D tiled load by a CTA of a pair (cta_group::2): into its own shared memory, completing on an
// mbarrier of either CTA (a shared::cluster address).
JF_DEV void tma_load_2d_pair(uint32_t smem_dst, const void* tmap, uint32_t bar, int c0, int c1, uint64_t policy,
                             bool on) {
  asm volatile(
      "{\n\t.reg .pred q;\n\tsetp.ne.b32 q, %6, 0;\n\t"
      "@q cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%2, %3}], [%4], %5;\n\t}" ::"r"(smem_dst),
      "l"(tmap), "r"(c0), "r"(c1), "r"(bar), "l"(policy), "r"((int)on)
      : "memory");
}

JF_DEV void tma_prefetch_desc(const void* tmap) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(tmap) : "memory");
}

// ------------------------------------------------------------------------------------------
// tcgen05 (5th-generation tensor cores, accumulator in tensor memory)
// ------------------------------------------------------------------------------------------
JF_DEV void tmem_alloc(uint32_t smem_result, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols)
               : "memory");
}
JF_DEV void tmem_relinquish() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory"); }
JF_DEV void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
// One lane of a converged warp.
JF_DEV bool elect_one() {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(r));
  return r != 0;
}
// The same for a pair of CTAs (a cluster of two): allocation by one warp of each CTA.
JF_DEV void tmem_alloc_pair(uint32_t smem_result, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_result), "r"(ncols)
               : "memory");
}
JF_DEV void tmem_relinquish_pair() { asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory"); }
JF_DEV void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
JF_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
JF_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// D[tmem] (+)= A[smem] * B[smem]^T, kind::f16 (bf16 inputs, fp32 accumulate), one CTA.
JF_DEV void tc_mma_bf16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem], kind::f16 with the A operand (packed 16-bit values, two to a
// column) in tensor memory.
JF_DEV void tc_mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrive once on an mbarrier when all previously issued tcgen05 MMAs of this thread complete.
JF_DEV void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// A pair's MMA (M = 256: 128 rows of A and of D in each CTA, half of B's rows in each), issued by one
// thread of the cluster's rank 0; and the arrival, on the mbarrier at this offset in both CTAs, once
// all previously issued ones are complete.
JF_DEV void tc_mma_bf16_pair(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
JF_DEV void tc_commit_pair(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;" ::"r"(bar),
      "h"((uint16_t)3)
      : "memory");
}

// The same arrival on rank 0's mbarrier alone.
JF_DEV void tc_commit_pair_local(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// Load 16 consecutive fp32 columns of this warp's 32 TMEM lanes (lane = thread).
JF_DEV void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// Load 32 consecutive fp32 columns of this warp's 32 TMEM lanes (lane = thread).
JF_DEV void tmem_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

// Store 16 consecutive 32-bit columns of this warp's 32 TMEM lanes (lane = thread); complete after
// tmem_wait_st().
JF_DEV void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]),
      "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
      : "memory");
}
JF_DEV void tmem_wait_st() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// Shared-memory matrix descriptor for a K-major operand tile written by TMA with 128-byte
// swizzle: rows of 128 bytes, 8-row swizzle atoms `sbo` bytes apart (stride byte offset),
// descriptor version 1, layout type 2 (SWIZZLE_128B).
JF_DEV uint64_t sdesc_k_sw128(uint32_t saddr, uint32_t sbo = 1024u) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(16u >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Shared-memory descriptor of an MN-major operand with the 128-byte swizzle: rows of 64 MN
// elements (128 bytes) at consecutive K indices, swizzled in 8-row groups `sbo` bytes apart (stride
// byte offset); consecutive 64-element MN atoms `lbo` bytes apart (leading byte offset).
JF_DEV uint64_t sdesc_mn_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor, kind::f16: fp32 accumulator, bf16 A and B, both K-major, M x N.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}
// The same with fp16 A and B (A and B of one MMA always share their type).
__host__ __device__ constexpr uint32_t idesc_f16_f32(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// ------------------------------------------------------------------------------------------
// Small numeric helpers
// ------------------------------------------------------------------------------------------
template <typename T>
JF_DEV T to_act(float v);
template <>
JF_DEV float to_act<float>(float v) { return v; }
template <>
JF_DEV bf16 to_act<bf16>(float v) { return __float2bfloat16_rn(v); }

JF_DEV float act_to_f32(float v) { return v; }
JF_DEV float act_to_f32(bf16 v) { return __bfloat162float(v); }

JF_DEV float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

JF_DEV float silu_f(float x) { return x / (1.0f + __expf(-x)); }
