// Thin inline-PTX wrappers for the sm_103a features the kernels use:
// mbarriers, TMA tensor loads and stores, and the tcgen05 tensor-core family (TMEM
// allocation, MMA with shared-memory / tensor-memory operands, commits, and
// tensor-memory loads and stores).  Every wait in this file is bounded: it
// gives up after a wall-clock limit read from %globaltimer or when a
// CTA-wide abort flag is raised, and reports failure to the caller, so a
// missing arrive can never spin a warp forever.
#pragma once

#include <cstdint>
#include <cuda.h>

namespace sva {
namespace ptx {

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ---------------------------------------------------------------- launches
//
// Programmatic dependent launch: a kernel launched with the attribute may start
// while the kernel before it in the stream still runs (once every block of that
// one has called pdl_launch_dependents or exited), and calls pdl_wait before it
// touches any memory that another kernel may write or read: pdl_wait returns
// when every earlier kernel has completed and its writes are visible.

__device__ __forceinline__ void pdl_wait() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void pdl_launch_dependents() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Loads of what a caller passes: an earlier kernel may still be writing it
// while this one is resident ahead of its pdl_wait.  The read-only path (__ldg,
// ld.global.nc) is defined only for memory that nothing writes as long as the
// kernel runs, so it is kept for the rotation tables; these are ordinary loads,
// which stay behind pdl_wait (both are volatile).

__device__ __forceinline__ float4 ld_global_f4(const void* p) {
  float4 v;
  asm volatile("ld.global.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "l"(p));
  return v;
}

// One word, or `other` without a load where `load` is false.
__device__ __forceinline__ uint32_t ld_global_u32_if(const uint32_t* p, bool load, uint32_t other) {
  uint32_t v;
  asm volatile(
      "{\n"
      " .reg .pred q;\n"
      " setp.ne.u32 q, %2, 0;\n"
      " mov.b32 %0, %3;\n"
      " @q ld.global.u32 %0, [%1];\n"
      "}\n"
      : "=&r"(v)
      : "l"(p), "r"((uint32_t)load), "r"(other));
  return v;
}

// ---------------------------------------------------------------- mbarrier

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Has the phase with the given parity completed?  Never suspends (try_wait may,
// for microseconds, where the phase is far off or never comes).
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n"
      " .reg .pred p;\n"
      " mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n"
      "}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits for the phase with the given parity to complete.  Returns false if
// `abort_flag` becomes non-zero or `timeout_ns` of wall-clock time elapse
// first; the caller then takes its error path.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          const volatile int* abort_flag, uint64_t timeout_ns) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  uint32_t polls = 0;
  while (true) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((++polls & 31u) == 0u) {
      if (*abort_flag) return false;
      if (globaltimer_ns() - t0 > timeout_ns) return false;
    }
  }
}

// ---------------------------------------------------------------- TMA

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tma_load_2d_hint(void* dst, const CUtensorMap* map, uint64_t* bar,
                                                 int32_t c0, int32_t c1, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint"
      " [%0], [%1, {%3, %4}], [%2], %5;" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "l"(policy)
      : "memory");
}

__device__ __forceinline__ void tma_load_4d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int32_t c0, int32_t c1, int32_t c2, int32_t c3) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2),
      "r"(c3)
      : "memory");
}

__device__ __forceinline__ uint64_t l2_policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// Tile store shared -> global through the tensor map (bulk-group
// completion); elements outside the tensor's extent are not written.
__device__ __forceinline__ void tma_store_2d(const CUtensorMap* map, uint32_t src, int32_t c0,
                                             int32_t c1) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(src), "r"(c0), "r"(c1)
               : "memory");
}

__device__ __forceinline__ void bulk_commit_group() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Waits until at most N committed bulk groups of this thread still read
// their shared-memory source.
template <int N>
__device__ __forceinline__ void bulk_wait_group_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

// Waits until at most N committed bulk groups of this thread are incomplete
// (their global writes done).
template <int N>
__device__ __forceinline__ void bulk_wait_group() {
  asm volatile("cp.async.bulk.wait_group %0;" ::"n"(N) : "memory");
}

// Makes this thread's generic-proxy shared-memory writes visible to the
// async proxy (a TMA store that reads them next).
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void st_shared_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c,
                                             uint32_t d) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c),
               "r"(d)
               : "memory");
}

__device__ __forceinline__ uint4 ld_shared_v4(uint32_t addr) {
  uint4 v;
  asm volatile("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}

// ---------------------------------------------------------------- clusters

// The shared::cluster address of the variable at `addr` (a shared::cta
// address of this CTA) in the CTA of rank `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}

__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n"
               "barrier.cluster.wait.acquire.aligned;" ::: "memory");
}

__device__ __forceinline__ void st_cluster_v4(uint32_t cluster_addr, float a, float b, float c,
                                              float d) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(cluster_addr), "f"(a),
               "f"(b), "f"(c), "f"(d)
               : "memory");
}

__device__ __forceinline__ void st_cluster_f32(uint32_t cluster_addr, float a) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(cluster_addr), "f"(a) : "memory");
}

__device__ __forceinline__ float ld_shared_f32(uint32_t addr) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(addr) : "memory");
  return v;
}

// ---------------------------------------------------------------- tcgen05

// Allocates `ncols` tensor-memory columns (power of two, >= 32); the base
// address is written to shared memory at `dst`.  Must be executed by one
// whole warp.
__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst)),
               "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

// Instruction descriptor for kind::f16 with bf16 A and B and an fp32
// accumulator.  Field layout (PTX ISA, tcgen05 instruction descriptor):
// [4,6) D format (1 = f32), [7,10) A format (1 = bf16), [10,13) B format,
// [15] A major (0 = K-major), [16] B major (1 = MN-major), [17,23) N >> 3,
// [24,29) M >> 4.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(uint32_t M, uint32_t N, bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((b_mn_major ? 1u : 0u) << 16) |
         ((N >> 3) << 17) | ((M >> 4) << 24);
}

// Shared-memory matrix descriptor for a 128-byte-swizzled operand whose
// swizzle atoms start on 1024-byte boundaries.  [0,14) start >> 4,
// [16,30) leading-dimension byte offset >> 4, [32,46) stride-dimension byte
// offset >> 4, [46,48) version = 1, [61,64) layout = 2 (128B swizzle).
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t saddr, uint32_t lbo_bytes,
                                                uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>((lbo_bytes >> 4) & 0x3FFFu) << 16;
  d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1u) << 46;
  d |= static_cast<uint64_t>(2u) << 61;
  return d;
}

// Warp-wide calls: every lane of a converged warp executes them and elect.sync
// picks the issuing lane (the lowest active one, so always the same thread: a
// commit tracks the MMAs of the thread that issues it).  A loop that stays
// warp-uniform keeps descriptors and TMEM addresses in the uniform datapath;
// issuing from a lane-0-only branch was measured about 8% slower end to end in
// the attention kernel.

// D[tmem] (+)= A[smem] * B[smem]
__device__ __forceinline__ void mma_ss_warp(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      " .reg .pred p, e;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// D[tmem] (+)= A[tmem] * B[smem]
__device__ __forceinline__ void mma_ts_warp(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      " .reg .pred p, e;\n"
      " setp.ne.b32 p, %4, 0;\n"
      " elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
      "}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Runs of MMAs over consecutive K slices with one election for the run (an
// election per MMA costs the issuing warp about as long as a 128 x 64 x 16 MMA
// takes the tensor pipe).  The first MMA accumulates where `accumulate` says,
// the others always.
//
// Four smem x smem MMAs, descriptors `step` (in 16-byte units) apart; the first
// overwrites D.
__device__ __forceinline__ void mma_ss_warp_x4(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                               uint64_t step, uint32_t idesc) {
  asm volatile(
      "{\n"
      " .reg .pred z, t, e;\n"
      " setp.ne.b32 z, 0, 0;\n"
      " setp.eq.b32 t, 0, 0;\n"
      " elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %5, %9, z;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %2, %6, %9, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %3, %7, %9, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], %4, %8, %9, t;\n"
      "}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(a_desc + step), "l"(a_desc + 2 * step), "l"(a_desc + 3 * step),
      "l"(b_desc), "l"(b_desc + step), "l"(b_desc + 2 * step), "l"(b_desc + 3 * step), "r"(idesc)
      : "memory");
}

// Eight tmem x smem MMAs over 128 keys: A (packed bf16) advances by 8 columns,
// B (MN-major, 128-byte rows) by 16 rows = 2048 bytes.
__device__ __forceinline__ void mma_ts_warp_x8(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                               uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n"
      " .reg .pred p, t, e;\n"
      " setp.ne.b32 p, %18, 0;\n"
      " setp.eq.b32 t, 0, 0;\n"
      " elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %9, %17, p;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%2], %10, %17, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%3], %11, %17, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%4], %12, %17, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%5], %13, %17, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%6], %14, %17, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%7], %15, %17, t;\n"
      " @e tcgen05.mma.cta_group::1.kind::f16 [%0], [%8], %16, %17, t;\n"
      "}\n" ::"r"(d_tmem),
      "r"(a_tmem), "r"(a_tmem + 8), "r"(a_tmem + 16), "r"(a_tmem + 24), "r"(a_tmem + 32),
      "r"(a_tmem + 40), "r"(a_tmem + 48), "r"(a_tmem + 56), "l"(b_desc), "l"(b_desc + 128),
      "l"(b_desc + 256), "l"(b_desc + 384), "l"(b_desc + 512), "l"(b_desc + 640),
      "l"(b_desc + 768), "l"(b_desc + 896), "r"(idesc), "r"(accumulate)
      : "memory");
}

// Arrives once on `bar` when every tcgen05 operation that the issuing lane
// issued so far has completed.
__device__ __forceinline__ void mma_commit_warp(uint64_t* bar) {
  asm volatile(
      "{\n"
      " .reg .pred e;\n"
      " elect.sync _|e, 0xffffffff;\n"
      " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
      "}\n" ::"r"(smem_u32(bar))
      : "memory");
}

#define SVA_R8(i) "=r"(r[i]), "=r"(r[i + 1]), "=r"(r[i + 2]), "=r"(r[i + 3]), \
                  "=r"(r[i + 4]), "=r"(r[i + 5]), "=r"(r[i + 6]), "=r"(r[i + 7])
#define SVA_W8(i) "r"(r[i]), "r"(r[i + 1]), "r"(r[i + 2]), "r"(r[i + 3]), \
                  "r"(r[i + 4]), "r"(r[i + 5]), "r"(r[i + 6]), "r"(r[i + 7])
#define SVA_RW8(i) "+r"(r[i]), "+r"(r[i + 1]), "+r"(r[i + 2]), "+r"(r[i + 3]), \
                   "+r"(r[i + 4]), "+r"(r[i + 5]), "+r"(r[i + 6]), "+r"(r[i + 7])

// Each thread of the warp reads 32 consecutive 32-bit columns of its own
// lane (lane = warp's 32-lane quarter + lane id) starting at `taddr`.
// The registers are not valid until tmem_wait_ld(r) has run.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32"
      " {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : SVA_R8(0), SVA_R8(8), SVA_R8(16), SVA_R8(24)
      : "r"(taddr));
}

// tmem_ld32 that also returns the maximum of the 32 loaded fp32 values
// (tcgen05.ld.red, sm_103a): a row max of S without a max tree in registers.
// `mx`, like the registers, is valid only after a tcgen05.wait::ld that
// names it (tmem_wait_ld_max).
__device__ __forceinline__ void tmem_ld32_max(uint32_t taddr, uint32_t (&r)[32], float& mx) {
  asm volatile(
      "tcgen05.ld.red.sync.aligned.32x32b.x32.max.f32"
      " {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, %32, [%33];"
      : SVA_R8(0), SVA_R8(8), SVA_R8(16), SVA_R8(24), "=f"(mx)
      : "r"(taddr));
}

// Waits for this thread's outstanding tensor-memory loads.  Taking the
// registers as read-write operands keeps the compiler from hoisting their
// uses above the wait.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&r)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : SVA_RW8(0), SVA_RW8(8), SVA_RW8(16), SVA_RW8(24)
               :
               : "memory");
}

// 16-lane forms (shape 16x32bx2): a warp reads or writes 16 TMEM lanes (its
// lane quarter's half at the address), and the two half-warps take different
// columns: thread t < 16 gets lane t at columns [c, c + 32), thread t >= 16
// gets lane t - 16 at columns [c + OFF, c + OFF + 32).  So two threads share
// one row and each holds 32 consecutive columns of it.
template <int OFF>
__device__ __forceinline__ void tmem_ld16x2_32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.16x32bx2.x32.b32"
      " {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32], %33;"
      : SVA_R8(0), SVA_R8(8), SVA_R8(16), SVA_R8(24)
      : "r"(taddr), "n"(OFF));
}

// tmem_ld16x2_32 that also returns the maximum of the thread's 32 values.
template <int OFF>
__device__ __forceinline__ void tmem_ld16x2_32_max(uint32_t taddr, uint32_t (&r)[32], float& mx) {
  asm volatile(
      "tcgen05.ld.red.sync.aligned.16x32bx2.x32.max.f32"
      " {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, %32, [%33], %34;"
      : SVA_R8(0), SVA_R8(8), SVA_R8(16), SVA_R8(24), "=f"(mx)
      : "r"(taddr), "n"(OFF));
}

template <int OFF>
__device__ __forceinline__ void tmem_st16x2_32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x32bx2.x32.b32 [%0], %33,"
      " {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      SVA_W8(0), SVA_W8(8), SVA_W8(16), SVA_W8(24), "n"(OFF)
      : "memory");
}

// Same as tmem_st16x2_32 with the 32 columns taken from two 16-register halves.
template <int OFF>
__device__ __forceinline__ void tmem_st16x2_32_halves(uint32_t taddr, const uint32_t* a,
                                                      const uint32_t* b) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x32bx2.x32.b32 [%0], %33,"
      " {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
      "r"(a[8]), "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]),
      "r"(a[15]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
      "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]), "r"(b[12]), "r"(b[13]),
      "r"(b[14]), "r"(b[15]), "n"(OFF)
      : "memory");
}

// Orders reads of tmem_ld*_max results after the loads completed.
__device__ __forceinline__ void tmem_wait_ld_max2(float (&mx)[2]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" : "+f"(mx[0]), "+f"(mx[1]) : : "memory");
}

// Orders reads of four tmem_ld32_max results after the loads completed.
__device__ __forceinline__ void tmem_wait_ld_max(float (&mx)[4]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+f"(mx[0]), "+f"(mx[1]), "+f"(mx[2]), "+f"(mx[3])
               :
               : "memory");
}

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0],"
      " {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      SVA_W8(0), SVA_W8(8), SVA_W8(16), SVA_W8(24)
      : "memory");
}

// Same as tmem_st32 with the 32 columns taken from two 16-register halves.
__device__ __forceinline__ void tmem_st32_halves(uint32_t taddr, const uint32_t* a,
                                                 const uint32_t* b) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0],"
      " {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,"
      "%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};" ::"r"(taddr),
      "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(a[4]), "r"(a[5]), "r"(a[6]), "r"(a[7]),
      "r"(a[8]), "r"(a[9]), "r"(a[10]), "r"(a[11]), "r"(a[12]), "r"(a[13]), "r"(a[14]),
      "r"(a[15]), "r"(b[0]), "r"(b[1]), "r"(b[2]), "r"(b[3]), "r"(b[4]), "r"(b[5]), "r"(b[6]),
      "r"(b[7]), "r"(b[8]), "r"(b[9]), "r"(b[10]), "r"(b[11]), "r"(b[12]), "r"(b[13]),
      "r"(b[14]), "r"(b[15])
      : "memory");
}

__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

#undef SVA_R8
#undef SVA_W8
#undef SVA_RW8

}  // namespace ptx
}  // namespace sva
