// Device-side building blocks for the sm_103a kernels: mbarriers with bounded
// waits, 1-D bulk async copies (global -> shared), and the tcgen05 tensor-core
// instructions (TMEM allocation, MMA, commit, TMEM loads).  All inline PTX.
#pragma once
#include <cstdint>
#include <cuda_runtime.h>

#include "pn_internal.h"

namespace pn {

// ---------------------------------------------------------------- status ---
// Device-detected errors are recorded in one int32 word; the first error wins.
__device__ __forceinline__ void set_status(int32_t* status, int32_t code) {
  if (status) atomicCAS(status, 0, code);
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// -------------------------------------------------------------- mbarrier ---
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

// Makes barrier initialisation visible to the async proxy and other threads.
__device__ __forceinline__ void fence_barrier_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
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
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Waits for the phase with the given parity to complete.  Gives up after
// timeout_ns nanoseconds, or as soon as *abort becomes non-zero, and returns
// false in that case.  No wait in this library is unbounded.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, uint64_t timeout_ns,
                                          volatile int32_t* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
#pragma unroll 1
    for (int i = 0; i < 32; ++i)
      if (mbar_try_wait(bar, parity)) return true;
    if (*abort) return false;
    if (globaltimer_ns() - t0 > timeout_ns) return false;
  }
}

// ------------------------------------------------- flags across CTAs ---
// Global flags written by one CTA and read by others in the same launch.
__device__ __forceinline__ int32_t ld_acquire_gpu(const int32_t* p) {
  int32_t v;
  asm volatile("ld.acquire.gpu.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_release_gpu(int32_t* p, int32_t v) {
  asm volatile("st.release.gpu.global.b32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}
// Orders this thread's generic-proxy global accesses with later async-proxy
// (bulk copy) accesses: used by a writer after building data that other
// CTAs' bulk copies read, and by a reader before issuing such copies.
__device__ __forceinline__ void fence_proxy_async_global() {
  asm volatile("fence.proxy.async.global;" ::: "memory");
}
// Waits until *p >= need (acquire).  Gives up after timeout_ns nanoseconds or
// once *abort is non-zero and returns false then.
__device__ __forceinline__ bool wait_flag_geq(const int32_t* p, int32_t need, uint64_t timeout_ns,
                                              volatile int32_t* abort) {
  if (ld_acquire_gpu(p) >= need) return true;
  const uint64_t t0 = globaltimer_ns();
  while (true) {
    __nanosleep(64);
    if (ld_acquire_gpu(p) >= need) return true;
    if (*abort) return false;
    if (globaltimer_ns() - t0 > timeout_ns) return false;
  }
}

// ----------------------------------------------------------- bulk copies ---
// 1-D bulk copy global -> shared memory, completion counted in bytes on the
// mbarrier.  Both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_g2s(uint32_t dst_smem, const void* src, uint32_t bytes,
                                         uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          dst_smem),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

// Same, with an L2 cache-policy hint (operand tiles are re-read by other CTAs).
__device__ __forceinline__ void bulk_g2s_hint(uint32_t dst_smem, const void* src, uint32_t bytes,
                                              uint64_t* bar, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes.L2::cache_hint [%0], "
      "[%1], %2, [%3], %4;" ::"r"(dst_smem),
      "l"(src), "r"(bytes), "r"(smem_u32(bar)), "l"(policy)
      : "memory");
}

// 2-D tensor copy global -> shared memory (zeros outside the tensor),
// completion counted in bytes on the mbarrier.
__device__ __forceinline__ void tma_load_2d(uint32_t dst_smem, const void* map, int x, int y,
                                            uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, "
      "%3}], [%4];" ::"r"(dst_smem),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(smem_u32(bar))
      : "memory");
}

// 1-D bulk copy shared -> global memory in the calling thread's bulk group.
// Both addresses 16-byte aligned, size a multiple of 16.
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src_smem, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst),
               "r"(src_smem), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}
// Waits until at most N of this thread's bulk groups still read shared memory.
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}
// Waits until every bulk group of this thread has completed.
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}
// Orders this thread's generic-proxy shared-memory writes before later
// async-proxy (bulk copy) reads of them.
__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// Per-thread asynchronous copies global -> shared memory (16 bytes, both
// addresses 16-byte aligned, or 4 bytes): `bytes` of the source are read, the
// rest of the destination is zeroed.
__device__ __forceinline__ void cp_async16(uint32_t dst_smem, const void* src, uint32_t bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst_smem), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst_smem, const void* src, uint32_t bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst_smem), "l"(src),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void cp_async_commit() {
  asm volatile("cp.async.commit_group;" ::: "memory");
}
// Waits until at most N of this thread's groups are in flight.
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Programmatic dependent launch.  A kernel launched with programmatic stream
// serialisation may start while the kernel before it in the stream still
// runs; pdl_wait() returns once that kernel (and, transitively, everything
// before it) has completed and its memory is visible (a no-op for a normal
// launch).  Every kernel of the product path calls it before touching global
// memory, then pdl_trigger() lets the next kernel's CTAs be scheduled, so
// their launch overlaps this kernel's run instead of following its end.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

__device__ __forceinline__ uint64_t policy_evict_last() {
  uint64_t p;
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(p));
  return p;
}

// ------------------------------------------------------------ tcgen05 ---
__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem_word, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem_word)),
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

// Shared-memory matrix descriptor for a K-major operand tile stored with the
// 128-byte swizzle: rows of 128 bytes, groups of 8 rows 1024 bytes apart.
//   bits  0-13 start address >> 4      bits 16-29 leading byte offset >> 4
//   bits 32-45 stride byte offset >> 4 bits 46-47 descriptor version (1)
//   bits 61-63 layout (2 = 128-byte swizzle)
__device__ __forceinline__ uint64_t sdesc_sw128(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;
  d |= static_cast<uint64_t>(1024 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(2) << 61;
  return d;
}

// Instruction descriptor (kind::f16 / kind::tf32 / kind::f8f6f4), dense,
// FP32 accumulator, both operands K-major.
//   bits 4-5 D format (1 = F32), 7-9 A format, 10-12 B format,
//   bits 17-22 N >> 3, bits 24-28 M >> 4.
__host__ __device__ constexpr uint32_t idesc_make(uint32_t ab_fmt, uint32_t M, uint32_t N) {
  return (1u << 4) | (ab_fmt << 7) | (ab_fmt << 10) | ((N >> 3) << 17) | ((M >> 4) << 24);
}

// Operand kinds of the tensor-core path.
enum MmaKind : int { KIND_F16 = 0, KIND_TF32 = 1, KIND_F8 = 2 };

template <int KIND>
__device__ __forceinline__ void mma_ss(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                       uint32_t idesc, uint32_t accumulate) {
  if constexpr (KIND == KIND_F16) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else if constexpr (KIND == KIND_TF32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}

// Arrives once on the mbarrier when every tcgen05 operation this thread
// issued before has completed.
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// 32 lanes x 32 consecutive 32-bit columns: thread t of the warp receives the
// 32 columns of TMEM lane (warp's lane quarter * 32 + t).
__device__ __forceinline__ void tmem_ld_32x32b_x32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_ld_wait() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ------------------------------------------------------- CTA pairs ---
// Two CTAs of a cluster sharing one tensor-core tile (cta_group::2): the
// pair's MMA reads A and B halves from both CTAs' shared memory at the same
// offsets and writes each CTA's TMEM; rank 0 issues it.
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_id_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t nclusters_x() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}
// Address of the same shared-memory location in CTA `rank` of the cluster.
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
// Arrive on an mbarrier of the other CTA of a pair (the default release
// semantics at CTA scope).  The pair's arrivals only report that this CTA's
// tcgen05 loads of an accumulator have completed (tcgen05.wait::ld, then the
// thread-sync fence), so no data is published through them and no fence at
// cluster scope is needed (issued per operand stage, such fences measured at
// half the pair's MMA rate).
__device__ __forceinline__ void mbar_arrive_peer(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// 2-D tensor copy global -> this CTA's shared memory for a CTA pair
// (cta_group::2): the completion is counted on `bar_cluster`, an mbarrier of
// either CTA of the pair (the pair's operand stages all complete on rank 0's
// barrier, which the MMA issuer waits on).
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst_smem, const void* map, int x, int y,
                                                 uint32_t bar_cluster, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%2, %3}], [%4], %5;" ::"r"(dst_smem),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(bar_cluster), "l"(policy)
      : "memory");
}
// Every thread of both CTAs: release / acquire at cluster scope.
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::
                   : "memory");
}
__device__ __forceinline__ void tmem_alloc_pair(uint32_t* dst_smem_word, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem_word)),
               "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish_pair() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc_pair(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
template <int KIND>
__device__ __forceinline__ void mma_pair(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
  if constexpr (KIND == KIND_F16) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else if constexpr (KIND == KIND_TF32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::2.kind::f8f6f4 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}
// Arrives once on the mbarrier at this offset in every CTA of cta_mask when
// the pair MMAs issued before have completed.
__device__ __forceinline__ void mma_commit_pair(uint64_t* bar, uint16_t cta_mask) {
  asm volatile(
      "tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 "
      "[%0], %1;" ::"r"(smem_u32(bar)),
      "h"(cta_mask)
      : "memory");
}

// Hardware base-2 logarithm / exponential (MUFU), subnormals supported.
__device__ __forceinline__ float lg2_approx(float x) {
  float r;
  asm("lg2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float ex2_approx(float x) {
  float r;
  asm("ex2.approx.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

// OR-reduction across the `count` threads of named barrier `id`.
__device__ __forceinline__ bool bar_red_or(bool v, uint32_t id, uint32_t count) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, %2, %3, p;\n\tselp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"(static_cast<uint32_t>(v)), "r"(id), "r"(count)
      : "memory");
  return r != 0;
}

__device__ __forceinline__ void bar_sync_named(uint32_t id, uint32_t count) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(count) : "memory");
}

// Offset of byte b (0..127) of row r (0..127) inside one 16 KB operand tile
// image laid out with the 128-byte swizzle: the 16-byte chunk index is XORed
// with the row index modulo 8.
__host__ __device__ __forceinline__ uint32_t sw128_offset(uint32_t r, uint32_t b) {
  return r * 128u + ((((b >> 4) ^ (r & 7u)) & 7u) << 4) + (b & 15u);
}

// Two FP32 values in one register pair; their products, sums and fused products
// in one instruction (each rounded as by itself).
__device__ __forceinline__ uint64_t f32x2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ void f32x2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
__device__ __forceinline__ uint64_t f32x2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f32x2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t f32x2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// x / s for a power of two s: a multiply by the exact reciprocal when 1/s is
// a normal float (identical rounding), else a division.
__device__ __forceinline__ float div_pow2(float x, float s, float inv, bool inv_ok) {
  return inv_ok ? x * inv : x / s;
}
__device__ __forceinline__ bool recip_exact(float s) {
  return s >= 1.1754944e-38f && s <= 8.507059e37f;
}

// x^(2^k - 1) = x * x^2 * x^4 * ... * x^(2^(k-1)) (k correctly rounded
// squarings and products); 1 for k = 0.
__device__ __forceinline__ float pow_pm1(float x, int k) {
  float r = 1.0f;
  for (int t = 0; t < k; ++t) {
    r *= x;
    x *= x;
  }
  return r;
}

// Gradient factor of the adjoint: acc * x'^(p-1) / s with x' = x / s, p = 2^k,
// s a power of two.  x' = m 2^e is split by frexpf and the chain
// x'^(2^k - 1) = x' x'^2 x'^4 ... x'^(2^(k-1)) runs on mantissas in
// [0.5, 1) with the exponents summed exactly, each product renormalised, so
// no intermediate under- or overflows however small x' is; the total
// exponent is applied once at the end (ldexpf: one rounding, into the
// subnormal range if the result lies there).  x = 0 gives 0 for k >= 1.
static __device__ __noinline__ float grad_factor_frexp(float acc, float x, float s, int k) {
  int ls, ex;
  frexpf(s, &ls);
  ls -= 1;                        // s = 2^ls
  float xm = frexpf(x, &ex);      // x = xm 2^ex, so x' = xm 2^(ex - ls)
  ex -= ls;
  float rm = 1.0f;
  int re = 0;
  // A product of two values in [0.5, 1] lies in [0.25, 1) (it cannot round
  // up to 1), so renormalising it into [0.5, 1) is at most one doubling:
  // the same mantissa and exponent as frexpf of the product.
  for (int t = 0; t < k; ++t) {
    rm *= xm;
    re += ex;
    if (rm < 0.5f) {
      rm *= 2.0f;
      re -= 1;
    }
    xm *= xm;
    ex *= 2;
    if (xm < 0.5f) {
      xm *= 2.0f;
      ex -= 1;
    }
  }
  return ldexpf(acc * rm, re - ls);
}

// The same, bit for bit (rounding does not depend on the scale of a mantissa),
// for p <= 128 without a branch: with the mantissa in [0.75, 1.5) the chain stays
// between 2^-53 and 2^75, so it is renormalised once, at the end, and the
// exponent goes on in two factors of normal powers of two, the second 1 unless
// the result leaves the range of normal values.  About 40 instructions; with x'
// uniform half of the entries took the renormalising loop at p = 64, some 150
// instructions for every warp.  With the row-wise epilogue: a 2048^3 gradient GEMM in 3xTF32 185 -> 95 us.
__device__ __forceinline__ float grad_factor(float acc, float x, float s, int k) {
  if (k > 7) return grad_factor_frexp(acc, x, s, k);
  // s = 2^ls and x = m 2^ex; subnormal values scaled up first
  const bool tiny_s = s < 1.17549435e-38f, tiny_x = x < 1.17549435e-38f;
  const int ls = static_cast<int>(__float_as_uint(tiny_s ? s * 16777216.0f : s) >> 23) -
                 (tiny_s ? 127 + 24 : 127);
  const uint32_t xb = __float_as_uint(tiny_x ? x * 16777216.0f : x);
  const bool upper = (xb & 0x00400000u) != 0u;  // mantissa in [1.5, 2): halve it
  const int ex = static_cast<int>(xb >> 23) - (tiny_x ? 127 + 24 : 127) + (upper ? 1 : 0);
  float y = __uint_as_float((xb & 0x007fffffu) | (upper ? 0x3f000000u : 0x3f800000u));
  float r = 1.0f;
  for (int t = 0; t < k; ++t) {
    r = __fmul_rn(r, y);
    y = __fmul_rn(y, y);
  }
  // r = m 2^(exponent - 126) with m in [0.5, 1) (k = 0: r = 1 as it is)
  const uint32_t rb = __float_as_uint(r), one = k == 0 ? 0x00800000u : 0u;
  const int e = (ex - ls) * ((1 << k) - 1) - ls + static_cast<int>((rb - one) >> 23) - 126;
  const float g = __fmul_rn(acc, __uint_as_float((rb & 0x007fffffu) | (0x3f000000u + one)));
  // g's own exponent joins e (unless g is 0, subnormal, infinite or a NaN), so that
  // only the last factor rounds
  const uint32_t gb = __float_as_uint(g), eg = (gb >> 23) & 0xffu;
  const bool plain = eg - 1u < 254u;
  const float m = plain ? __uint_as_float((gb & 0x807fffffu) | 0x3f800000u) : g;
  const int et = plain ? e + static_cast<int>(eg) - 127 : e;
  const int e1 = min(max(et, -126), 127), e2 = min(max(et - e1, -126), 127);
  const float v = __fmul_rn(__fmul_rn(m, __uint_as_float(static_cast<uint32_t>(e1 + 127) << 23)),
                            __uint_as_float(static_cast<uint32_t>(e2 + 127) << 23));
  return k > 0 && x == 0.0f ? acc * 0.0f : v;  // (a NaN or infinite sum is not hidden)
}

// Smallest power of two >= m (m > 0, finite); 1 for m == 0.  Returns +inf
// when that power is beyond the float range.
__device__ __forceinline__ float pow2_ceil_f(float m) {
  if (!(m > 0.0f)) return 1.0f;
  int e;
  const float f = frexpf(m, &e);
  return ldexpf(1.0f, f == 0.5f ? e - 1 : e);
}

}  // namespace pn
