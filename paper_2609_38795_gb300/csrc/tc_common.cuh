// Device primitives for the sm_103a kernels: mbarriers with bounded waits, TMA tile copies,
// and the 5th-generation tensor-core path (tcgen05.mma into tensor memory, tcgen05.ld out).
#pragma once

#include <cstdint>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#define ALR_DEV __device__ __forceinline__

namespace alr {

// Status word values written by kernels (mirrors ALR_ERR_TIMEOUT in the C header).
constexpr int kStatusTimeout = 4;

// A pipeline wait gives up after this much wall time (ns).  Legitimate waits in these
// kernels last microseconds; a wait this long means a producer will never arrive.
constexpr uint64_t kWaitLimitNs = 1500ull * 1000ull * 1000ull;

constexpr float kLog2e = 1.4426950408889634f;
constexpr float kLn2 = 0.6931471805599453f;

ALR_DEV uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

ALR_DEV uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// 2^x on the special-function unit (PTX ex2.approx; flushes denormal results to zero).
ALR_DEV float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// The exponent every column gets relative to the reference m is fma(z, log2 e, b(m)) with
// b(m) = -m log2 e rounded, which at z = m is not 0 but the rounding residual of m log2 e (exactly
// representable, up to ~4e-6 at |m| ~ 40): every exponential summed against m carries the factor
// 2^r.  It cancels between a row's sums and is taken off where log S stands alone, so that the
// log-probabilities keep their precision.
ALR_DEV float exp_residual(float m) { return fmaf(m, kLog2e, -m * kLog2e); }

// Exponent of the step from the reference m to one with b = b(nm), nm >= m: the difference of the
// rounded offsets, so that sums that carry m's factor 2^r carry nm's after it (multiplied by
// exp(m - nm) instead, the terms met before each new maximum keep another factor than the rest:
// 1e-6 at |m| ~ 30).
ALR_DEV float ref_step(float m, float b) { return __fadd_rn(b, __fmul_rn(m, kLog2e)); }

// ------------------------------------------------------ paired fp32 arithmetic ---
// Two fp32 lanes in one 64-bit register, combined by the sm_100-family packed instructions:
// each lane is computed exactly as the scalar instruction would, in one issue slot for both.
ALR_DEV uint64_t f2_pack(float a, float b) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
ALR_DEV void f2_unpack(uint64_t v, float& a, float& b) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v));
}
ALR_DEV uint64_t f2_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
ALR_DEV uint64_t f2_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
ALR_DEV uint64_t f2_sub(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
ALR_DEV uint64_t f2_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
// 2^a and 2^b of a packed pair (two special-function operations).
ALR_DEV uint64_t f2_ex2(uint64_t v) {
  float a, b;
  f2_unpack(v, a, b);
  return f2_pack(ex2(a), ex2(b));
}
// Three-input maximum (one instruction); no NaN inputs occur where it is used.
ALR_DEV float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// Programmatic dependent launch (launch.h): every thread calls pdl_wait before its first global
// access.  Kernels read what an earlier one wrote through plain pointers and loads: the read-only
// path (__ldg, and what the compiler makes of const __restrict__) is for data that no one writes
// during the kernel's whole lifetime, which begins before the wait, so the wait does not order it.
// pdl_release lets the next kernel be scheduled once some thread of every block has called it (or
// the block has ended).  The tensor-core kernels call it when their work is done: blocks of the
// next kernel that sit on the SMs for the whole of a long kernel, waiting, cost power (the text8b
// step 106.4 -> 109.1 ms with the call at their start).
ALR_DEV void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
ALR_DEV void pdl_release() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
ALR_DEV void pdl_wait_and_release() {
  pdl_wait();
  pdl_release();
}

// ---------------------------------------------------------------- mbarrier ---
ALR_DEV void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}

ALR_DEV void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

ALR_DEV void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

ALR_DEV void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

// One bounded probe of the phase with the given parity.  A thread whose phase is not yet
// complete is suspended in hardware until the phase completes or at most kSuspendHintNs
// elapses.  In practice it wakes far more often (a waiting thread of the loss kernel probes
// every few tens of cycles while the CTA's barriers are busy), so kernels keep the number of
// waiting warps small: one warp waits and the others sleep in a named barrier.
constexpr uint32_t kSuspendHintNs = 20000;

ALR_DEV bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t done;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(done)
      : "r"(smem_u32(bar)), "r"(parity), "r"(kSuspendHintNs)
      : "memory");
  return done != 0;
}

// Per-CTA abort word shared by all roles: once any wait times out, every other wait of the
// CTA returns promptly instead of running into its own limit.
struct AbortFlag {
  volatile int* smem;
  int* status;   // per-device status word in global memory
};

// A suspended waiter wakes every few tens of cycles while the CTA's barriers are busy; the
// clock and the abort word are checked only on every kWaitCheckEvery-th wake-up, so a wake-up
// costs a handful of instructions.
constexpr uint32_t kWaitCheckEvery = 16;

// Wait until the phase with the given parity has completed.  Returns false (after recording
// the timeout) if the limit elapses or another role of the CTA already gave up.
ALR_DEV bool mbar_wait(uint64_t* bar, uint32_t parity, const AbortFlag& ab) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t i = 1;; ++i) {
    if (mbar_try_wait(bar, parity)) return true;
    if (i % kWaitCheckEvery == 0) {
      if (*ab.smem) return false;
      if (global_timer_ns() - t0 > kWaitLimitNs) {
        *ab.smem = 1;
        atomicExch(ab.status, kStatusTimeout);
        return false;
      }
    }
  }
}

// Drain wait used while shutting down after an abort: bounded, records nothing.
ALR_DEV void mbar_wait_drain(uint64_t* bar, uint32_t parity) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > kWaitLimitNs) return;
  }
}

// ------------------------------------------------------------------- TMA ---
ALR_DEV void tma_prefetch_desc(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

ALR_DEV void tma_load_2d(void* smem_dst, const CUtensorMap* map, uint64_t* bar, int x, int y) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(smem_dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y)
      : "memory");
}

ALR_DEV void tma_store_2d(const CUtensorMap* map, const void* smem_src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(smem_u32(smem_src)), "r"(x), "r"(y)
               : "memory");
}

ALR_DEV void tma_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
ALR_DEV void tma_store_wait_read_all() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}
ALR_DEV void tma_store_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
// Wait until at most the most recent bulk store group is still reading shared memory.
ALR_DEV void tma_store_wait_read_le1() {
  asm volatile("cp.async.bulk.wait_group.read 1;" ::: "memory");
}

// Make generic-proxy shared-memory writes visible to the async proxy (TMA store reads).
ALR_DEV void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

ALR_DEV void named_bar_sync(int id, int nthreads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}

// ---------------------------------------------------------------- tcgen05 ---
ALR_DEV void tmem_alloc(uint32_t* smem_result, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(smem_result)),
               "r"(ncols)
               : "memory");
}
ALR_DEV void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
ALR_DEV void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols)
               : "memory");
}
ALR_DEV void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
ALR_DEV void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }

// Shared-memory matrix descriptor for a 128-byte-swizzled operand tile.
//   bits  0-13 start address >> 4      bits 16-29 leading-dimension byte offset >> 4
//   bits 32-45 stride-dimension byte offset >> 4   bits 46-48 fixed 0b001
//   bits 61-63 swizzle mode (2 = 128-byte swizzle)
// K-major tiles: rows of 128 bytes along K, 8-row atoms 1024 bytes apart (SBO); LBO unused.
// MN-major tiles: rows of 128 bytes along MN (one row per k), 8-k atoms 1024 bytes apart
// (SBO), consecutive 128-byte MN chunks `lbo` bytes apart (LBO).
ALR_DEV uint64_t sdesc_sw128(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4) |
         (static_cast<uint64_t>((lbo & 0x3FFFFu) >> 4) << 16) |
         (static_cast<uint64_t>((sbo & 0x3FFFFu) >> 4) << 32) | (1ull << 46) | (2ull << 61);
}

// Instruction descriptor for kind::f16 (bf16 inputs) or kind::tf32, fp32 accumulation.
//   bits 4-5 D type (1 = f32); 7-9 A type, 10-12 B type (1 = bf16, 2 = tf32);
//   bit 15 A MN-major; bit 16 B MN-major; bits 17-22 N >> 3; bits 24-28 M >> 4.
__host__ __device__ constexpr uint32_t idesc_make(bool tf32, int M, int N, bool a_mn, bool b_mn) {
  return (1u << 4) | ((tf32 ? 2u : 1u) << 7) | ((tf32 ? 2u : 1u) << 10) |
         ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         (static_cast<uint32_t>(N >> 3) << 17) | (static_cast<uint32_t>(M >> 4) << 24);
}

template <bool kTf32>
ALR_DEV void mma_issue(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                       uint32_t accumulate) {
  if constexpr (kTf32) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  } else {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(tmem_d),
        "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
        : "memory");
  }
}

// Arrive on `bar` once every tcgen05 operation this thread issued so far has completed.
ALR_DEV void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// Load 32 consecutive 32-bit columns of this warp's 32 TMEM lanes (one lane per thread).
// The registers are valid only after tmem_ld_wait(); pass them through reg_fence() after the
// wait so that no use can be scheduled above it.
ALR_DEV void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
      "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
}

template <int n>
ALR_DEV void reg_fence(uint32_t (&r)[n]) {
#pragma unroll
  for (int i = 0; i < n; ++i) asm volatile("" : "+r"(r[i]));
}

ALR_DEV void tmem_ld_wait() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

ALR_DEV bool elect_one_lane() { return (threadIdx.x & 31u) == 0; }

// ------------------------------------------------------------------ cluster coordinates ---
// (Constant for a kernel's lifetime: their reads are not volatile, so the compiler may re-read
// them instead of holding them in registers.)  The kernel forms that share operand tiles across
// the CTAs of a cluster, and their PTX, are built into a library of their own from
// csrc_cluster/; these sources only name the coordinates and the cluster barrier.
ALR_DEV uint32_t cluster_ctarank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}

ALR_DEV uint32_t cluster_id_x() {
  uint32_t r;
  asm("mov.u32 %0, %%clusterid.x;" : "=r"(r));
  return r;
}

ALR_DEV uint32_t n_clusters_x() {
  uint32_t r;
  asm("mov.u32 %0, %%nclusterid.x;" : "=r"(r));
  return r;
}

ALR_DEV uint32_t cluster_nctarank() {
  uint32_t r;
  asm("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}

// Shared::cluster address of the object at the same offset as `p` in CTA `rank`'s shared memory.
ALR_DEV uint32_t cluster_smem_addr(const void* p, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(smem_u32(p)), "r"(rank));
  return r;
}

ALR_DEV int ld_cluster_s32(uint32_t cluster_addr) {
  int v;
  asm volatile("ld.shared::cluster.s32 %0, [%1];" : "=r"(v) : "r"(cluster_addr) : "memory");
  return v;
}

ALR_DEV float4 ld_cluster_v4(uint32_t cluster_addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(cluster_addr)
               : "memory");
  return v;
}

// All threads of every CTA of the cluster: arrive (release) and wait (acquire).
ALR_DEV void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" :::
                   "memory");
}

// The form of a kernel that runs without clusters: no CTA shares its operand tiles.
struct NoCluster {
  static constexpr int kCtas = 1;
};

// The form of the plain GEMM whose clusters split the contraction of one tile: the CTAs share no
// operand tile, only their partial sums, through distributed shared memory.
struct SplitCluster {
  static constexpr int kCtas = 1;
};

ALR_DEV uint8_t* align_1024(uint8_t* p) {
  return reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(p) + 1023) & ~uintptr_t(1023));
}

}  // namespace alr
