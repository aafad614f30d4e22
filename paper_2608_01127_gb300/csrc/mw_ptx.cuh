// Inline-PTX building blocks for sm_103a: mbarriers, TMA (cp.async.bulk),
// tcgen05 MMA / TMEM data movement, and the shared-memory / instruction
// descriptors the tcgen05 MMAs consume.  Written from the public PTX ISA.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <stdint.h>

namespace mw {

// Bits of the device status word: a bounded wait gave up / the dynamic
// shared memory was not 1024-byte aligned (the kernel then does nothing).
constexpr unsigned kDevTimeout = 1u;
constexpr unsigned kDevMisaligned = 2u;

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ uint64_t global_timer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}

// ------------------------------------------------------------------ mbarrier

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count));
}

__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Shared abort state of one CTA: a flag that every bounded wait polls, so
// that one expired wait releases all roles, plus the time budget.
struct WaitCtl {
  volatile int* abort;     // shared memory
  unsigned* status;        // device status word (global)
  uint64_t budget_ns;      // per wait
};

// Waits for the phase with the given parity; gives up after the budget (or
// when another role of the CTA already gave up), records the timeout in the
// status word and returns false.  Never traps.  The abort flag and the clock
// are looked at only every 32nd poll (try_wait itself suspends the thread for
// a while): a read of the clock before the first one delayed every wait.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, const WaitCtl& ctl) {
  uint64_t t0 = 0;
  for (uint32_t spins = 1; !mbar_try_wait(bar, parity); ++spins) {
    if ((spins & 31u) != 0u) continue;
    if (*ctl.abort) return false;
    const uint64_t t = global_timer_ns();
    if (t0 == 0) t0 = t;
    if (t - t0 > ctl.budget_ns) {
      *ctl.abort = 1;
      atomicOr(ctl.status, kDevTimeout);
      return false;
    }
  }
  return true;
}

// The same for a whole converged warp: every lane gets the same answer, so
// that .sync.aligned tcgen05 instructions after it are never divergent.  The
// loop itself is uniform (a vote a poll): a vote over mbar_wait's answers
// took 104 cycles for a phase that was complete already, this form 59.
__device__ __forceinline__ bool warp_wait(uint64_t* bar, uint32_t parity, const WaitCtl& ctl) {
  uint64_t t0 = 0;
  for (uint32_t spins = 1; !__all_sync(0xffffffffu, mbar_try_wait(bar, parity)); ++spins) {
    if ((spins & 31u) != 0u) continue;
    const uint64_t t = global_timer_ns();
    if (t0 == 0) t0 = t;
    const bool late = t - t0 > ctl.budget_ns;
    if (__any_sync(0xffffffffu, late || *ctl.abort)) {
      if (late) {
        *ctl.abort = 1;
        atomicOr(ctl.status, kDevTimeout);
      }
      return false;
    }
  }
  return true;
}

// Bounded wait used only on the abort path (lets in-flight copies land
// before the CTA exits): ignores the abort flag.
__device__ __forceinline__ void drain_wait(uint64_t* bar, uint32_t parity, uint64_t budget_ns) {
  const uint64_t t0 = global_timer_ns();
  while (!mbar_try_wait(bar, parity)) {
    if (global_timer_ns() - t0 > budget_ns) return;
  }
}

// ------------------------------------------------------------------ TMA

__device__ __forceinline__ void prefetch_tmap(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

// 3-D tiled load into shared memory, completion signalled as transaction
// bytes on `bar`.  c0 is the innermost (element) coordinate: callers keep
// c0 * 2 bytes a multiple of 16.
__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar,
                                            int c0, int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// 3-D tiled reduce-add of a shared-memory box into global memory (element
// type and box from the map; here f32), tracked as a bulk async-group of the
// issuing thread.  Coordinates must not be negative; c0 * element size must be
// a multiple of 16 bytes.
__device__ __forceinline__ void tma_reduce_add_3d(const CUtensorMap* map, const void* src, int c0,
                                                  int c1, int c2) {
  asm volatile(
      "cp.reduce.async.bulk.tensor.3d.global.shared::cta.add.tile.bulk_group"
      " [%0, {%2, %3, %4}], [%1];" ::"l"(reinterpret_cast<uint64_t>(map)),
      "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// 3-D tiled store of a shared-memory box into global memory (element type,
// box and swizzle from the map), tracked as a bulk async-group of the
// issuing thread.  Rows past the map's extents are not written;
// coordinates must not be negative; c0 * element size must be a multiple of
// 16 bytes.
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int c0,
                                             int c1, int c2) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group"
      " [%0, {%2, %3, %4}], [%1];" ::"l"(reinterpret_cast<uint64_t>(map)),
      "r"(smem_u32(src)), "r"(c0), "r"(c1), "r"(c2)
      : "memory");
}

// Barrier ID (1..15) over THREADS threads (a multiple of 32) of the CTA.
template <int ID, int THREADS>
__device__ __forceinline__ void named_barrier_sync() {
  static_assert(ID >= 1 && ID <= 15 && THREADS % 32 == 0, "named barrier");
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}

__device__ __forceinline__ void bulk_commit_group() {
  asm volatile("cp.async.bulk.commit_group;" ::: "memory");
}

// Waits until all but the issuing thread's N newest bulk groups have finished
// reading shared memory (their sources may be overwritten afterwards).
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(N) : "memory");
}

// Waits until the issuing thread's committed bulk groups have completed.
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
}

// Contiguous global -> shared copy; both addresses 16-byte aligned, size a
// multiple of 16.
__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes,
                                          uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::
          "r"(smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void fence_proxy_async_smem() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

// ------------------------------------------------------------------ tcgen05

__device__ __forceinline__ void tmem_alloc(uint32_t* dst_smem, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                   smem_u32(dst_smem)),
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

// The MMA helpers below are warp-collective: all 32 lanes of the issuing
// warp call them converged, and one lane chosen by elect.sync issues the
// instruction.  Keeping the issuing warp's control flow uniform lets the
// compiler hold descriptors in uniform registers; a single divergent lane
// issuing measured ~40% slower per MMA because the tensor core's queue is
// only about two instructions deep.  elect.sync picks the same (lowest) lane
// every time, so tcgen05.commit tracks the MMAs that lane issued.

// The high word shared by all 128-byte-swizzle operand descriptors (see
// sdesc_sw128): stride byte offset 1024, version 1, swizzle mode 2.
constexpr uint32_t kSw128Hi = (1024u >> 4) | (1u << 14) | (2u << 29);

// D(tmem) (+)= A(smem) * B(smem)^T, kind::f16 (bf16 in, f32 acc); operands
// given by the low words of their sdesc_sw128 descriptors (the issuing warps
// hold many of them: one register each instead of two).
__device__ __forceinline__ void umma_ss(uint32_t d_tmem, uint32_t a_desc, uint32_t b_desc,
                                        uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t.reg .b64 a, b;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "mov.b64 a, {%1, %5};\n\t"
      "mov.b64 b, {%2, %5};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(a_desc), "r"(b_desc), "r"(idesc), "r"(accumulate), "n"(kSw128Hi)
      : "memory");
}

// D (+)= A B^T with tf32 operands (kind::tf32, K = 8 per instruction).
__device__ __forceinline__ void umma_ss_tf32(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc,
                                             uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

// umma_ss with A read from tensor memory.
__device__ __forceinline__ void umma_ts(uint32_t d_tmem, uint32_t a_tmem, uint32_t b_desc,
                                        uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p, e;\n\t.reg .b64 b;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "mov.b64 b, {%2, %5};\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "@e tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(a_tmem), "r"(b_desc), "r"(idesc), "r"(accumulate), "n"(kSw128Hi)
      : "memory");
}

// Arrive (once) on `bar` when every tcgen05 op issued so far by the elected
// lane has completed.
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "{\n\t.reg .pred e;\n\t"
      "elect.sync _|e, 0xffffffff;\n\t"
      "@e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n\t}\n" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_wait_ld() {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 consecutive 32-bit columns of this thread's lane (shape 32x32b).
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
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

__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(
          taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
      "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]),
      "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

// 16 consecutive 32-bit columns of this thread's lane (shape 32x32b).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
      "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15])
      : "memory");
}

// Per-warpgroup register re-split (all warps of a warpgroup execute it).
template <int N>
__device__ __forceinline__ void regs_dec() {
  asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(N));
}
template <int N>
__device__ __forceinline__ void regs_inc() {
  asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(N));
}

// ------------------------------------------------------------------ descriptors
//
// Shared-memory matrix descriptor (tcgen05 form): start address >> 4 in bits
// 0-13, leading-dimension byte offset >> 4 in 16-29, stride-dimension byte
// offset >> 4 in 32-45, the fixed version value 1 in bits 46-47, base offset
// 0 (every swizzle atom here is 1024-byte aligned), swizzle mode in 61-63
// (2 = 128-byte swizzle).
//
// All operand tiles here use the 128-byte swizzle that TMA writes: a tile is
// a set of "regions" of 64 bf16 columns; inside a region row r sits at byte
// r*128 and its 16-byte chunk c is stored at chunk (c ^ (r & 7)).
//   K-major operand (the contraction index runs along a region row):
//     SBO = 1024 (next group of 8 rows); LBO unused.  The k-th 16-wide K step
//     starts 32*k bytes into the region (the hardware applies the XOR).
//   MN-major operand (the contraction index runs down the rows):
//     LBO = byte distance between regions (next 64 MN columns),
//     SBO = 1024 (next group of 8 contraction rows); a 16-deep K step
//     advances 16 rows = 2048 bytes.
// The low word; the high word is kSw128Hi for every operand here (SBO 1024).
__device__ __forceinline__ uint32_t sdesc_sw128(uint32_t saddr, uint32_t lbo_bytes) {
  return ((saddr & 0x3FFFFu) >> 4) | (((lbo_bytes >> 4) & 0x3FFFu) << 16);
}

// The same descriptor for a start address `bytes` further on (a multiple of
// 16): only the 14-bit address field changes, and it cannot carry for the
// in-range shared-memory addresses used here.
__device__ __forceinline__ uint32_t sdesc_add(uint32_t desc, uint32_t bytes) {
  return desc + (bytes >> 4);
}
__device__ __forceinline__ uint64_t sdesc_add(uint64_t desc, uint32_t bytes) {
  return desc + static_cast<uint64_t>(bytes >> 4);
}

// The same descriptor with the 32-byte swizzle (mode 6) that a TMA copy with
// CU_TENSOR_MAP_SWIZZLE_32B writes: rows of 32 bytes (8 tf32), 8-row atoms of
// 256 bytes, 16-byte chunk c of row r at chunk c ^ ((r >> 2) & 1).  K-major
// operand with K = 8 tf32: SBO = 256 (next 8 rows); LBO unused.
__device__ __forceinline__ uint64_t sdesc_sw32(uint32_t saddr, uint32_t sbo_bytes) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);
  d |= static_cast<uint64_t>(1) << 16;  // LBO 16 bytes, as the K-major 128-byte form passes
  d |= static_cast<uint64_t>((sbo_bytes >> 4) & 0x3FFFu) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  d |= static_cast<uint64_t>(6) << 61;
  return d;
}

// Instruction descriptor for kind::tf32 with f32 accumulation, A and B
// K-major: D format f32 (bits 4-5 = 1), A and B format tf32 (= 2).
__host__ __device__ constexpr uint32_t idesc_tf32_f32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

// Instruction descriptor for kind::f16 with bf16 A/B and f32 accumulation:
// D format (bits 4-5) = 1 (f32), A format (7-9) = 1 (bf16), B format (10-12)
// = 1 (bf16), A major (15) and B major (16): 0 = K-major, 1 = MN-major,
// N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__host__ __device__ constexpr uint32_t idesc_bf16_f32(int M, int N, bool a_mn_major,
                                                      bool b_mn_major) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn_major ? 1u : 0u) << 15) |
         ((b_mn_major ? 1u : 0u) << 16) | (static_cast<uint32_t>(N >> 3) << 17) |
         (static_cast<uint32_t>(M >> 4) << 24);
}

// ------------------------------------------------------------------ math

__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}

__device__ __forceinline__ float ex2_approx(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Programmatic dependent launch: a kernel launched with programmatic
// stream serialization may start while the previous kernel in the stream
// finishes; pdl_wait blocks until that kernel has completed and its memory
// is visible (a no-op for a kernel launched without the attribute), and
// pdl_trigger lets the next such kernel be scheduled early.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// Packed fp32 pair arithmetic (one instruction for two lanes of work).
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;"
      : "=l"(d)
      : "l"(*reinterpret_cast<uint64_t*>(&a)), "l"(*reinterpret_cast<uint64_t*>(&b)),
        "l"(*reinterpret_cast<uint64_t*>(&c)));
  return *reinterpret_cast<float2*>(&d);
}

__device__ __forceinline__ float2 add2(float2 a, float2 b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;"
      : "=l"(d)
      : "l"(*reinterpret_cast<uint64_t*>(&a)), "l"(*reinterpret_cast<uint64_t*>(&b)));
  return *reinterpret_cast<float2*>(&d);
}

__device__ __forceinline__ float2 mul2(float2 a, float2 b) {
  uint64_t d;
  asm("mul.rn.f32x2 %0, %1, %2;"
      : "=l"(d)
      : "l"(*reinterpret_cast<uint64_t*>(&a)), "l"(*reinterpret_cast<uint64_t*>(&b)));
  return *reinterpret_cast<float2*>(&d);
}

// 32 bytes to global memory as one store (p 32-byte aligned): whole sectors
// where every lane writes a row of its own.
__device__ __forceinline__ void store_32b(void* p, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// 32 consecutive values of an output row as bf16 to p (16-byte aligned): the
// first n16 of its four 16-byte pieces.  wide: p is 32-byte aligned, and whole
// sectors go out as one store each; 16-byte stores, every lane in a row of its
// own, fill half a sector and take the SM's path to L2 twice as long (forward
// of 20 heads x 1505 rows of 128: 25.0 -> 24.5 us; backward of 24 heads x 14080
// rows of 64: 1251 -> 1243 us).
__device__ __forceinline__ void store_row32(__nv_bfloat16* p, const float (&v)[32], int n16,
                                            bool wide) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t w[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = pack_bf16x2(v[16 * h + 2 * k], v[16 * h + 2 * k + 1]);
    uint4* dst = reinterpret_cast<uint4*>(p) + 2 * h;
    if (wide && 2 * h + 2 <= n16) {
      store_32b(dst, w);
    } else {
      if (2 * h < n16) dst[0] = make_uint4(w[0], w[1], w[2], w[3]);
      if (2 * h + 1 < n16) dst[1] = make_uint4(w[4], w[5], w[6], w[7]);
    }
  }
}

// Temporal RoPE (a channel pair turned by an angle): the (cos, sin) of
// f * omega for an integer frame 0 <= f <= 2^24 and omega = om_hi + om_lo.
// The angle is reduced to about [-pi, pi] before the fast sine and cosine:
// the FMA yields the exact rounding error of f * om_hi (Dekker's product),
// and 2 pi is subtracted in two parts (Cody and Waite), the first of which
// cancels exactly, so the reduced angle stays within ~1e-6 rad however
// large f * omega is.
__device__ __forceinline__ float2 rope_cos_sin(int f, float om_hi, float om_lo) {
  const float two_pi_hi = 6.28318548202514648f;    // 2 pi rounded to float
  const float two_pi_lo = -1.74845553146951e-07f;  // 2 pi - two_pi_hi
  const float ff = static_cast<float>(f);           // exact up to 2^24
  const float th = ff * om_hi;
  const float err = fmaf(ff, om_hi, -th);           // f * om_hi - th, exactly
  const float k = rintf(th * 0.15915494309189535f);
  float r = fmaf(-k, two_pi_hi, th);
  r = fmaf(-k, two_pi_lo, r);
  r += fmaf(ff, om_lo, err);
  float sn, cs;
  __sincosf(r, &sn, &cs);
  return make_float2(cs, sn);
}

// The bf16 pair (x0, x1) in one 32-bit word (x0 in the low half) turned by
// the angle whose (cos, sin) is csn: (x0 c - x1 s, x0 s + x1 c), rounded to
// bf16 (two packed operations).
__device__ __forceinline__ uint32_t rope_turn(uint32_t w, float2 csn) {
  const float x0 = __uint_as_float(w << 16), x1 = __uint_as_float(w & 0xffff0000u);
  const float2 y = fma2(make_float2(-x1, x1), make_float2(csn.y, csn.x), mul2(make_float2(x0, x0), csn));
  return pack_bf16x2(y.x, y.y);
}

}  // namespace mw
