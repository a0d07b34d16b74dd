// Device and host helpers of the tensor-core kernel: PTX wrappers for mbarriers,
// bulk copies and tcgen05, bit -> e2m1 expansion.
#pragma once
#include <cuda_fp16.h>

#include <cstdint>
#include <cstdlib>

#include "snn_internal.h"

namespace snn {
namespace {

constexpr uint32_t WAIT_LIMIT = 1u << 20;  // try_wait attempts before a wait gives up

// ---------------------------------------------------------------- PTX helpers
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// try_wait with a suspend-time hint: the hardware parks the thread until the phase completes
// or about `ns` nanoseconds have passed, so a waiting thread issues almost no instructions
// and wakes as soon as the barrier flips.
__device__ __forceinline__ uint32_t mbar_try_hint(uint32_t bar, uint32_t parity, uint32_t ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity), "r"(ns)
      : "memory");
  return ok;
}
// non-blocking test of the phase: a wait that is already over costs one short instruction
__device__ __forceinline__ uint32_t mbar_test(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok;
}
// Bounded wait for the phase with the given parity; false when the limit ran out.  (Not unrolled: the roles share the
// instruction caches, and every wait of the kernel is a copy of this.)
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  if (mbar_test(bar, parity)) return true;
#pragma unroll 1
  for (uint32_t it = 0; it < WAIT_LIMIT; ++it)
    if (mbar_try_hint(bar, parity, 1000u)) return true;
  return false;
}
// Bounded wait for a thread whose wait is not on the critical path.  `ns` scales the time the
// hardware may keep the thread parked per attempt; the attempt limit bounds the whole wait
// (to a second or so) whatever the hardware makes of the hint.
__device__ __forceinline__ bool mbar_wait_backoff(uint32_t bar, uint32_t parity, uint32_t ns) {
#pragma unroll 1
  for (uint32_t it = 0; it < WAIT_LIMIT; ++it)
    if (mbar_try_hint(bar, parity, 20u * ns)) return true;
  return false;
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(bar)
               : "memory");
}
// One box of a four-dimensional tensor into shared memory; elements outside the tensor read as zeros.
__device__ __forceinline__ void tma_load_4d(uint32_t dst, const void* map, int c0, int c1, int c2, int c3, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cta.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4, %5}], [%6];" ::"r"(dst),
      "l"(map), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(bar)
      : "memory");
}
__device__ __forceinline__ void raise_status(int* status, int code) {
  *reinterpret_cast<volatile int*>(status) = code;
  __threadfence_system();
}
__device__ __forceinline__ void fence_proxy_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

// One lane of a fully active warp (the same one every time); the others get false.
__device__ __forceinline__ bool elect_one() {
  uint32_t elected;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(elected));
  return elected != 0;
}

// Barrier ID among THREADS of the CTA's threads, whole warps (which come together first: the barrier counts warps).
template <int ID, int THREADS>
__device__ __forceinline__ void bar_sync_some() {
  __syncwarp();
  asm volatile("bar.sync %0, %1;" ::"n"(ID), "n"(THREADS) : "memory");
}

// Programmatic dependent launch: a kernel launched with the serialization attribute may start
// while its predecessor in the stream still runs; grid_dep_wait() blocks until the predecessor has
// completed and its writes are visible (a no-op for an ordinary launch), grid_dep_launch() lets the
// successor start being scheduled.
__device__ __forceinline__ void grid_dep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// Shared-memory matrix descriptor, K-major, no swizzle: rows 16 B apart inside an
// 8-row group, groups `sbo` bytes apart, the two 16-byte K chunks `lbo` bytes apart.
__device__ __forceinline__ uint64_t make_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3ffffu) >> 4);
  d |= (uint64_t)((lbo >> 4) & 0x3fffu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3fffu) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version for this architecture
  return d;
}

// (MMAs: issued by the lanes for which `on` is not 0.)
// fp16 operands, fp32 accumulators: D[128 x N] (+)= A[128 x 16] * B[N x 16]^T
__device__ __forceinline__ void mma_ss_f16(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate, uint32_t on = 1u) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %5, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(on)
      : "memory");
}

// Block-scaled 4-bit MMA (e2m1 operands, one ue8m0 scale per 32 elements along K, fp32 accumulators):
// D[128 x N] (+)= A[128 x 64] * B[N x 64]^T.  +1, -1 and 0 are exact e2m1 values, unit scales leave the
// products alone and every partial sum of a 3x3 layer is an integer far below 2^24, so the fp32
// accumulators hold the exact sums.  sfa / sfb are tensor-memory addresses of the scale factors.
__device__ __forceinline__ void mma_ss_fp4(uint32_t d_tmem, uint64_t adesc, uint64_t bdesc, uint32_t idesc,
                                           uint32_t accumulate, uint32_t sfa, uint32_t sfb, uint32_t on = 1u) {
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %4, 0;\n\tsetp.ne.b32 q, %7, 0;\n\t"
      "@q tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%6], p;\n\t}" ::"r"(d_tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate), "r"(sfa), "r"(sfb), "r"(on)
      : "memory");
}
// One 32-bit value into 32 consecutive tensor-memory columns of this warp's 32 lanes.
__device__ __forceinline__ void tmem_fill32(uint32_t taddr, uint32_t v) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], {%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,"
      "%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1,%1};" ::"r"(taddr),
      "r"(v)
      : "memory");
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

// 32 columns of the warp's 32 lanes.  The load is asynchronous: its registers hold nothing a program may read, copy or
// carry around a loop before the wait.  The compiler does not know that, so load and wait are one statement.
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n\t"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}

// One column of the warp's 32 lanes.
__device__ __forceinline__ uint32_t tmem_ld1(uint32_t taddr) {
  uint32_t v;
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];\n\ttcgen05.wait::ld.sync.aligned;" : "=r"(v) : "r"(taddr) : "memory");
  return v;
}

// 16 bytes to shared memory at a 32-bit shared-space address
__device__ __forceinline__ void sts16(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
// 32 activation bits -> 32 e2m1 nibbles (16 bytes): +1.0 is 0x2, -1.0 is 0xA.  Channel 4n + k of the word sits in nibble
// n of word k, where its sign bit is one shift away: seven instructions (the order of the channels along K is free as
// long as the weights have the same; in natural order the bits have to be spread first, twenty instructions).
// sign = 0x88888888 and one = 0x22222222, or both 0 for a pixel that does not exist.  Bits of channels that do not
// exist may be anything: their weights are zero.
__device__ __forceinline__ uint4 expand_word_fp4(uint32_t bits, uint32_t sign, uint32_t one) {
  return make_uint4((~(bits << 3) & sign) | one, (~(bits << 2) & sign) | one, (~(bits << 1) & sign) | one, (~bits & sign) | one);
}

// 32 x 32 -> 64-bit product in one instruction (element offsets of pixels: both factors are non-negative 32-bit)
__device__ __forceinline__ size_t wide_mul(uint32_t a, uint32_t b) { return (size_t)a * (size_t)b; }

}  // namespace
}  // namespace snn
