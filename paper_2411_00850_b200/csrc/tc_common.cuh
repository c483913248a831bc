// Device and host helpers shared by the kernels that use the 5th-generation tensor cores: mbarriers with bounded
// waits, plain (non-multicast) TMA tile loads, shared-memory matrix descriptors, tcgen05 commit / load wrappers and
// the driver entry point that encodes tensor maps.  Internal; every function has internal linkage.
#pragma once

#include <cuda.h>

#include "common.cuh"

namespace gwq_tc {

constexpr long long kSpinCycles = GWQ_DEFAULT_WAIT_CYCLES;   // about half a second of SM clock

static __device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }

static __device__ __forceinline__ void mbar_init(unsigned bar, unsigned count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count));
}
static __device__ __forceinline__ void mbar_arrive(unsigned bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}
static __device__ __forceinline__ void mbar_expect_tx(unsigned bar, unsigned bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
// Bounded wait for the phase with the given parity: gives up (false) after `limit` cycles, or as
// soon as another role of the CTA has given up.  A first, non-blocking test decides the common case and
// makes a limit of zero mean exactly "give up unless the phase has completed already".
static __device__ __forceinline__ bool mbar_wait(unsigned bar, unsigned parity, volatile int* abort_flag, long long limit) {
  unsigned done;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
      : "=r"(done)
      : "r"(bar), "r"(parity)
      : "memory");
  if (done) return true;
  if (limit <= 0) return false;
  const long long t0 = clock64();
  // Sixteen tests to a round, four instructions each: warps that wait share the issue slots with those that work (70B block at 16
  // tokens 257.2 -> 253.7 us against a loop in C; suspending the thread for up to 2 us per test instead, 28672 x 8192 at 8 tokens 64 -> 86:
  // it does not wake at once).
  for (;;) {
    asm volatile(
        "{\n .reg .pred p, q;\n .reg .u32 n;\n mov.u32 n, 16;\n"
        "AGAIN:\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n @p bra DONE;\n"
        " sub.u32 n, n, 1;\n setp.ne.u32 q, n, 0;\n @q bra AGAIN;\n"
        "DONE:\n selp.b32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
    if (*abort_flag || clock64() - t0 > limit) return false;
  }
}

// The same wait made by all 32 lanes of a converged warp, with one verdict for the whole warp (a lane that gave up
// alone would leave the others at the next warp-level synchronisation).
static __device__ __forceinline__ bool mbar_wait_warp(unsigned bar, unsigned parity, volatile int* abort_flag, long long limit) {
  return __all_sync(0xFFFFFFFFu, mbar_wait(bar, parity, abort_flag, limit));
}

// True while no kernel has given up on the layer (later calls then do no work until the host has read the status).  Other
// CTAs write the word while this one starts, so that two reads may differ.  Threads that meet at a warp-level operation or
// at a barrier without a limit have to go by ONE read: of one lane, handed round the warp, or of one thread before a barrier of
// all that share the verdict, handed round through shared memory.  (Warps that each looked for themselves could start
// differently, and one that skips its loop never comes to a named barrier inside it.)
static __device__ __forceinline__ bool no_one_gave_up(const int32_t* status) {
  return *reinterpret_cast<const volatile int32_t*>(status) == 0;
}

static __device__ __forceinline__ void tma_load_2d(unsigned dst, const CUtensorMap* map, int c0, int c1, unsigned bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
      ::"r"(dst), "l"(map), "r"(c0), "r"(c1), "r"(bar)
      : "memory");
}

// Shared-memory matrix descriptor, K-major, 128-byte swizzle: rows of 128 bytes, 8-row atoms
// 1024 bytes apart (tile base 1024-byte aligned).
static __device__ __forceinline__ uint64_t umma_desc(unsigned smem_addr) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr >> 4) & 0x3FFFu);   // start address, 16-byte units
  d |= (uint64_t)1 << 16;                        // leading byte offset (not used by swizzled K-major)
  d |= (uint64_t)(1024 >> 4) << 32;              // stride byte offset: next 8-row atom
  d |= (uint64_t)1 << 46;                        // descriptor version of this architecture
  d |= (uint64_t)2 << 61;                        // layout type: 128-byte swizzle
  return d;
}

// True in one lane of a converged warp.  MMAs are issued by that lane inside code that the whole warp runs, so that their
// descriptors stay in uniform registers: from a branch that one thread takes, an MMA of up to 96 columns costs its issuer 54 cycles
// and a chain of four 490; this way 16 at 32 columns with A in tensor memory, 40 with A in shared memory.  The lane is the same one
// every time (the election is deterministic for a mask) but need not be lane 0, and a tcgen05.commit tracks the MMAs of its own
// thread alone: a kernel that issues by election also commits by election, on the give-up path too.
static __device__ __forceinline__ bool elect_one() {
  unsigned elected;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xFFFFFFFF;\n selp.b32 %0, 1, 0, p;\n}\n" : "=r"(elected));
  return elected != 0;
}

static __device__ __forceinline__ void umma_f16(unsigned tmem_d, uint64_t da, uint64_t db, unsigned idesc, unsigned accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
      ::"r"(tmem_d), "l"(da), "l"(db), "r"(idesc), "r"(accumulate)
      : "memory");
}
static __device__ __forceinline__ void umma_commit(unsigned bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar) : "memory");
}

static __device__ __forceinline__ void tmem_ld32(unsigned taddr, unsigned (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,"
      "%29,%30,%31}, [%32];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr)
      : "memory");
}


typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static inline EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* ptr = nullptr;
    cudaDriverEntryPointQueryResult qres;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &ptr, cudaEnableDefault, &qres) == cudaSuccess &&
        qres == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(ptr);
  }
  return fn;
}


}  // namespace gwq_tc
