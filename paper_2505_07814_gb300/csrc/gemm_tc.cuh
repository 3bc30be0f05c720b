// gemm_tc.cuh -- what the 5th-generation tensor-core kernels (gemm_ws.cuh, dftgemm.cuh) share: descriptors of
// shared-memory operands and instructions, bounded mbarrier waits, tensor-memory loads.
//
// Operands lie in shared memory in the tensor core's canonical K-major layout without swizzle: 8-row x 16-byte core
// matrices, LBO = 128 B between core matrices along K, SBO = 1024 B between 8-row groups.  The tensor core's own
// accumulation drifts over long K, so the kernels sum every 64 of K into a fresh TMEM region and add it to FP32
// registers with round-to-nearest adds.
#pragma once
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <type_traits>

#include "pty.h"

namespace pty {

constexpr int TC_BM = 128;
constexpr int TC_LBO = 128, TC_SBO = 1024;
constexpr long TC_SPIN = PTY_WAIT_POLLS_DEFAULT;  // non-blocking mbarrier polls before a wait gives up (well under a second)

__device__ __forceinline__ uint32_t tc_smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor: start address, LBO, SBO (all >> 4), descriptor version 1,
// no swizzle.
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr) {
  return (uint64_t)((addr >> 4) & 0x3FFF) | ((uint64_t)(TC_LBO >> 4) << 16) | ((uint64_t)(TC_SBO >> 4) << 32) |
         ((uint64_t)1 << 46);
}
// Instruction descriptor of kind::f16: FP32 accumulator, A and B of type H (bf16 or fp16), both
// K-major, M = 128, N = BN.
template <class H, int BN>
__host__ __device__ constexpr uint32_t tc_idesc() {
  constexpr uint32_t ab = std::is_same<H, __nv_bfloat16>::value ? 1u : 0u;
  return (1u << 4) | (ab << 7) | (ab << 10) | ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
}

__device__ __forceinline__ bool tc_try_wait(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n.reg .pred p;\nmbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.b32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// Bounded wait of at most `limit` polls; false on timeout.
__device__ __forceinline__ bool tc_wait(uint32_t bar, uint32_t parity, long limit = TC_SPIN) {
  for (long i = 0; i < limit; ++i)
    if (tc_try_wait(bar, parity)) return true;
  return false;
}
// Poll limit of the pipeline's waits (the final drain before TMEM is released always takes
// TC_SPIN); pty_set_wait_limit changes it for tests that make a wait run out.
long stage_wait_limit();

// Completes this warp's tensor-memory loads into r.  The loads are asynchronous and only their own asm statements name r,
// so without the statements after the wait a use of r could be placed before it.
template <int N>
__device__ __forceinline__ void tc_ld_wait(uint32_t (&r)[N]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int j = 0; j < N; ++j) asm volatile("" : "+r"(r[j]));
}
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,"
      "%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]),
        "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  tc_ld_wait(r);
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

}  // namespace pty
