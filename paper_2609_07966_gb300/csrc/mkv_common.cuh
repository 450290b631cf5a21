// Shared device helpers of libmkv (sm_103a).  Inline PTX wrappers for the
// staging copies (cp.async), shared-memory matrix loads (ldmatrix) and the
// fp16 x fp16 -> fp32 tensor-core tile product used by the decode kernels.
#pragma once

#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "mkv.h"

namespace mkv {

constexpr int kNumSMs = 152;          // GB300: 2 dies x 76 SMs
constexpr float kLog2e = 1.4426950408889634f;

__host__ __device__ __forceinline__ int64_t ceil_div_dev(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Programmatic dependent launch: the FP16-family kernels of a decode step (append, FP16 / H2O /
// page-list decode, H2O update) are launched with the programmatic stream-serialization attribute,
// so a kernel may be scheduled while its predecessor in the stream is still running.  It waits here
// for that grid's completion and memory before its first global access, then lets its own
// successor be scheduled (which waits the same way); a successor can only be scheduled once every
// CTA of this grid has passed this point, so it never holds resources a CTA of this grid is waiting
// for.  The two launches of mkv_kvquant_step have the attribute as well and place the two
// instructions themselves: the quantization waits first and then lets the decode start, which reads
// tables and the query (finished before the quantization was allowed to run) and waits before it touches
// the cache; near its end the decode lets the next step's quantization be scheduled.  The KVQuant calls one by
// one and the fused RocketKV step launch plainly: there the attribute measured slower.
__device__ __forceinline__ void pdl_wait_and_trigger() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte global->shared copy; `src_bytes` = 0 writes zeros (a masked row).
__device__ __forceinline__ void cp_async16(void* smem, const void* gmem, int src_bytes = 16) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_addr(smem)), "l"(gmem),
               "r"(src_bytes));
}
__device__ __forceinline__ void cp_async8(void* smem, const void* gmem, int src_bytes = 8) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;\n" ::"r"(smem_addr(smem)), "l"(gmem),
               "r"(src_bytes));
}
__device__ __forceinline__ void cp_async4(void* smem, const void* gmem, int src_bytes = 4) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;\n" ::"r"(smem_addr(smem)), "l"(gmem),
               "r"(src_bytes));
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_async_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

// Four 8x8 b16 matrices from shared memory (row addresses from lanes 0..31).
__device__ __forceinline__ void ldsm_x4(uint32_t r[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_addr(p)));
}
__device__ __forceinline__ void ldsm_x4_t(uint32_t r[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_addr(p)));
}

// D(16x8 f32) += A(16x16 f16, row) * B(16x8 f16, col).
__device__ __forceinline__ void mma16816(float c[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                         uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ uint32_t pack_half2(float lo, float hi) {
  __half2 h = __floats2half2_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&h);
}

// Two and four neighbouring results, rounded to fp16, at an even index of an output row: together where the caller's
// pointer is 4-byte aligned (it only has to be an fp16 pointer).
__device__ __forceinline__ void store_out2(__half* p, float x, float y) {
  if ((reinterpret_cast<uintptr_t>(p) & 3) == 0) {
    *reinterpret_cast<__half2*>(p) = __floats2half2_rn(x, y);
  } else {
    p[0] = __float2half_rn(x);
    p[1] = __float2half_rn(y);
  }
}
__device__ __forceinline__ void store_out4(__half* p, float x, float y, float z, float w) {
  store_out2(p, x, y);
  store_out2(p + 2, z, w);
}

// Exact fp16 -> fp32 widening of raw bits.
__device__ __forceinline__ float h2f(uint16_t bits) { return __half2float(__ushort_as_half(bits)); }

// Order-preserving map fp32 -> uint32 (larger float -> larger key).
__device__ __forceinline__ uint32_t f32_key(float x) {
  uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

}  // namespace mkv
