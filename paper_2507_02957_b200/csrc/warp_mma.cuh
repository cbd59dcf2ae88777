// Warp-level matrix instructions (m16n8k16, bf16 operands, float32 accumulator) for stages whose accumulator, softmax or
// shrinkage and next operand belong to the same 16 rows.  The accumulator's layout of one product is the A operand's
// layout of the next, so the chain of a row block runs inside one warp: no barrier, no tensor-memory or shared-memory
// round trip between a product and the arithmetic on it.  Measured on one B200: 983 multiply-adds per clock and SM
// (8 cycles per instruction and sub-core), against about 4096 for tcgen05.mma: worth it where the chain, not the
// products' rate, is what a layer waits for.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "sm100_ptx.cuh"

namespace csat {
namespace wmma16 {

// d += a b.  Lane l = 4 g + t holds of the 16 x 8 accumulator rows g, g + 8 (registers 0, 1 and 2, 3), columns 2 t, 2 t + 1
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1));
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const __nv_bfloat16* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"((uint32_t)__cvta_generic_to_shared(p)) : "memory");
}
// 16 bytes global -> shared; zeros where !in
__device__ __forceinline__ void cp16(__nv_bfloat16* s, const void* g, bool in) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"((uint32_t)__cvta_generic_to_shared(s)), "l"(g), "r"(in ? 16 : 0));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

__device__ __forceinline__ uint32_t pack(float a, float b) { return ptx::pack_bf16(a, b); }
using ptx::add_sat;
using ptx::ex2;
using ptx::fma_sat;

// the 16 x D float32 rows x (accumulator layout, NT = D / 8 tiles of 8 columns) as bf16 A operands of D / 16 steps
template <int NT> __device__ __forceinline__ void to_operand(uint32_t (&a)[NT / 2][4], const float (&x)[NT][4]) {
#pragma unroll
  for (int k = 0; k < NT / 2; ++k) {
    a[k][0] = pack(x[2 * k][0], x[2 * k][1]);
    a[k][1] = pack(x[2 * k][2], x[2 * k][3]);
    a[k][2] = pack(x[2 * k + 1][0], x[2 * k + 1][1]);
    a[k][3] = pack(x[2 * k + 1][2], x[2 * k + 1][3]);
  }
}

// bf16 rows of NT tiles to global memory, 8 bytes per lane and instruction, whole 32-byte sectors: lanes t and t ^ 1 swap so
// that the even one holds four columns of tile j, the odd one of tile j + 1.  row[u]: the place of row g + 8 u, or null.
template <int NT>
__device__ __forceinline__ void store_rows(__nv_bfloat16* const (&row)[2], const float (&x)[NT][4], int t) {
  const bool odd = t & 1;
#pragma unroll
  for (int j = 0; j < NT; j += 2)
#pragma unroll
    for (int u = 0; u < 2; ++u) {
      const uint32_t p0 = pack(x[j][2 * u], x[j][2 * u + 1]), p1 = pack(x[j + 1][2 * u], x[j + 1][2 * u + 1]);
      const uint32_t got = __shfl_xor_sync(0xffffffffu, odd ? p0 : p1, 1);
      if (row[u])
        *reinterpret_cast<uint2*>(row[u] + 8 * (j + (odd ? 1 : 0)) + 2 * (t & 2)) = odd ? make_uint2(got, p1) : make_uint2(p0, got);
    }
}

}  // namespace wmma16
}  // namespace csat
