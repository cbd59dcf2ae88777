// Arithmetic on a query's row that the attention / recovery kernels share: packed float32, the exponential on the FMA pipe,
// 32-byte stores, the unit of the recurrence.
#pragma once
#include "sm100_ptx.cuh"

#include <cuda_runtime.h>
#include <stdint.h>

namespace csat {
namespace rowmath {

__device__ __forceinline__ float max3(float a, float b, float c) {
  float y;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(y) : "f"(a), "f"(b), "f"(c));
  return y;
}
// 32-byte store (the address is 32-byte aligned)
__device__ __forceinline__ void st_global_v8(void* p, const uint32_t (&r)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(r[0]), "r"(r[1]), "r"(r[2]),
               "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// two-element packed fp32 arithmetic (one instruction for both halves of a register pair): the compiler's float2
// builtins, so that it sees the register pairs (inline assembly on 64-bit registers cost extra moves and spills)
using F2 = float2;
__device__ __forceinline__ F2 pack2(float lo, float hi) { return make_float2(lo, hi); }
__device__ __forceinline__ F2 pack2u(uint32_t lo, uint32_t hi) { return make_float2(__uint_as_float(lo), __uint_as_float(hi)); }
__device__ __forceinline__ void unpack2(F2 v, float& lo, float& hi) { lo = v.x; hi = v.y; }
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ F2 add2(F2 a, F2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ F2 sub2(F2 a, F2 b) { return __fadd2_rn(a, make_float2(-b.x, -b.y)); }
__device__ __forceinline__ F2 mul2(F2 a, F2 b) { return __fmul2_rn(a, b); }

// exp2 of both halves on the FMA pipe (the MUFU unit is the bottleneck of the softmax: 4 lanes per clock and
// sub-core).  x <= ~9; anything below -120 (masked columns are -inf) gives 2^-120.  Round-to-nearest split
// x = i + f, f in [-1/2, 1/2]; 2^f by a cubic fitted to 7.5e-5 relative error (P is rounded to bf16, 3.9e-3,
// and the row sum tolerates far more); 2^i by adding i to the exponent field.
__device__ __forceinline__ void exp2_poly2(F2 x2, float& p0, float& p1) {
  float x0, x1;
  unpack2(x2, x0, x1);
  x2 = pack2(fmaxf(x0, -120.f), fmaxf(x1, -120.f));
  const F2 magic = pack2(12582912.f, 12582912.f);          // 1.5 * 2^23: the sum's low mantissa bits hold i
  const F2 t2 = add2(x2, magic);
  const F2 f2 = sub2(x2, sub2(t2, magic));
  F2 q2 = fma2(f2, pack2(0.055171459913253784f, 0.055171459913253784f), pack2(0.2426108568906784f, 0.2426108568906784f));
  q2 = fma2(q2, f2, pack2(0.6932609677314758f, 0.6932609677314758f));
  q2 = fma2(q2, f2, pack2(0.9999281167984009f, 0.9999281167984009f));
  float t0, t1, q0, q1;
  unpack2(t2, t0, t1);
  unpack2(q2, q0, q1);
  p0 = __int_as_float(__float_as_int(q0) + (__float_as_int(t0) << 23));
  p1 = __int_as_float(__float_as_int(q1) + (__float_as_int(t1) << 23));
}

// The recurrence in units of 2 theta needs z / (2 theta) far from overflow.  theta = mu lambda may be so small, or zero in float32,
// that it is not: kernels with both forms then keep the data's units, the others take a unit of 2^-70 of the row's largest
// magnitude: as a threshold that is less than a rounding of what is above 2^-46 of that magnitude, and little of the rest.
__device__ __forceinline__ bool threshold_is_a_unit(float theta) { return theta >= 0x1p-50f; }
// The row is `scale` times the N columns of tensor memory from addr on.  (To be called before the row is read into registers: a
// branch between that and their first use cost 1 % of both kernels, with thresholds that never took it.)
template <int N> __device__ __forceinline__ float unit_threshold(float theta, uint32_t addr, float scale) {
  if (threshold_is_a_unit(theta)) return theta;
  float mx = 0x1p-56f;                                        // a normal number after the scaling below
#pragma unroll 1
  for (int c0 = 0; c0 < N; c0 += 16) {
    uint32_t a[16];
    ptx::tmem_ld_32x32b_x16(addr + c0, a);
    ptx::tmem_wait_ld();
#pragma unroll
    for (int e = 0; e < 16; ++e) mx = fmaxf(mx, fabsf(__uint_as_float(a[e]) * scale));
  }
  return fmaxf(theta, fminf(mx, 3.402823466e38f) * 0x1p-70f);  // (an infinity in the row stays one)
}

constexpr int kPolyEvery = 4;          // every 4th pair of scores takes the polynomial exp2 (measured best of 1, 2, 3, 4, none)

}  // namespace rowmath
}  // namespace csat
