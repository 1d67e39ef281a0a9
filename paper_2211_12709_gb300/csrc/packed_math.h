// packed_math.h -- two FP32 values per instruction (fma.rn.f32x2 and kin), GELU
// with its derivative in that form.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "fno_internal.h"

namespace fno {

typedef unsigned long long u64;

// d = a b + d on two packed floats
__device__ __forceinline__ void fma2(u64& d, u64 a, u64 b) {
  asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(d) : "l"(a), "l"(b));
}
__device__ __forceinline__ u64 mul2(u64 a, u64 b) {
  u64 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 add2(u64 a, u64 b) {
  u64 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ u64 pack2(float a, float b) {
  u64 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float2 unpack2(u64 v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}

// d2 = GELU'(v) and z2 = GELU(v) of two values (phi2_as, gelu_as and
// gelu_grad_as of fno_internal.h in packed arithmetic, the same operations)
__device__ __forceinline__ void gelu2(u64 v, u64& z2, u64& d2) {
  const float2 a = unpack2(v);
  const u64 u = pack2(fabsf(a.x) * 0.70710678118654752f, fabsf(a.y) * 0.70710678118654752f);
  u64 den = pack2(1.0f, 1.0f);
  fma2(den, pack2(0.3275911f, 0.3275911f), u);
  const float2 df = unpack2(den);
  const u64 t = pack2(rcp_approx(df.x), rcp_approx(df.y));
  u64 q = pack2(-1.453152027f, -1.453152027f);
  fma2(q, pack2(1.061405429f, 1.061405429f), t);
  u64 r = pack2(1.421413741f, 1.421413741f);
  fma2(r, q, t);
  q = pack2(-0.284496736f, -0.284496736f);
  fma2(q, r, t);
  r = pack2(0.254829592f, 0.254829592f);
  fma2(r, q, t);
  r = mul2(r, t);
  const float2 ef = unpack2(mul2(mul2(u, u), pack2(-1.4426950408889634f, -1.4426950408889634f)));
  const u64 e = pack2(ex2_approx(ef.x), ex2_approx(ef.y));
  const u64 c = mul2(r, e);  // 1 - erf(u)
  u64 c2 = pack2(2.0f, 2.0f);
  fma2(c2, c, pack2(-1.0f, -1.0f));
  const float2 cf = unpack2(c), c2f = unpack2(c2);
  const u64 phi2 = pack2(a.x >= 0.f ? c2f.x : cf.x, a.y >= 0.f ? c2f.y : cf.y);
  const u64 hp = mul2(phi2, pack2(0.5f, 0.5f));
  z2 = mul2(v, hp);
  d2 = hp;
  fma2(d2, mul2(v, e), pack2(0.39894228040143268f, 0.39894228040143268f));
}

}  // namespace fno
