// Accurate gate functions of the GRU cell, two columns at a time (split-operand kernel; accurate variant of the pipelined kernel).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

namespace marl {

constexpr float TS_LOG2E = 1.44269504088896340736f;

#ifdef __CUDACC__
__device__ __forceinline__ float ts_ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ts_rcp(float x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float ts_min(float x, float y) {  // (a NaN stays)
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(x), "f"(y));
  return d;
}
// Two fp32 values side by side (fma.rn.f32x2 and its like: each half rounds like the scalar operation).
typedef unsigned long long ts_f2;
__device__ __forceinline__ ts_f2 f2(float lo, float hi) {
  ts_f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ ts_f2 f2(float v) { return f2(v, v); }
__device__ __forceinline__ void f2_get(ts_f2 v, float& lo, float& hi) { asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v)); }
__device__ __forceinline__ ts_f2 f2_fma(ts_f2 a, ts_f2 b, ts_f2 c) {
  ts_f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ ts_f2 f2_mul(ts_f2 a, ts_f2 b) {
  ts_f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ ts_f2 f2_add(ts_f2 a, ts_f2 b) {
  ts_f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}

// The GRU's gate math on two columns: accumulators r, z, candidate input, candidate hidden; biases (b[0], b[1] already
// times -log2 e; HALVED: accumulators and biases of r and z are half the sums, as they are); h in and out.  Bound by the special-function unit (16 results per clock and SM), so reciprocals are
// shared: 1 / (dr dz) serves reset and update gate, one more both candidates - 4.5 special functions per column
// instead of 6 - and everything else runs two columns per instruction.
//   sigmoid(v) = 1 / (1 + 2^s), s = -log2(e) v: the approximate exponential's 2^-22.5 enters with weight
//   sigmoid (1 - sigmoid) <= 1/4.  Exponents are cut at 60: the products of two denominators stay finite.
//   tanh(u): below 0.6 the odd polynomial u + u^3 P(u^2), P a degree-4 minimax fit (weighted least squares iterated to
//   equal ripple, 2.8e-9), else 1 - 2 / (1 + e^(2 |u|)), where the exponential's error has faded to an ulp.
template <bool HALVED>
__device__ __forceinline__ void gates2(const float (&v)[4][2], const ts_f2* b, float& h0, float& h1) {
  const ts_f2 one = f2(1.0f);
  float s0, s1, z0, z1;
  if constexpr (HALVED) {
    f2_get(f2_mul(f2_add(f2(v[0][0], v[0][1]), b[0]), f2(-2.0f * TS_LOG2E)), s0, s1);
    f2_get(f2_mul(f2_add(f2(v[1][0], v[1][1]), b[1]), f2(-2.0f * TS_LOG2E)), z0, z1);
  } else {
    f2_get(f2_fma(f2(v[0][0], v[0][1]), f2(-TS_LOG2E), b[0]), s0, s1);
    f2_get(f2_fma(f2(v[1][0], v[1][1]), f2(-TS_LOG2E), b[1]), z0, z1);
  }
  const ts_f2 dr = f2_add(f2(ts_ex2(ts_min(s0, 60.f)), ts_ex2(ts_min(s1, 60.f))), one);
  const ts_f2 dz = f2_add(f2(ts_ex2(ts_min(z0, 60.f)), ts_ex2(ts_min(z1, 60.f))), one);
  float p0, p1;
  f2_get(f2_mul(dr, dz), p0, p1);
  const ts_f2 inv = f2(ts_rcp(p0), ts_rcp(p1));
  const ts_f2 rg = f2_mul(inv, dz), zg = f2_mul(inv, dr);
  const ts_f2 u = f2_fma(rg, f2_add(f2(v[3][0], v[3][1]), b[3]), f2_add(f2(v[2][0], v[2][1]), b[2]));
  float u0, u1, d0, d1;
  f2_get(u, u0, u1);
  const float a0 = fabsf(u0), a1 = fabsf(u1);
  f2_get(f2_add(f2(ts_ex2(ts_min(2.0f * TS_LOG2E * a0, 60.f)), ts_ex2(ts_min(2.0f * TS_LOG2E * a1, 60.f))), one), d0, d1);
  const float q = ts_rcp(d0 * d1);
  float g0, g1, l0, l1;
  f2_get(f2_fma(f2(q * d1, q * d0), f2(-2.0f), one), g0, g1);
  const ts_f2 w = f2_mul(u, u);
  ts_f2 p = f2_fma(f2(-0.00589515688f), w, f2(0.0207959712f));
  p = f2_fma(p, w, f2(-0.0537838303f));
  p = f2_fma(p, w, f2(0.133319244f));
  p = f2_fma(p, w, f2(-0.333332986f));
  f2_get(f2_fma(f2_mul(p, w), u, u), l0, l1);
  const ts_f2 c = f2(a0 < 0.6f ? l0 : copysignf(g0, u0), a1 < 0.6f ? l1 : copysignf(g1, u1));
  f2_get(f2_fma(zg, f2_fma(c, f2(-1.0f), f2(h0, h1)), c), h0, h1);  // (1 - z) * cand + z * h
}
#endif

}  // namespace marl
