// Demodulation of one symbol by packed fp32 arithmetic (Def. III.1 / III.2 on
// the Q8.8 grid), shared by the fused decode and the public demodulation.
#pragma once

#include <stdint.h>

#include "host_util.cuh"

namespace grand {

// Demodulation constants of one constellation for the packed floating-point
// arithmetic on both axes (axes_fast): each value twice.
struct AxisConst {
  float2 q;      // 256 / d
  float2 nz;     // -0 (see grid2)
  float2 t0;     // -(1.5 * 2^23 - 256 sqrt(M) + 512)
  float2 g;      // sqrt(M) - 2: the range of the thresholds' indices
  float s, c;    // t s + c: that range scaled to [0, 1]
  float lim;     // |a q| up to which the ordering key is exact in 23 bits
  float side;    // sqrt(M)
  uint64_t below_top;  // labels of four symbols, m bits an axis: every bit but the top one of each axis
};

// Constants of axes_fast for sqrt(M) = 2^m. t + 512 = round(a q) + 256 sqrt(M);
// the nearest inner threshold (ties down) is k = floor((t + 255) / 512) =
// round((t - 3/4) / 512) within [0, sqrt(M) - 2]; with one inner threshold
// (QPSK) it is 0.
inline AxisConst axis_const(int m, const QamConst& qc) {
  const double side = (double)(1 << m), range = side - 2.0;
  auto twice = [](double v) { return make_float2((float)v, (float)v); };
  AxisConst c;
  c.q = make_float2(qc.q[m], qc.q[m]);
  c.nz = make_float2(-0.0f, -0.0f);
  c.t0 = twice(-(12582912.0 - 256.0 * side + 512.0));
  c.g = twice(range);
  c.s = m > 1 ? (float)(1.0 / (512.0 * range)) : 0.0f;
  c.c = m > 1 ? (float)(-0.75 / (512.0 * range)) : 0.0f;
  c.lim = (float)(256.0 * side + 1500.0);  // distances up to 2012: keys below 2^23
  c.side = (float)side;
  c.below_top = ((1ull << 8 * m) - 1ull) / ((1ull << m) - 1ull) * ((1ull << (m - 1)) - 1ull);
  return c;
}

constexpr float kMagic = 12582912.0f;  // 1.5 * 2^23: adding it rounds to the nearest integer, ties to even

// Two floats in one 64-bit register pair, one instruction for both.
typedef unsigned long long F2;
__device__ __forceinline__ F2 pack2(float a, float b) {
  F2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b));
  return r;
}
__device__ __forceinline__ F2 pack2(float2 v) { return pack2(v.x, v.y); }
__device__ __forceinline__ float2 unpack2(F2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
  F2 r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
  F2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
  F2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
// Both axes of a symbol on the Q8.8 grid (the reading of demod_axis_q) in
// floating point: the integers involved are below 2^24, so every step is
// exact, the FMA pipe takes what would crowd the integer ALU, and the packed
// forms do I and Q in one instruction (about 10 instructions for what took
// 50 in integer form). x = a q rounded to float. k = index of the inner
// decision threshold nearest to the received value (threshold k separates the
// levels k and k + 1), e = the signed distance to it. Ties between two
// thresholds go to the lower one, so that the neighbour of a value on a level
// is the lower level; |e| > 256 says the value lies beyond the outermost level,
// where the far threshold has no neighbour level. For |x| up to 2^22; beyond,
// k stays right and |e| stays above 256.
struct Axes {
  float2 kb;  // k plus 1.5 * 2^23: k in the low 6 bits of the representation
  float2 k, e;
};

// The constants of one constellation in registers. The empty statements keep
// the compiler from building the pairs anew for every symbol (packed
// instructions take no immediates), which was 30 of 240 instructions a frame.
struct AxisRegs {
  F2 q, nz, t0, g, magic, unmagic, m512;
  float s, c, lim, side;
};
__device__ __forceinline__ AxisRegs axis_regs(const AxisConst& a, float2 nz) {
  AxisRegs r;
  r.q = pack2(a.q);
  r.nz = pack2(nz);
  r.t0 = pack2(a.t0);
  r.g = pack2(a.g);
  r.magic = pack2(kMagic, kMagic);
  r.unmagic = pack2(-kMagic, -kMagic);
  r.m512 = pack2(-512.0f, -512.0f);
  asm volatile("" : "+l"(r.q), "+l"(r.t0), "+l"(r.g), "+l"(r.magic), "+l"(r.unmagic), "+l"(r.m512));
  r.s = a.s;
  r.c = a.c;
  r.lim = a.lim;
  r.side = a.side;
  return r;
}
// Both coordinates on the grid, rounded to float as the definition has it. A
// multiply-add with -0, which no compiler can know to be one: left as a product
// (mul.rn.f32x2), it was joined with the addition of 1.5 * 2^23 that follows,
// .rn notwithstanding, and a product that rounds to a half (-768.5) went to the
// other integer. That moved a threshold's distance by one: 4 of 200,000 frames
// had an alternative too few.
__device__ __forceinline__ F2 grid2(F2 v, const AxisRegs& c) { return fma2(v, c.q, c.nz); }

__device__ __forceinline__ Axes axes_fast(F2 x, const AxisRegs& c) {
  const F2 t = add2(add2(x, c.magic), c.t0);  // round(x) + 256 sqrt(M) - 512
  const float2 ts = unpack2(t);
  // threshold index: the nearest one, clamped to the inner thresholds by the
  // saturation, rounded by the addition; no value lies on a tie (the offset is
  // a quarter of the grid)
  const float uI = __saturatef(__fmaf_rn(ts.x, c.s, c.c)), uQ = __saturatef(__fmaf_rn(ts.y, c.s, c.c));
  const F2 kb = fma2(pack2(uI, uQ), c.g, c.magic);
  const F2 k = add2(kb, c.unmagic);
  Axes r;
  r.kb = unpack2(kb);
  r.k = unpack2(k);
  r.e = unpack2(fma2(k, c.m512, t));
  return r;
}
}  // namespace grand
