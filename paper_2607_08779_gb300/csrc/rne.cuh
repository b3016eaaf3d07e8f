// rne.cuh -- round-to-nearest-even of the exact quotient w / s in fp32
// arithmetic, shared by the quantizer and the sign diagnostics (the
// rounding of eq:quantizer; ties of the exact quotient go to even).
#pragma once

#include "sss_internal.cuh"

namespace sss {

// 1.5 * 2^23: adding it to |v| < 2^22 rounds v to an integer (ties to even)
// held in the low mantissa bits.
constexpr float kMagic = 12582912.0f;

// The exact-residual side decision for one weight whose rounded code is
// u (c = u - OFF the integer w*r rounded to): when w*r lies within 2^-18
// of the half-integer h between c and its neighbour, the sign of the
// single-rounding residual w - h*s places the exact quotient; a zero
// residual is an exact tie -> even.  Returns the corrected code.
template <int OFF>
__device__ __forceinline__ int fix_tie(float w, float s, float r, int u) {
  const float c = static_cast<float>(u - OFF);
  const float dd = __fmaf_rn(w, r, -c);  // w*r - c
  if (fabsf(__fsub_rn(fabsf(dd), 0.5f)) <= 0x1p-18f) {
    const float h = __fadd_rn(c, copysignf(0.5f, dd));   // the half-integer at stake
    const float e = __fmaf_rn(-h, s, w);                  // w - h*s, one rounding
    const float side = (s > 0.f) ? e : -e;                // sign of (w/s - h)
    const float lo = __fsub_rn(h, 0.5f), hi = __fadd_rn(h, 0.5f);
    float cc;
    if (side > 0.f) {
      cc = hi;
    } else if (side < 0.f) {
      cc = lo;
    } else {  // exact tie: to even
      cc = (static_cast<int>(lo) & 1) ? hi : lo;
    }
    u += static_cast<int>(__fsub_rn(cc, c));
  }
  return u;
}

// Stored code u = RNE(w / s) + OFF of the EXACT quotient, given r = RN(1/s)
// (OFF = 2^(q-1) for the symmetric grids, 0 for the min-max grid; OFF is
// even, so the parity of the rounded sum is that of the code).  One FMA
// rounds w*r straight to an integer; a second FMA gives the remainder
// w*r - c.  Only when that remainder is within 2^-18 of +-1/2 can the exact
// quotient fall on the other side of the half-integer (|w*r - w/s| <=
// 16 * 2^-24 here); fix_tie then decides it.
template <int OFF>
__device__ __forceinline__ int code_of(float w, float s, float r) {
  constexpr float MAGIC = kMagic + static_cast<float>(OFF);
  const float t = __fmaf_rn(w, r, MAGIC);
  const int u = __float_as_int(t) - __float_as_int(kMagic);
  const float dd = __fmaf_rn(w, r, __fsub_rn(MAGIC, t));  // w*r - c; MAGIC - t = -c exactly
  if (fabsf(__fsub_rn(fabsf(dd), 0.5f)) <= 0x1p-18f) return fix_tie<OFF>(w, s, r, u);
  return u;
}

// two fp32 values as the packed operand of the two-wide fp32 instructions
// (each half rounds as the scalar instruction)
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// The same for 2N weights at once (w[p] holds weights 2p and 2p + 1; the same
// codes as 2N calls of code_of): every weight's rounding in one straight line,
// two weights to an instruction, and a single branch, taken only when some
// weight lies within 2^-18 of a half-integer (w*r - c is at most 1/2 in
// magnitude), into the exact side decisions.  That branch takes weight e from
// wat(e), which must return the value held in w, so that w need not stay in
// registers past the straight line.  t[e] is returned as the float kMagic + u,
// whose low bits are the code: it is clamped and packed as it is.
template <int OFF, int N, class Wat>
__device__ __forceinline__ void codes_of(const uint64_t (&w)[N], float s, float r,
                                         float (&t)[2 * N], Wat wat) {
  constexpr float MAGIC = kMagic + static_cast<float>(OFF);
  const uint64_t r2 = pack2(r, r), m2 = pack2(MAGIC, MAGIC), neg1 = pack2(-1.f, -1.f);
  float near = 0.f;
#pragma unroll
  for (int p = 0; p < N; ++p) {
    const uint64_t t2 = fma2(w[p], r2, m2);
    float d0, d1;
    unpack2(fma2(w[p], r2, fma2(neg1, t2, m2)), d0, d1);  // w*r - c; MAGIC - t = -c exactly
    near = fmaxf(near, fmaxf(fabsf(d0), fabsf(d1)));
    unpack2(t2, t[2 * p], t[2 * p + 1]);
  }
  if (near >= 0.5f - 0x1p-18f) {  // unrolled: t stays in registers
#pragma unroll
    for (int e = 0; e < 2 * N; ++e) {
      const int u = __float_as_int(t[e]) - __float_as_int(kMagic);
      t[e] = __int_as_float(__float_as_int(kMagic) + fix_tie<OFF>(wat(e), s, r, u));
    }
  }
}

}  // namespace sss
