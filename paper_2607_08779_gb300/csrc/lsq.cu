// lsq.cu -- sss_quantize_lsq: symmetric-grid quantization with every
// group's scale refined by LSQ steps (Sec. 5 "Composition with learned
// rotations and grid parameters"; Appendix C: LSQ with s != 0 for the
// signed formats, s > 0 for the conventional ones).  The paper learns the
// scales through the model loss on calibration data; this path is the
// data-free reading on each group's own reconstruction loss
// L(s) = sum (s c_i - w_i)^2:
//   s_0 = the signed absmax scale gamma* alpha (or alpha > 0);
//   per step, in IEEE fp32 without fused multiply-add:
//     v_i = w_i / s,  c_i = clip(rint(v_i), -2^(q-1), 2^(q-1) - 1),
//     d_i = c_i - v_i inside the range, the clip value outside (LSQ's
//           straight-through estimate of dw^_i / ds),
//     t_i = (2 (s c_i - w_i)) d_i,  G = pairwise sum of t over the group
//           (t_i <- t_i + t_{i+h}, h = g/2, ..., 1),
//     s <- s - step * G, step = lr / sqrt(g (2^(q-1) - 1)) (LSQ's gradient
//           scale), keeping the sign of s (a step that would cross or reach
//           zero halves s instead);
//   then the codes of the refined scale by the quantizer's exact-quotient
//   rounding, packed in the library's layout, with the fp16 scale.
// In lsq_kernel G/32 lanes own a group, 32 elements each (lane l elements
// l + e G/32), so the pairwise sum is a tree in registers and its last log2(G/32)
// levels are shuffles -- the order above, bit for bit.
//
// Bound by instruction issue (65 % of the slots, the rest waiting on the ALU and
// FMA pipes): a step takes about 12 instructions per weight.
// The elements are held as packed pairs for the two-wide fp32 instructions,
// and the quotient w / s is formed from r = RN(1/s), once per step and group,
// by two residual corrections (Markstein, "Computation of elementary
// functions on the IBM RISC System/6000 processor", 1990: with a correctly
// rounded reciprocal and a quotient within one ulp, q + (w - q s) r rounds
// to RN(w / s)), which holds while nothing underflows; a group or step
// outside that range divides.  (One warp per group, a division per weight
// and five dependent shuffles per step took 567 us for 20 steps on 4096 x
// 4096 at q = 4, g = 32; this takes 170 us.  Few groups still go that way.)
#include <math.h>

#include <algorithm>

#include "rne.cuh"
#include "sss_internal.cuh"

namespace sss {
namespace {

constexpr int kLsqThreads = 256;

__device__ __forceinline__ uint64_t lq_pack(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ float2 lq_unpack(uint64_t v) {
  float2 f;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(f.x), "=f"(f.y) : "l"(v));
  return f;
}
__device__ __forceinline__ uint64_t lq_add(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t lq_mul(uint64_t a, uint64_t b) {
  uint64_t r;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ uint64_t lq_fma(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}

// in-lane levels of the pairwise sum: t_e + t_{e+16}, ..., t_e + t_{e+1}
__device__ __forceinline__ float lq_tree(uint64_t (&t)[16]) {
#pragma unroll
  for (int h = 8; h >= 1; h >>= 1)
#pragma unroll
    for (int p = 0; p < h; ++p) t[p] = lq_add(t[p], t[p + h]);
  const float2 f = lq_unpack(t[0]);
  return __fadd_rn(f.x, f.y);
}

// sum over the lane's 32 elements of (s c - w) d of one step (half of t)
template <int HALF>
__device__ __forceinline__ float lq_step_fast(const uint64_t (&x)[16], float s) {
  const float r = __frcp_rn(s);
  const uint64_t r2 = lq_pack(r, r), s2 = lq_pack(s, s), ns2 = lq_pack(-s, -s);
  const uint64_t magic = lq_pack(kMagic, kMagic), nmagic = lq_pack(-kMagic, -kMagic);
  const uint64_t neg1 = lq_pack(-1.f, -1.f);
  // the floats next to the clip values on the inside: a quotient outside
  // (-HALF, HALF - 1) is moved to one of them and rounds to the clip value
  const float lo = __int_as_float(__float_as_int(-static_cast<float>(HALF)) - 1);
  const float hi = __int_as_float(__float_as_int(static_cast<float>(HALF - 1)) - 1);
  uint64_t t[16];
#pragma unroll
  for (int p = 0; p < 16; ++p) {
    const uint64_t q0 = lq_mul(x[p], r2);
    const uint64_t q1 = lq_fma(lq_fma(q0, ns2, x[p]), r2, q0);
    const float2 v = lq_unpack(lq_fma(lq_fma(q1, ns2, x[p]), r2, q1));  // RN(w / s)
    const float va = fminf(fmaxf(v.x, lo), hi), vb = fminf(fmaxf(v.y, lo), hi);
    const uint64_t c = lq_add(lq_add(lq_pack(va, vb), magic), nmagic);  // rint
    const uint64_t in = lq_pack(va == v.x ? v.x : 0.f, vb == v.y ? v.y : 0.f);
    const uint64_t d = lq_fma(neg1, in, c);                   // c - v inside, c outside
    const uint64_t err = lq_fma(neg1, x[p], lq_mul(s2, c));  // RN(s c) - w
    // (scalar products: a packed one is contracted into the sum's first add)
    const float2 ef = lq_unpack(err), df = lq_unpack(d);
    t[p] = lq_pack(__fmul_rn(ef.x, df.x), __fmul_rn(ef.y, df.y));
  }
  return lq_tree(t);
}
// the same by division, and any magnitudes (2 err rounds before the product)
template <int HALF>
__device__ __noinline__ float lq_step_slow(const uint64_t (&x)[16], float s) {
  constexpr float QN = -static_cast<float>(HALF), QP = static_cast<float>(HALF - 1);
  uint64_t t[16];
#pragma unroll 1
  for (int p = 0; p < 16; ++p) {
    float o[2];
    const float2 xp = lq_unpack(x[p]);
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float w = e ? xp.y : xp.x;
      const float v = __fdiv_rn(w, s);
      float c, d;
      if (v <= QN) {
        c = d = QN;
      } else if (v >= QP) {
        c = d = QP;
      } else {
        c = fminf(fmaxf(rintf(v), QN), QP);
        d = __fsub_rn(c, v);
      }
      o[e] = __fmul_rn(__fmul_rn(2.f, __fsub_rn(__fmul_rn(s, c), w)), d);
    }
    t[p] = lq_pack(o[0], o[1]);
  }
  return lq_tree(t);
}

template <int Q, bool SIGNED, int G>
__global__ void __launch_bounds__(kLsqThreads)
    lsq_kernel(const float* __restrict__ w, int64_t ngroups, int steps, float step,
               uint8_t* __restrict__ codes, uint16_t* __restrict__ scales,
               uint32_t* __restrict__ status) {
  constexpr int L = G / 32;  // lanes per group
  constexpr int HALF = 1 << (Q - 1);
  const int l = threadIdx.x & (L - 1);
  const int64_t nthreads = ngroups * L;
  const int64_t stride = static_cast<int64_t>(gridDim.x) * kLsqThreads;
  // block-uniform trip count: every lane joins the shuffles
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * kLsqThreads; base < nthreads;
       base += stride) {
    const int64_t ti = base + threadIdx.x;
    const bool valid = ti < nthreads;
    const int64_t grp = (valid ? ti : 0) / L;
    uint64_t x[16];  // elements l + L e, e = 2p in the low half, 2p + 1 in the high
    if constexpr (L == 1) {
      const float4* src = reinterpret_cast<const float4*>(w + grp * G);
      const bool al = (reinterpret_cast<uintptr_t>(w) & 15u) == 0;  // (w is 4-byte aligned)
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        float4 v;
        if (al) {
          v = __ldg(src + j);
        } else {
          const float* f = w + grp * G + 4 * j;
          v = make_float4(__ldg(f), __ldg(f + 1), __ldg(f + 2), __ldg(f + 3));
        }
        x[2 * j] = lq_pack(v.x, v.y);
        x[2 * j + 1] = lq_pack(v.z, v.w);
      }
    } else {
#pragma unroll
      for (int p = 0; p < 16; ++p)
        x[p] = lq_pack(__ldg(w + grp * G + l + L * (2 * p)), __ldg(w + grp * G + l + L * (2 * p + 1)));
    }
    // the (signed) absmax scale, as the quantizer forms it; and whether every
    // weight is zero or of ordinary magnitude
    float mx = lq_unpack(x[0]).x, mn = mx;
    unsigned bad = 0;
    bool plain = true;
#pragma unroll
    for (int p = 0; p < 16; ++p) {
      const float2 f = lq_unpack(x[p]);
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const float v = e ? f.y : f.x;
        mx = fmaxf(mx, v);
        mn = fminf(mn, v);
        bad |= is_nonfinite(v);
        plain &= v == 0.f || (fabsf(v) >= 0x1p-40f && fabsf(v) <= 0x1p+20f);
      }
    }
#pragma unroll
    for (int o = L / 2; o >= 1; o >>= 1) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    const float M = fmaxf(mx, -mn);
    const float gamma = (SIGNED && mx > -mn) ? -1.f : 1.f;
    const float alpha = __fmul_rn(M, 1.0f / HALF);
    const bool zero = (alpha == 0.f) || bad;
    float s = zero ? 0.f : gamma * alpha;
    // ---- LSQ steps (every lane runs them all: the group's sum is shuffled;
    // a zero group's s stays 0) ----
    for (int it = 0; it < steps; ++it) {
      const float as = fabsf(s);
      float gsum = 0.f;
      if (!zero) {
        if (plain && as >= 0x1p-40f && as <= 0x1p+20f)
          gsum = __fmul_rn(2.f, lq_step_fast<HALF>(x, s));  // exact: all terms normal
        else
          gsum = lq_step_slow<HALF>(x, s);
      }
#pragma unroll
      for (int o = L / 2; o >= 1; o >>= 1)
        gsum = __fadd_rn(gsum, __shfl_xor_sync(0xffffffffu, gsum, o));
      if (!zero) {
        float sn = __fsub_rn(s, __fmul_rn(step, gsum));
        if (__fmul_rn(sn, s) <= 0.f) sn = __fmul_rn(s, 0.5f);
        s = sn;
      }
    }
    // ---- codes of the refined scale (exact-quotient rounding) ----
    int u[32];
    if (zero) {
#pragma unroll
      for (int e = 0; e < 32; ++e) u[e] = HALF;
    } else {
      float ss = s, sig = 1.f;
      const float as = fabsf(s) * static_cast<float>(HALF);  // about ||w||_inf
      if (as < 0x1p-96f || as > 0x1p+96f) {  // keep 1/s normal: scale w and s by 2^+-64
        sig = (as < 1.f) ? 0x1p+64f : 0x1p-64f;
        ss = __fmul_rn(s, sig);
      }
      const float r = __frcp_rn(ss);
#pragma unroll
      for (int p = 0; p < 16; ++p) {
        const float2 f = lq_unpack(x[p]);
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float v = e ? f.y : f.x;
          const int up = code_of<HALF>(sig == 1.f ? v : __fmul_rn(v, sig), ss, r);
          u[2 * p + e] = max(0, min(up, 2 * HALF - 1));
        }
      }
    }
    const uint16_t s16 = __half_as_ushort(__float2half_rn(s));
    // ---- pack: this lane's codes at their places in the group's words (the
    // rest zero), the lanes' words OR-ed together, and lane l stores its part
    constexpr int B = Q == 4 ? 4 : 2;     // bits of a code in the first plane
    constexpr int CW = 32 / B;            // codes per word
    constexpr int NW = G / CW;            // words of the first plane
    uint32_t W[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) W[i] = 0u;
#pragma unroll
    for (int e = 0; e < 32; ++e) {  // element l + L e: word L e / CW, since L divides CW
      const uint32_t c = static_cast<uint32_t>(Q == 3 ? (u[e] & 3) : u[e]);
      W[L * e / CW] |= c << (B * ((L * e) % CW));
    }
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      W[i] <<= B * l;
#pragma unroll
      for (int o = L / 2; o >= 1; o >>= 1) W[i] |= __shfl_xor_sync(0xffffffffu, W[i], o);
    }
    uint32_t H[L];
    if constexpr (Q == 3) {
#pragma unroll
      for (int i = 0; i < L; ++i) H[i] = 0u;
#pragma unroll
      for (int e = 0; e < 32; ++e)
        H[L * e / 32] |= static_cast<uint32_t>(u[e] >> 2) << ((L * e) % 32);
#pragma unroll
      for (int i = 0; i < L; ++i) {
        H[i] <<= l;
#pragma unroll
        for (int o = L / 2; o >= 1; o >>= 1) H[i] |= __shfl_xor_sync(0xffffffffu, H[i], o);
      }
    }
    if (valid) {
      uint32_t* dst = reinterpret_cast<uint32_t*>(codes + grp * (G * Q / 8));
      constexpr int PW = NW / L;  // words per lane
#pragma unroll
      for (int i = 0; i < NW; ++i)
        if (i / PW == l) dst[i] = W[i];
      if constexpr (Q == 3) {
#pragma unroll
        for (int i = 0; i < L; ++i)
          if (i == l) dst[NW + i] = H[i];
      }
      if (l == 0) {
        scales[grp] = s16;
        unsigned flags = bad ? SSS_FLAG_NONFINITE : 0u;
        if ((s16 & 0x7fffu) == 0x7c00u) flags |= SSS_FLAG_RANGE;
        if (flags != 0u && status != nullptr) atomicOr(status, flags);
      }
    }
  }
}

// The same with a warp per group, for few groups: lane l holds elements l + 32 e,
// so the in-lane levels of the pairwise sum come first and the last five are
// shuffles.  More instructions per weight (a division, and the shuffles for one to
// four weights), but a step takes 0.2 us where 32 weights in a row take 0.7.
template <int Q, bool SIGNED, int G>
__global__ void __launch_bounds__(kLsqThreads)
    lsq_warp_kernel(const float* __restrict__ w, int64_t ngroups, int steps, float step,
                    uint8_t* __restrict__ codes, uint16_t* __restrict__ scales,
                    uint32_t* __restrict__ status) {
  constexpr int E = G / 32;  // elements per lane
  constexpr int HALF = 1 << (Q - 1);
  constexpr float QN = -static_cast<float>(HALF), QP = static_cast<float>(HALF - 1);
  const int lane = threadIdx.x & 31;
  const int64_t warps = static_cast<int64_t>(gridDim.x) * (kLsqThreads / 32);
  for (int64_t grp = static_cast<int64_t>(blockIdx.x) * (kLsqThreads / 32) + (threadIdx.x >> 5);
       grp < ngroups; grp += warps) {  // warp-uniform
    float x[E];
#pragma unroll
    for (int e = 0; e < E; ++e) x[e] = __ldcs(w + grp * G + lane + 32 * e);
    // the (signed) absmax scale, as the quantizer forms it
    float mx = x[0], mn = x[0];
    unsigned bad = 0;
#pragma unroll
    for (int e = 0; e < E; ++e) {
      mx = fmaxf(mx, x[e]);
      mn = fminf(mn, x[e]);
      bad |= is_nonfinite(x[e]);
    }
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) {
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
      mn = fminf(mn, __shfl_xor_sync(0xffffffffu, mn, o));
      bad |= __shfl_xor_sync(0xffffffffu, bad, o);
    }
    const float M = fmaxf(mx, -mn);
    const float gamma = (SIGNED && mx > -mn) ? -1.f : 1.f;
    const float alpha = __fmul_rn(M, 1.0f / HALF);
    const bool zero = (alpha == 0.f) || bad;
    float s = zero ? 0.f : gamma * alpha;
    // ---- LSQ steps ----
    if (!zero) {
      for (int it = 0; it < steps; ++it) {
        float t[E];
#pragma unroll
        for (int e = 0; e < E; ++e) {
          const float v = __fdiv_rn(x[e], s);
          float c, d;
          if (v <= QN) {
            c = QN;
            d = QN;
          } else if (v >= QP) {
            c = QP;
            d = QP;
          } else {
            c = fminf(fmaxf(rintf(v), QN), QP);
            d = __fsub_rn(c, v);
          }
          const float err = __fsub_rn(__fmul_rn(s, c), x[e]);
          t[e] = __fmul_rn(__fmul_rn(2.f, err), d);
        }
#pragma unroll
        for (int h = E / 2; h >= 1; h >>= 1)
#pragma unroll
          for (int e = 0; e < h; ++e) t[e] = __fadd_rn(t[e], t[e + h]);
        float gsum = t[0];
#pragma unroll
        for (int o = 16; o >= 1; o >>= 1) gsum = __fadd_rn(gsum, __shfl_xor_sync(0xffffffffu, gsum, o));
        float sn = __fsub_rn(s, __fmul_rn(step, gsum));
        if (__fmul_rn(sn, s) <= 0.f) sn = __fmul_rn(s, 0.5f);
        s = sn;
      }
    }
    // ---- codes of the refined scale (exact-quotient rounding) ----
    int u[E];
    if (zero) {
#pragma unroll
      for (int e = 0; e < E; ++e) u[e] = HALF;
    } else {
      float ss = s, sig = 1.f;
      const float as = fabsf(s) * static_cast<float>(HALF);  // about ||w||_inf
      if (as < 0x1p-96f || as > 0x1p+96f) {  // keep 1/s normal: scale w and s by 2^+-64
        sig = (as < 1.f) ? 0x1p+64f : 0x1p-64f;
        ss = __fmul_rn(s, sig);
      }
      const float r = __frcp_rn(ss);
#pragma unroll
      for (int e = 0; e < E; ++e) {
        const int up = code_of<HALF>(sig == 1.f ? x[e] : __fmul_rn(x[e], sig), ss, r);
        u[e] = max(0, min(up, 2 * HALF - 1));
      }
    }
    const uint16_t s16 = __half_as_ushort(__float2half_rn(s));
    // ---- pack: element l + 32 e is code l of run e of the group ----
#pragma unroll
    for (int e = 0; e < E; ++e) {
      if constexpr (Q == 4) {  // run e: 4 words, word l/8 holds codes 8(l/8) .. +7
        uint32_t v = static_cast<uint32_t>(u[e]) << (4 * (lane & 7));
#pragma unroll
        for (int o = 1; o < 8; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
        if ((lane & 7) == 0)
          reinterpret_cast<uint32_t*>(codes + grp * (G / 2) + 16 * e)[lane >> 3] = v;
      } else if constexpr (Q == 2) {  // run e: 2 words, word l/16 holds codes 16(l/16) .. +15
        uint32_t v = static_cast<uint32_t>(u[e]) << (2 * (lane & 15));
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
        if ((lane & 15) == 0)
          reinterpret_cast<uint32_t*>(codes + grp * (G / 4) + 8 * e)[lane >> 4] = v;
      } else {  // q = 3: run e's low-plane words 2e, 2e+1; high-plane word G/16 + e
        uint32_t v = static_cast<uint32_t>(u[e] & 3) << (2 * (lane & 15));
#pragma unroll
        for (int o = 1; o < 16; o <<= 1) v |= __shfl_xor_sync(0xffffffffu, v, o);
        const uint32_t hi = __ballot_sync(0xffffffffu, (u[e] >> 2) & 1);
        uint32_t* base = reinterpret_cast<uint32_t*>(codes + grp * (3 * G / 8));
        if ((lane & 15) == 0) base[2 * e + (lane >> 4)] = v;
        if (lane == 0) base[G / 16 + e] = hi;
      }
    }
    if (lane == 0) {
      scales[grp] = s16;
      unsigned flags = bad ? SSS_FLAG_NONFINITE : 0u;
      if ((s16 & 0x7fffu) == 0x7c00u) flags |= SSS_FLAG_RANGE;
      if (flags != 0u && status != nullptr) atomicOr(status, flags);
    }
  }
}

// Whether a warp per group takes less time than 32 weights per thread: both in us
// as measured over 64 .. 16384 x 1024 with 0 .. 50 steps.  Where the lines cross
// (in 2^20 weights): groups of 32, 0.9 without steps and 0.45 at 20; of 128, 5 and
// 0.65.  (20 steps at q = 4, g = 32: 64 x 1024 6.4 us against 19.3, 256 x 1024 12.1
// against 19.6, 512 x 1024 21.5 against 19.4, 4096 x 1024 141 against 54.)
bool few_groups(int64_t weights, int group, int steps) {
  const double m = static_cast<double>(weights) / (1 << 20);
  const int64_t sms = device_sm_count(), blocks = (weights / 32 + kLsqThreads - 1) / kLsqThreads;
  const double waves = static_cast<double>((blocks + sms - 1) / sms);
  const double base = group == 32 ? 4.6 : (group == 64 ? 3.0 : 2.0);
  const double per_step = group == 32 ? 1.55 : (group == 64 ? 1.35 : 1.15);
  const double start = group == 64 ? 5.0 + 2.1 * waves : 4.5 + 1.6 * waves;
  return 2.3 + m * (base + per_step * steps) < start + (0.18 + 0.49 * waves) * steps;
}

template <int Q, bool SIGNED, int G>
cudaError_t lsq_run(const float* w, const sss_qtensor_t& t, int steps, float step,
                    uint32_t* status, cudaStream_t stream) {
  const int64_t ngroups = t.n * (t.k / G);
  const bool few = few_groups(ngroups * G, G, steps);
  const int64_t threads = ngroups * (few ? 32 : G / 32);
  const int64_t want = (threads + kLsqThreads - 1) / kLsqThreads;
  const int grid = static_cast<int>(
      std::max<int64_t>(1, std::min<int64_t>(want, static_cast<int64_t>(device_sm_count()) * 8)));
  if (few)
    lsq_warp_kernel<Q, SIGNED, G><<<grid, kLsqThreads, 0, stream>>>(w, ngroups, steps, step,
                                                                    t.codes, t.scales, status);
  else
    lsq_kernel<Q, SIGNED, G><<<grid, kLsqThreads, 0, stream>>>(w, ngroups, steps, step, t.codes,
                                                               t.scales, status);
  return cudaGetLastError();
}

template <int Q, bool SIGNED>
cudaError_t lsq_g(const float* w, const sss_qtensor_t& t, int steps, float step,
                  uint32_t* status, cudaStream_t stream) {
  switch (t.group) {
    case 32: return lsq_run<Q, SIGNED, 32>(w, t, steps, step, status, stream);
    case 64: return lsq_run<Q, SIGNED, 64>(w, t, steps, step, status, stream);
    case 128: return lsq_run<Q, SIGNED, 128>(w, t, steps, step, status, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_quantize_lsq(const float* w, const sss_qtensor_t& t, int steps, float lr,
                                uint32_t* status, cudaStream_t stream) {
  // LSQ's gradient scale 1/sqrt(g (2^(q-1) - 1)), times the rate, in fp32
  const float gscale = static_cast<float>(
      1.0 / sqrt(static_cast<double>(t.group) * static_cast<double>((1 << (t.q - 1)) - 1)));
  const float step = lr * gscale;
  const bool sgn = t.grid == SSS_GRID_SIGNED_SYM;
  switch (t.q) {
    case 2: return sgn ? lsq_g<2, true>(w, t, steps, step, status, stream)
                       : lsq_g<2, false>(w, t, steps, step, status, stream);
    case 3: return sgn ? lsq_g<3, true>(w, t, steps, step, status, stream)
                       : lsq_g<3, false>(w, t, steps, step, status, stream);
    case 4: return sgn ? lsq_g<4, true>(w, t, steps, step, status, stream)
                       : lsq_g<4, false>(w, t, steps, step, status, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace sss
