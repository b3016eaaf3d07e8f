// gemv_cluster.cu -- decode GEMV for batches of 2..16 activation vectors over
// packed q = 2 and q = 4 codes (sm_103a): thread-block clusters split k, the
// group scales meet the tensor cores' integer dots in fp32.
//
// y[b][r] = sum_k w^[r][k] x[b][k] as the Appendix B.3 expansion, per group:
// s (sum u x - 2^(q-1) sum x), or s sum u x + m sum x for the min-max grid.
//
//  * The batch fills the columns of mma.sync m16n8k16.  An mma's four quads
//    take their k from one 32-code sub-chunk, eight codes each, so its result
//    belongs to one group and the scale is applied to it in fp32 (4 FFMA per
//    group, tile and column block): the weight operand is the bare code, one
//    AND per pair, where an operand that carries its scale needs an AND, a
//    subtract and a multiply, and rounds to fp16.  A code field masked in
//    place is the fp16 subnormal u 2^pos 2^-24, exact; the staged x carries
//    2^-pos.  The symmetric offset enters as the accumulator's start value.
//  * The tensor core lines products up by the operands' exponent fields, so the
//    leading zeros of a subnormal cost the result low bits.  At q = 2 the fields
//    are taken as high in the mantissa as they go, pos 6 and 8 (at pos 0 .. 4 the
//    error against 64 bits was 2e-6 of the result, 1e-7 to 2e-7 now; the symmetric
//    grids' weights are exact in fp16 there, so that gemv_batch.cu has 2e-7 to
//    4e-6).  At q = 4, pos 0 and 4, it is 5e-7 against 2e-4; CUT shapes, which the
//    general kernel computes to 2e-7 .. 3e-7, take pos 2 and 6.
//  * ldmatrix hands quad t the t-th 32-bit word of a row's 16 bytes.  q = 4:
//    the words of one sub-chunk.  q = 2: 16 bytes are two sub-chunks, and one
//    shuffle and two byte permutes give every quad eight codes of each.
//  * A warp's tile is 32 rows (each B operand then feeds two mmas, which
//    balances shared-memory reads and instruction issue), a step 128 codes; its
//    codes and scales come through a private ring of 16-byte cp.async copies,
//    no barriers.
//  * CUT, a k that is no multiple of 256 or scale rows of 2-byte alignment: a
//    row's last step may be cut short.  Codes past k are not copied and meet
//    zeros of x; scales past the row are zeros.  (14336 x 4128 and x 4160, q = 4,
//    batch 4: 27 and 30 us in the general kernel, 18.5 and 14 here; batch 16: 90
//    and 116 us, 25 and 20 here: that kernel repeats its mmas per batch row.)
//  * A cluster of S CTAs shares its row tiles and splits k: each CTA stages
//    only k/S of x (staging all of x in every CTA, 128 KB at batch 16 and k =
//    4096, took as long as a small matrix's weights); each warp stores its
//    partial sums into the shared memory of the CTA that owns the outputs, and
//    after one cluster barrier the owners add them in a fixed order.
// Measured (q = 4, g = 32, batch 4 / 16): 14336 x 4096 11.4 / 15.5 us, 4096 x
// 4096 5.2 / 8.5 us, 4096 x 14336 10.5 / 18.7 us; the kernel with the scaled
// fp16 operand took 13.3 / 18.1, 7.4 / 10.5 and 16.4 / 32.8 us.  Bound at batch
// 4 by the start (launch, staging x: about 3500 cycles) and the copies in
// flight, at batch 16 by instruction issue (about 450 instructions per step,
// 43 % of the slots used) and the mma chains behind it.  The min-max grid with
// groups of 32 pays for its exactness at large n and k: 8192 x 16384 at batch 2
// 28.6 us against 26.0 with fp16-rounded weights (q = 4).
#include <cooperative_groups.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <type_traits>

#include "gemv_common.cuh"

namespace cg = cooperative_groups;

namespace sss {
namespace {

using namespace gv;

constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
constexpr int kRows = 32;   // rows of a tile
constexpr int kStep = 128;  // codes of a step
constexpr int kSmemMax = 227 * 1024;
constexpr int kMaxCluster = 8;

struct ClusterArgs {
  const uint8_t* codes;
  const uint16_t* scales;
  const uint16_t* mins;
  const uint16_t* x;  // bf16 [batch][k]
  float* y;           // [batch][n]
  int64_t n, k;
  int batch;
  int ntiles;
  int nsteps;     // k / 128, rounded up
  int csteps;     // steps per CTA of a cluster
  int wsteps;     // steps per warp of a tile's group
  int salign;     // bytes the scale rows are aligned to: 16, 8, 4 or 2
  int calign;     // bytes the code rows are aligned to: 16 or 8
  int lgkw;       // log2(warps per tile)
  int rounds;     // tiles per warp group and pass (the partial array's depth)
  uint32_t* status;
};

__device__ __forceinline__ void cp_async(uint32_t dst, const void* src, int bytes) {
  // (the 4- and 8-byte forms exist with .ca only)
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
  else if (bytes == 8)
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(dst), "l"(src) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst), "l"(src) : "memory");
}
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }

__device__ __forceinline__ void ldmatrix4(uint32_t (&w)[4], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
               : "r"(addr)
               : "memory");
}
// D = A B + C
__device__ __forceinline__ void mma_c(float (&d)[4], uint32_t a0, uint32_t a1, uint32_t a2,
                                      uint32_t a3, uint32_t b0, uint32_t b1, float c0, float c1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 "
      "{%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%10,%11,%10,%11};\n"
      : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(c0), "f"(c1));
}

// NBLK column blocks of 8; D ring stages
template <int Q, bool ASYM, int G, int NBLK, int D>
struct Shape {
  static constexpr int NBC = 8 * NBLK;
  static constexpr int SEG = kStep / G < 1 ? 1 : kStep / G;  // groups a step touches
  static constexpr int P = 16 * Q;                           // code bytes of a row in a step
  // Scales come in blocks of several steps: a copy of one step's few bytes per
  // row costs a 32-byte sector per row each time (at q = 2, g = 64 with mins,
  // twice the codes' own sectors).  A block is copied with the first step that
  // needs it and shares the ring's depth.
  static constexpr int BS = G == 32 ? 2 : 4;                 // steps of a block
  static constexpr int SB = BS * kStep / G * 2;              // its bytes per row: 16, 16, 8
  static constexpr int CODE = kRows * P;
  static constexpr int BLOCK = kRows * SB * (ASYM ? 2 : 1);
  static constexpr int STAGE = CODE + BLOCK;                 // of ring memory per slot
  static constexpr int RING = kWarps * D * STAGE;
  static constexpr int XSTEP = 4 * NBLK * 512;               // staged x bytes per step
  static constexpr int BSTEP = SEG * NBC * 4;                // row sums per step
  static constexpr int PART = kWarps * NBC * kRows * 4;      // partials per round
  static constexpr size_t bytes(int csteps, int rounds) {
    return static_cast<size_t>(RING) + static_cast<size_t>(csteps) * (XSTEP + BSTEP) +
           static_cast<size_t>(rounds) * PART;
  }
};

// One output by plain fp32 arithmetic, for a sum that came out infinite or NaN.
// An activation from 65520 on is infinite as the operand, and its product with the
// codes meets the offset's product as inf - inf; here it meets the dequantised
// weight, which has a sign.  (14336 x 4096, q = 2 min-max, one such batch row: 117
// us at batch 4, 287 at batch 16; a warp per output, 128 and 142, made every other
// call 1 to 3 % slower, this 0.2 %.)
template <int Q, bool ASYM, int G>
__device__ __noinline__ float plain_dot(const ClusterArgs& a, int64_t r, int col) {
  const int64_t ng = a.k / G;
  const uint8_t* codes = a.codes + r * (a.k * Q / 8);
  const uint4* x = reinterpret_cast<const uint4*>(a.x + col * a.k);
  float y = 0.f;
  for (int64_t g = 0; g < ng; ++g) {
    const float s = __half2float(__ushort_as_half(a.scales[r * ng + g]));
    const float m = ASYM ? __half2float(__ushort_as_half(a.mins[r * ng + g])) : 0.f;
    float d = 0.f;
    for (int i = 0; i < G / 8; ++i, codes += Q) {  // eight codes: q bytes
      const uint32_t c = Q == 4 ? *reinterpret_cast<const uint32_t*>(codes)
                                : *reinterpret_cast<const uint16_t*>(codes);
      const uint4 xv = *x++;
      const uint32_t w[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        const float u = static_cast<float>((c >> (Q * e)) & ((1u << Q) - 1u));
        const float xe = __uint_as_float(e & 1 ? w[e / 2] & 0xFFFF0000u : w[e / 2] << 16);
        d = fmaf(ASYM ? fmaf(s, u, m) : s * (u - static_cast<float>(1 << (Q - 1))), xe, d);
      }
    }
    y += d;
  }
  return y;
}

// CUT: k is not a multiple of 256, or scale rows are aligned to 2 bytes only.
template <int Q, bool ASYM, int G, int NBLK, int D, bool CUT>
__global__ void __launch_bounds__(kThreads, 1)
    gemv_cluster_kernel(const __grid_constant__ ClusterArgs a) {
  using SH = Shape<Q, ASYM, G, NBLK, D>;
  constexpr int NBC = SH::NBC, SEG = SH::SEG, P = SH::P, SB = SH::SB, BS = SH::BS;
  constexpr int HALF = 1 << (Q - 1);
  constexpr int CPR = P / 16;  // 16-byte chunks of a row in a step
  constexpr float kScale = Q == 2 ? 0x1p-18f : (CUT ? 0x1p-22f : 0x1p-24f);  // of the mmas' results
  extern __shared__ __align__(128) unsigned char smem[];
  cg::cluster_group cluster = cg::this_cluster();
  const int S = static_cast<int>(cluster.num_blocks()), lgS = 31 - __clz(S);
  const int rank = static_cast<int>(cluster.block_rank());
  const int nclus = static_cast<int>(gridDim.x) / S;
  const int cid = static_cast<int>(blockIdx.x) / S;

  // ---- shared memory: ring | x | row sums | partials ----
  const uint32_t ring0 = su32(smem);
  const uint32_t xs_a = ring0 + SH::RING;
  float* bsum = reinterpret_cast<float*>(smem + SH::RING + a.csteps * SH::XSTEP);
  float* part = bsum + a.csteps * SEG * NBC;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gq = lane >> 2, tq = lane & 3;
  const int lgkw = a.lgkw, KW = 1 << lgkw, ngrp = kWarps >> lgkw;
  const int grp = warp >> lgkw, kw = warp & (KW - 1);
  // this CTA's steps of k, and this warp's upw ones from s0 + u0 on
  const int s0 = rank * a.csteps;
  const int ns = max(0, min(a.csteps, a.nsteps - s0));
  const int u0 = min(ns, kw * a.wsteps), upw = min(a.wsteps, ns - u0);
  const int64_t row_bytes = a.k * Q / 8;
  const int64_t nG = a.k / G;
  const int pass_tiles = a.rounds * ngrp;  // tiles of a pass, per cluster
  const int share = NBC * kRows / S;        // outputs of a tile per CTA
  const int my_tiles = cid < a.ntiles ? (a.ntiles - cid + nclus - 1) / nclus : 0;

  // "this CTA has started": the peers store into its shared memory, which they
  // may do only once they know that it runs
  if (S > 1) asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  // in this order: a next kernel that reads its weights early then finds written
  // what the launches before this one wrote
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  // ---- the warp's stream: its steps of tiles grp, grp + ngrp, ... of the
  // cluster's (tile j of the cluster is tile cid + j nclus) ----
  const uint32_t my_ring = ring0 + static_cast<uint32_t>(warp) * (D * SH::STAGE);
  const int wt = grp < my_tiles ? (my_tiles - grp + ngrp - 1) / ngrp : 0;  // tiles of this warp
  const int total = wt * upw;
  int ft = 0, fleft = 0;  // fetch cursor: tile number, steps left in it
  const uint8_t* cp[4];
  const uint16_t* sp = nullptr;
  const uint16_t* mp = nullptr;
  int fstep = 0, fblk = 0;  // step of the row, block slot in use
  auto fetch_tile = [&]() {
    if (ft >= wt) return;
    const int64_t r0 = (static_cast<int64_t>(cid) + static_cast<int64_t>(grp + ft * ngrp) * nclus) * kRows;
#pragma unroll
    for (int i = 0; i < CPR; ++i) {  // chunk lane + 32 i of the stage
      const int64_t r = min(r0 + (lane + 32 * i) / CPR, a.n - 1);  // (rows past n: never stored)
      cp[i] = a.codes + r * row_bytes + static_cast<int64_t>(s0 + u0) * P + 16 * (lane % CPR);
    }
    const int64_t r = min(r0 + lane, a.n - 1);
    fstep = s0 + u0;
    sp = a.scales + r * nG;
    if constexpr (ASYM) mp = a.mins + r * nG;
    fleft = upw;
  };
  auto fetch = [&](int slot) {
    const uint32_t st = my_ring + static_cast<uint32_t>(slot) * SH::CODE;
#pragma unroll
    for (int i = 0; i < CPR; ++i) {
      const int row = (lane + 32 * i) / CPR, c = lane % CPR;
      const int sw = Q == 4 ? (c ^ ((row >> 1) & 3)) : (c ^ ((row >> 2) & 1));
      const uint32_t dst = st + static_cast<uint32_t>(row * P + 16 * sw);
      // (the last step of a row may be cut short; what then lies in the slot's
      // rest meets zeros of x, and any bits masked to a code are finite)
      const int left = CUT ? static_cast<int>(row_bytes) - fstep * P - 16 * c : 16;
      if (!CUT || Q == 4 || a.calign == 16) {
        if (left > 0) cp_async(dst, cp[i], 16);
      } else {
        if (left > 0) cp_async(dst, cp[i], 8);
        if (left > 8) cp_async(dst + 8, cp[i] + 8, 8);
      }
      cp[i] += P;
    }
    if (fleft == upw || fstep % BS == 0) {  // lane: row `lane` of the next block
      fblk = fblk + 1 == D ? 0 : fblk + 1;
      const uint32_t bl = my_ring + D * SH::CODE + static_cast<uint32_t>(fblk) * SH::BLOCK +
                          static_cast<uint32_t>(lane * SB);
      const int g0 = fstep / BS * (SB / 2);
      // (a row's last block may be cut short: zeros for the groups past its end
      // that its last step still computes)
      const int left = static_cast<int>(nG - g0) * 2;
      auto copy = [&](auto n_tag) {
        constexpr int N = decltype(n_tag)::value;
#pragma unroll
        for (int o = 0; o < SB; o += N)
          if (o < left) {
            cp_async(bl + o, reinterpret_cast<const uint8_t*>(sp + g0) + o, N);
            if constexpr (ASYM)
              cp_async(bl + kRows * SB + o, reinterpret_cast<const uint8_t*>(mp + g0) + o, N);
          } else if constexpr (CUT) {
#pragma unroll
            for (int z = 0; z < N; z += 4) {
              asm volatile("st.shared.u32 [%0], %1;" ::"r"(bl + o + z), "r"(0u) : "memory");
              if constexpr (ASYM)
                asm volatile("st.shared.u32 [%0], %1;" ::"r"(bl + kRows * SB + o + z), "r"(0u)
                             : "memory");
            }
          }
      };
      // an odd number of groups per row: no asynchronous copy is that narrow
      auto copy2 = [&]() {
#pragma unroll
        for (int m = 0; m < (ASYM ? 2 : 1); ++m) {
          const uint16_t* src = (m ? mp : sp) + g0;
          uint32_t v[SB / 4];
#pragma unroll
          for (int j = 0; j < SB / 4; ++j) {
            const uint32_t lo = 4 * j < left ? __ldg(src + 2 * j) : 0u;
            const uint32_t hi = 4 * j + 2 < left ? __ldg(src + 2 * j + 1) : 0u;
            v[j] = lo | hi << 16;
          }
#pragma unroll
          for (int j = 0; j < SB / 4; ++j)
            asm volatile("st.shared.u32 [%0], %1;" ::"r"(bl + m * (kRows * SB) + 4 * j), "r"(v[j])
                         : "memory");
        }
      };
      if (SB == 16 && a.salign == 16) copy(std::integral_constant<int, 16>{});
      else if (a.salign >= 8) copy(std::integral_constant<int, 8>{});
      else if (!CUT || a.salign == 4) copy(std::integral_constant<int, 4>{});
      else if constexpr (CUT) copy2();
    }
    ++fstep;
    if (--fleft == 0) {
      ++ft;
      fetch_tile();
    }
  };

  // ---- stage x: a warp takes one batch row's 256 values at a time, a lane
  // eight (a quad's part of a sub-chunk), stored as pairs (e, e + 4) times
  // 2^-pos; four rows' loads are in flight together, the first four issued
  // before the weight ring's copies.  (Columns past the batch hold whatever
  // was there: an mma's columns do not mix, and theirs are never stored.) ----
  const int xunits = (ns + 1) / 2;  // of 256 values (the last may hold fewer; zeros past k)
  const int xvals =
      CUT ? static_cast<int>(min(static_cast<int64_t>(ns) * kStep, a.k - static_cast<int64_t>(s0) * kStep))
          : ns * kStep;
  const int lgu = xunits >= kWarps ? 4 : 32 - __clz(max(xunits - 1, 0));  // warps per row: 2^lgu
  const int rstep = kWarps >> lgu;  // rows taken side by side
  const int nr0 = warp >> lgu;
  uint4 xv[4];
  auto xload = [&](int ul, int nr) {
    const uint16_t* src = a.x + static_cast<int64_t>(s0) * kStep + ul * 256 + 8 * lane;
    const bool in = ul * 256 + 8 * lane < xvals;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = nr + i * rstep;
      xv[i] = in && r < a.batch
                  ? __ldg(reinterpret_cast<const uint4*>(src + static_cast<int64_t>(r) * a.k))
                  : make_uint4(0u, 0u, 0u, 0u);
    }
  };
  auto xput = [&](int ul, int nr) {
    const int st = 2 * ul + (lane >> 4);  // step of the CTA
    // part p of the sub-chunk is quad p's (q = 4), or quad 0, 2, 1, 3's
    const int sc = (lane >> 2) & 3, p = lane & 3;
    const int t = Q == 4 ? p : ((p >> 1) | ((p & 1) << 1));
    const uint32_t dst0 = xs_a + static_cast<uint32_t>((st * 4 + sc) * (NBLK * 512) + t * 16);
    float* b0 = bsum + (st * SEG + (lane & 15) / (G / 8)) * NBC;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int r = nr + i * rstep;
      const uint32_t wv[4] = {xv[i].x, xv[i].y, xv[i].z, xv[i].w};
      float f[8];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        f[2 * e] = __uint_as_float(wv[e] << 16);
        f[2 * e + 1] = __uint_as_float(wv[e] & 0xFFFF0000u);
      }
      uint32_t pr[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        // code e: pos 0, 4, then 0, 4 after a shift by 8 (q = 4; CUT: 2, 6, 2, 6, x
        // with 2^(2 - pos)); codes 0, 3, then 2, 1 after a shift by 4: pos 8, 6, 8, 6
        // (q = 2; x with 2^(6 - pos))
        constexpr float kMul[2][4] = {{1.f, 0.0625f, 1.f, 0.0625f}, {0.25f, 1.f, 0.25f, 1.f}};
        const float mul = kMul[Q == 4 ? 0 : 1][e];
        const int c = Q == 2 && (e & 1) ? 4 - e : e;
        __half2 hv = __floats2half2_rn(f[c] * mul, f[c + 4] * mul);
        pr[e] = *reinterpret_cast<uint32_t*>(&hv);
        // x as the operand holds it (exactly x from 2^-13 on): the row sum has to
        // meet the codes' product with the same values, or what fp16 rounded off
        // smaller ones would be left over times 2^(q-1)
        const float2 held = __half22float2(hv);
        f[c] = held.x * (1.f / mul);
        f[c + 4] = held.y * (1.f / mul);
      }
      float sum = ((f[0] + f[1]) + (f[2] + f[3])) + ((f[4] + f[5]) + (f[6] + f[7]));
#pragma unroll
      for (int o = 1; o < G / 8; o <<= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      if (st >= ns || r >= a.batch) continue;
      const uint32_t dst = dst0 + static_cast<uint32_t>((r >> 3) * 512 + (r & 7) * 64);
      asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(dst), "r"(pr[0]), "r"(pr[1]),
                   "r"(pr[2]), "r"(pr[3])
                   : "memory");
      // the row-sum term on the mma's scale: times -2^(q-1) as the start
      // value of the symmetric grids, plain for the min
      if (lane % (G / 8) == 0)
        b0[r] = ASYM ? sum * kScale : -static_cast<float>(HALF) * kScale * sum;
    }
  };
  const int ul0 = warp & ((1 << lgu) - 1);
  if (ul0 < xunits) xload(ul0, nr0);
  fetch_tile();
#pragma unroll
  for (int d = 0; d < D - 1; ++d) {
    if (d < total) fetch(d);
    cp_commit();
  }
  for (int ul = ul0; ul < xunits; ul += kWarps)
    for (int nr = nr0; nr < a.batch; nr += 4 * rstep) {
      if (ul != ul0 || nr != nr0) xload(ul, nr);
      xput(ul, nr);
    }
  __syncthreads();
  // every CTA of the cluster has started (long since: the staging lies between)
  if (S > 1) asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");

  float acc[2][NBLK][4];
#pragma unroll
  for (int m = 0; m < 2; ++m)
#pragma unroll
    for (int nb = 0; nb < NBLK; ++nb)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[m][nb][e] = 0.f;

  // RANGE as for the fp16 weight operand of the other kernels: the largest
  // |s| (and |m|) bit patterns; exact per group below if they could matter
  uint32_t smax = 0u, mmax = 0u;
  // byte selectors of the q = 2 exchange
  const uint32_t selA = tq < 2 ? 0x1100u : 0x7766u, selB = tq < 2 ? 0x5544u : 0x3322u;

  // step st of the CTA from code slot `slot` and scale block slot `blk`
  auto compute = [&](int slot, int blk, int st) {
    const uint32_t sb = my_ring + static_cast<uint32_t>(slot) * SH::CODE;
    // scales (mins) of rows gq, gq + 8, gq + 16, gq + 24: SEG of the block's,
    // from SEG x the step's place in it
    constexpr int NW = SEG > 2 ? 2 : 1;
    uint32_t sr[4][NW], mr[4][NW];
#pragma unroll
    for (int h = 0; h < 4; ++h) {
      const uint32_t sa = my_ring + D * SH::CODE + static_cast<uint32_t>(blk) * SH::BLOCK +
                          static_cast<uint32_t>((gq + 8 * h) * SB + (s0 + st) % BS * (2 * SEG));
#pragma unroll
      for (int m = 0; m < (ASYM ? 2 : 1); ++m) {
        uint32_t(&o)[NW] = m ? mr[h] : sr[h];
        const uint32_t ma = sa + m * (kRows * SB);
        if constexpr (SEG == 4) {
          asm volatile("ld.shared.v2.u32 {%0,%1}, [%2];" : "=r"(o[0]), "=r"(o[NW - 1]) : "r"(ma));
        } else if constexpr (SEG == 2) {
          asm volatile("ld.shared.u32 %0, [%1];" : "=r"(o[0]) : "r"(ma));
        } else {
          uint16_t v;
          asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(ma));
          o[0] = v;
        }
      }
#pragma unroll
      for (int i = 0; i < NW; ++i) {
        smax = __vmaxu2(smax, sr[h][i] & 0x7FFF7FFFu);
        if constexpr (ASYM) mmax = __vmaxu2(mmax, mr[h][i] & 0x7FFF7FFFu);
      }
    }
    const uint32_t xa = xs_a + static_cast<uint32_t>(st * SH::XSTEP + lane * 16);
    const float* bs = bsum + st * (SEG * NBC);
    uint32_t w[2][4];  // q = 2: the codes of the chunk's two sub-chunks
    // CUT: the step's own sum, added to the tile's at its end, with row sums and
    // the sub-chunk's mmas added in fp32: no more error than the general kernel's
    // short chains, which took these shapes before (against 64 bits 0.96 of it,
    // the geometric mean of 90 shapes and batches)
    float t[2][CUT ? NBLK : 1][4];
    if constexpr (CUT) {
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int nb = 0; nb < NBLK; ++nb)
#pragma unroll
          for (int e = 0; e < 4; ++e) t[m][nb][e] = 0.f;
    }
#pragma unroll
    for (int seg = 0; seg < SEG; ++seg) {
      float d[2][NBLK][4];
      float2 b[NBLK];
#pragma unroll
      for (int nb = 0; nb < NBLK; ++nb)
        b[nb] = *reinterpret_cast<const float2*>(bs + seg * NBC + 8 * nb + 2 * tq);
#pragma unroll
      for (int i = 0; i < 4 / SEG; ++i) {
        const int sc = seg * (4 / SEG) + i;  // sub-chunk of the step
        if constexpr (Q == 4) {
          ldmatrix4(w[0], sb + static_cast<uint32_t>(lane * P + 16 * (sc ^ ((lane >> 1) & 3))));
        } else if ((sc & 1) == 0) {
          ldmatrix4(w[0], sb + static_cast<uint32_t>(lane * P + 16 * ((sc >> 1) ^ ((lane >> 2) & 1))));
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            const uint32_t own = w[0][h], got = __shfl_xor_sync(0xffffffffu, own, 2);
            w[0][h] = __byte_perm(own, got, selA);
            w[1][h] = __byte_perm(own, got, selB);
          }
        }
        uint4 bv[NBLK];
#pragma unroll
        for (int nb = 0; nb < NBLK; ++nb)
          bv[nb] = lds128(xa + static_cast<uint32_t>((sc * NBLK + nb) * 512));
#pragma unroll
        for (int j = 0; j < 2; ++j) {  // the sub-chunk's two mmas: fields 2j, 2j + 1
          uint32_t f0[4], f1[4];
#pragma unroll
          for (int h = 0; h < 4; ++h) {
            if constexpr (Q == 4) {
              // pos 0 and 4; CUT: 2 and 6, for one more shift (see the top)
              const uint32_t v = CUT ? (j ? w[0][h] >> 6 : w[0][h] << 2) : (j ? w[0][h] >> 8 : w[0][h]);
              f0[h] = v & (CUT ? 0x003C003Cu : 0x000F000Fu);
              f1[h] = v & (CUT ? 0x03C003C0u : 0x00F000F0u);
            } else {
              const uint32_t v = w[sc & 1][h];
              // both bytes of a half hold the same four codes: code 0 at pos 8, 3 at
              // pos 6, and after a shift by 4 code 2 at pos 8, 1 at pos 6
              const uint32_t vs = j ? v >> 4 : v;
              f0[h] = vs & 0x03000300u;
              f1[h] = vs & 0x00C000C0u;
            }
          }
#pragma unroll
          for (int m = 0; m < 2; ++m)
#pragma unroll
            for (int nb = 0; nb < NBLK; ++nb) {
              const uint32_t b0 = j ? bv[nb].z : bv[nb].x, b1 = j ? bv[nb].w : bv[nb].y;
              if (CUT && (i > 0 || j > 0)) {
                float e[4];  // (added here: the tensor core's own sum truncates)
                mma_c(e, f0[2 * m], f0[2 * m + 1], f1[2 * m], f1[2 * m + 1], b0, b1, 0.f, 0.f);
#pragma unroll
                for (int z = 0; z < 4; ++z) d[m][nb][z] += e[z];
              } else if (i == 0 && j == 0)
                mma_c(d[m][nb], f0[2 * m], f0[2 * m + 1], f1[2 * m], f1[2 * m + 1], b0, b1,
                      ASYM || CUT ? 0.f : b[nb].x, ASYM || CUT ? 0.f : b[nb].y);
              else
                mma16816(d[m][nb], f0[2 * m], f0[2 * m + 1], f1[2 * m], f1[2 * m + 1], b0, b1);
            }
        }
      }
      // acc += s d (+ m row sum)
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t sw = sr[h][(seg >> 1) % NW];
        const float s = __half2float(__ushort_as_half(
            static_cast<unsigned short>((seg & 1) ? sw >> 16 : sw & 0xFFFFu)));
        float mn = 0.f;
        if constexpr (ASYM) {
          const uint32_t mw = mr[h][(seg >> 1) % NW];
          mn = __half2float(__ushort_as_half(
              static_cast<unsigned short>((seg & 1) ? mw >> 16 : mw & 0xFFFFu)));
        }
#pragma unroll
        for (int nb = 0; nb < NBLK; ++nb) {
          float* ac = (CUT ? t[h >> 1][nb] : acc[h >> 1][nb]) + 2 * (h & 1);
          const float* dd = d[h >> 1][nb] + 2 * (h & 1);
          ac[0] = fmaf(s, CUT && !ASYM ? dd[0] + b[nb].x : dd[0], ac[0]);
          ac[1] = fmaf(s, CUT && !ASYM ? dd[1] + b[nb].y : dd[1], ac[1]);
          if constexpr (ASYM) {
            ac[0] = fmaf(mn, b[nb].x, ac[0]);
            ac[1] = fmaf(mn, b[nb].y, ac[1]);
          }
        }
      }
    }
    if constexpr (CUT) {
#pragma unroll
      for (int m = 0; m < 2; ++m)
#pragma unroll
        for (int nb = 0; nb < NBLK; ++nb)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[m][nb][e] += t[m][nb][e];
    }
  };

  // ---- passes over up to pass_tiles tiles, each ended by the cluster's sums ----
  int gk = 0, slot = 0, blk = 0;
  for (int t0 = 0; t0 < my_tiles || t0 == 0; t0 += pass_tiles) {
    for (int i = 0; i < a.rounds && t0 + i * ngrp + grp < my_tiles; ++i) {
      for (int u = 0; u < upw; ++u, ++gk) {
        // stage `slot` has landed, and stage slot - 1, read last, is free
        cp_wait<D - 2>();
        __syncwarp();
        if (gk + D - 1 < total) fetch(slot == 0 ? D - 1 : slot - 1);
        cp_commit();
        if (u == 0 || (s0 + u0 + u) % BS == 0) blk = blk + 1 == D ? 0 : blk + 1;
        compute(slot, blk, u0 + u);
        slot = slot + 1 == D ? 0 : slot + 1;
      }
      // this warp's partial of the tile, to the CTAs that own its outputs:
      // column col and rows 8h .. 8h + 7 belong to rank (4h + 2 (col & 1)) S/8
      const int keep = 3 - lgS;
      const uint32_t mine = su32(
          part + ((static_cast<size_t>(rank) * (a.rounds * ngrp) + i * ngrp + grp) * KW + kw) * share);
#pragma unroll
      for (int o = 0; o < 8; ++o) {  // 2h + (col & 1)
        const int h = o >> 1, e = o & 1;
        const uint32_t li = static_cast<uint32_t>(((tq << keep) | (o & ((1 << keep) - 1))) * 8 + gq);
        uint32_t dst;
        asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(dst) : "r"(mine + 4u * li), "r"(o >> keep));
#pragma unroll
        for (int nb = 0; nb < NBLK; ++nb) {
          float& v = acc[h >> 1][nb][2 * (h & 1) + e];
          asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(dst + (static_cast<uint32_t>(nb) * 128u << keep)),
                       "f"(v)
                       : "memory");
          v = 0.f;
        }
      }
    }
    if (S == 1) __syncthreads();
    else cluster.sync();
    // the sums of this CTA's outputs, source CTA by source CTA and warp by warp
    // (warps without steps left zeros)
    const int nt = min(pass_tiles, my_tiles - t0);
    const int keep = 3 - lgS;
    const int64_t sstride = static_cast<int64_t>(a.rounds) * ngrp * KW * share;
    for (int idx = threadIdx.x; idx < nt * share; idx += kThreads) {
      const int j = idx / share, li = idx - j * share;
      const int o = (rank << keep) | ((li >> 3) & ((1 << keep) - 1));
      const int col = 2 * (li >> (3 + keep)) + (o & 1), row = 8 * (o >> 1) + (li & 7);
      const int64_t r = (static_cast<int64_t>(cid) + static_cast<int64_t>(t0 + j) * nclus) * kRows + row;
      if (r >= a.n || col >= a.batch) continue;
      const float* pb = part + static_cast<size_t>(j) * KW * share + li;
      float sum = 0.f;
      for (int c = 0; c < S; ++c, pb += sstride) {
#pragma unroll 4
        for (int w = 0; w < KW; ++w) sum += pb[w * share];
      }
      sum *= 1.f / kScale;
      if (__builtin_expect(!(fabsf(sum) <= 0x1.fffffep127f), 0))
        sum = plain_dot<Q, ASYM, G>(a, r, col);
      a.y[static_cast<int64_t>(col) * a.n + r] = sum;
    }
    // the sums are read before the next pass's partials arrive
    if (t0 + pass_tiles < my_tiles) {
      if (S == 1) __syncthreads();
      else cluster.sync();
    }
  }

  // ---- SSS_FLAG_RANGE ----
  if (a.status != nullptr) {
    const uint32_t s1 = max(smax & 0xFFFFu, smax >> 16), m1 = max(mmax & 0xFFFFu, mmax >> 16);
    bool big;
    if constexpr (!ASYM) {
      // |s| 2^(q-1) 16 >= 65520 exactly when |s| >= the fp16 that 4095 / 2^(q-1) rounds up to
      big = s1 >= static_cast<uint32_t>(__half_as_ushort(__float2half_ru(4095.f / HALF)));
    } else {
      const float top = __half2float(__ushort_as_half(static_cast<unsigned short>(s1))) *
                            static_cast<float>(2 * HALF - 1) +
                        __half2float(__ushort_as_half(static_cast<unsigned short>(m1)));
      big = false;
      if (__any_sync(0xffffffffu, !(top * 16.f < 65520.f))) {  // group by group, this warp's
        for (int j = 0; j < wt; ++j)
          for (int u = 0; u < upw; ++u) {
            const int64_t r =
                (static_cast<int64_t>(cid) + static_cast<int64_t>(grp + j * ngrp) * nclus) * kRows + lane;
            if (r >= a.n) continue;
            const int st = s0 + u0 + u;
            for (int i = 0; i < SEG; ++i) {
              const int64_t gi = static_cast<int64_t>(st) * kStep / G + i;
              if (CUT && gi >= nG) continue;
              const float s = fabsf(__half2float(__ushort_as_half(a.scales[r * nG + gi])));
              const float m = fabsf(__half2float(__ushort_as_half(a.mins[r * nG + gi])));
              big |= (s * static_cast<float>(2 * HALF - 1) + m) * 16.f >= 65520.f;
            }
          }
      }
    }
    if (__any_sync(0xffffffffu, big) && lane == 0) atomicOr(a.status, SSS_FLAG_RANGE);
  }
}

// The most clusters of S CTAs, one CTA per SM, that the device runs at once
// (GPCs of uneven size leave SMs over); 0 if it takes none.
int max_clusters(int lgS) {
  static std::mutex mu;
  static int cache[64][4];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
  std::lock_guard<std::mutex> lock(mu);
  int& c = cache[dev][lgS];
  if (c == 0) {
    auto kern = gemv_cluster_kernel<4, false, 32, 1, 3, false>;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(static_cast<unsigned>(device_sm_count()) / (1u << lgS) * (1u << lgS), 1, 1);
    cfg.blockDim = dim3(kThreads, 1, 1);
    cfg.dynamicSmemBytes = kSmemMax;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 1u << lgS;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    int v = 0;
    if (ensure_smem(kern, kSmemMax) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&v, kern, &cfg) != cudaSuccess || v < 1) {
      (void)cudaGetLastError();
      v = -1;
    }
    c = v;
  }
  return c < 0 ? 0 : c;
}

template <int Q, bool ASYM, int G, int NBLK, int D, bool CUT>
cudaError_t launch_c(ClusterArgs& a, cudaStream_t stream) {
  using SH = Shape<Q, ASYM, G, NBLK, D>;
  // Cluster size and warps per tile of least estimated time in SM cycles: the
  // busiest warp's steps or the SM's (its instruction issue or its share of
  // HBM), whichever is more, the staging of the CTA's x, and the end (a
  // barrier and the sums).
  int best_lgs = -1, best_lgkw = 0, best_rounds = 0, best_cs = 0;
  double best = 1e30;
  for (int lgs = 0; (1 << lgs) <= kMaxCluster; ++lgs) {
    const int S = 1 << lgs;
    if (S > a.nsteps) break;
    const int C = max_clusters(lgs);
    if (C < 1) continue;
    int cs = (a.nsteps + S - 1) / S;
    // whole scale blocks per CTA, unless that leaves one without steps
    const int csb = (cs + SH::BS - 1) / SH::BS * SH::BS;
    if ((S - 1) * csb < a.nsteps) cs = csb;
    if ((S - 1) * cs >= a.nsteps) continue;  // every CTA has steps
    const int tiles = (a.ntiles + std::min(C, a.ntiles) - 1) / std::min(C, a.ntiles);
    for (int lg = 0; (1 << lg) <= kWarps; ++lg) {
      const int kwn = 1 << lg, ngrp = kWarps >> lg;
      if (kwn > 1 && kwn > cs) break;
      const int rounds = (tiles + ngrp - 1) / ngrp;
      int fit = 0;
      while (fit < rounds && SH::bytes(cs, fit + 1) <= kSmemMax) ++fit;
      if (fit == 0) continue;
      const int passes = (rounds + fit - 1) / fit;
      // a step: a warp alone, and the SM's share of issue and HBM
      const double alone = 500.0 + 100.0 * NBLK;
      const double shared = std::max(SH::STAGE / 23.0, 45.0 + 35.0 * NBLK);
      const double busy = static_cast<double>(rounds) * ((cs + kwn - 1) / kwn) * alone;
      const double all = static_cast<double>(tiles) * cs * shared;
      const double items = std::ceil(static_cast<double>((cs + 1) / 2) * a.batch / kWarps);
      const double cost = std::max(busy, all) + 250.0 * items + passes * (S > 1 ? 900.0 : 100.0) +
                          static_cast<double>(tiles) * a.batch * kRows * kwn / kThreads * 6.0;
      if (cost < best) {
        best = cost;
        best_lgs = lgs;
        best_lgkw = lg;
        best_rounds = std::min(rounds, fit);
        best_cs = cs;
      }
    }
  }
  if (best_lgs < 0) return cudaErrorNotSupported;
  a.lgkw = best_lgkw;
  a.rounds = best_rounds;
  a.csteps = best_cs;
  a.wsteps = (best_cs + (1 << best_lgkw) - 1) >> best_lgkw;
  const int S = 1 << best_lgs;
  const int nclus = std::min(max_clusters(best_lgs), a.ntiles);
  auto kern = gemv_cluster_kernel<Q, ASYM, G, NBLK, D, CUT>;
  const size_t smem = SH::bytes(best_cs, best_rounds);
  cudaError_t e = ensure_smem(kern, kSmemMax);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(nclus * S), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = static_cast<unsigned>(S);
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kern, a);
}

template <int Q, bool ASYM, int G>
cudaError_t launch_n(ClusterArgs& a, cudaStream_t stream) {
  // (the min-max ring at 16 columns leaves x no room for a fourth stage)
  constexpr int D = Q == 4 ? 3 : 4, D16 = Q == 2 && !ASYM ? 4 : 3;
  if (a.k % 256 != 0 || a.salign == 2) {
    if (a.batch <= 8) return launch_c<Q, ASYM, G, 1, D, true>(a, stream);
    return launch_c<Q, ASYM, G, 2, D16, true>(a, stream);
  }
  if (a.batch <= 8) return launch_c<Q, ASYM, G, 1, D, false>(a, stream);
  return launch_c<Q, ASYM, G, 2, D16, false>(a, stream);
}

template <int Q, bool ASYM>
cudaError_t launch_g(int g, ClusterArgs& a, cudaStream_t stream) {
  switch (g) {
    case 32: return launch_n<Q, ASYM, 32>(a, stream);
    case 64: return launch_n<Q, ASYM, 64>(a, stream);
    case 128: return launch_n<Q, ASYM, 128>(a, stream);
  }
  return cudaErrorInvalidValue;
}

}  // namespace

// q = 2 and 4, any k; launch_gemv_cluster may still return
// cudaErrorNotSupported (a k whose staged x fits no cluster), without having
// launched anything.  Scale rows of 2-byte alignment come by loads that a warp
// waits for, a block at a time: with groups of 32, long rows, few of them to share
// the wait and little work per row, the general kernel is faster.  Time here over
// there, the geometric mean over n = 32 .. 512 and k = 2080 .. 12320: at batch 2
// 1.06 (q = 2 symmetric), 1.15 (q = 2 min-max), 0.97 (q = 4 symmetric) and 1.12
// (q = 4 min-max), at batch 4 0.95, 1.02, 0.92 and 1.01; k = 1056 and 1568 0.73 to
// 1.00.  The error here is a sixth of the general kernel's, so a tie comes here.
bool gemv_cluster_eligible(const sss_qtensor_t& t, const uint16_t* x, int batch, const float* y) {
  auto al = [](const void* p, size_t b) { return (reinterpret_cast<uintptr_t>(p) % b) == 0; };
  if (t.q == 3 || batch < 2 || batch > 16) return false;
  if (t.k <= 0 || t.n <= 0 || t.k % 32 != 0 || t.k > (int64_t{1} << 24)) return false;
  if (t.n > (int64_t{1} << 30)) return false;
  if (!al(t.codes, 16) || !al(t.scales, 2) || !al(x, 16) || !al(y, 4)) return false;
  if (t.grid == SSS_GRID_ASYM && !al(t.mins, 2)) return false;
  if (t.group == 32 && t.k / 32 % 2 != 0 && batch == 2 && t.n <= 512 && t.k >= 2048 &&
      (t.q == 2 || t.grid == SSS_GRID_ASYM))
    return false;
  return true;
}

cudaError_t launch_gemv_cluster(const sss_qtensor_t& t, const uint16_t* x, int batch, float* y,
                                uint32_t* status, cudaStream_t stream) {
  ClusterArgs a;
  memset(&a, 0, sizeof a);
  a.codes = t.codes;
  a.scales = t.scales;
  a.mins = t.mins;
  a.x = x;
  a.y = y;
  a.n = t.n;
  a.k = t.k;
  a.batch = batch;
  a.ntiles = static_cast<int>((t.n + kRows - 1) / kRows);
  a.nsteps = static_cast<int>((t.k + kStep - 1) / kStep);
  const bool asym = t.grid == SSS_GRID_ASYM;
  uintptr_t bits = reinterpret_cast<uintptr_t>(t.scales) | static_cast<uintptr_t>(t.k / t.group * 2);
  if (asym) bits |= reinterpret_cast<uintptr_t>(t.mins);
  a.salign = bits % 16 == 0 ? 16 : (bits % 8 == 0 ? 8 : (bits % 4 == 0 ? 4 : 2));
  a.calign = t.k * t.q / 8 % 16 == 0 ? 16 : 8;
  // The flag speaks of the fp16 weight operand that k a multiple of 256 is
  // documented to have; other shapes never raised it.
  a.status = t.k % 256 == 0 && bits % 4 == 0 ? status : nullptr;
  if (t.q == 2) return asym ? launch_g<2, true>(t.group, a, stream) : launch_g<2, false>(t.group, a, stream);
  if (t.q == 4) return asym ? launch_g<4, true>(t.group, a, stream) : launch_g<4, false>(t.group, a, stream);
  return cudaErrorNotSupported;
}

}  // namespace sss
