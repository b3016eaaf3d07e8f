// gemm.cu -- prefill GEMM over packed q-bit codes on the 5th-generation
// tensor cores (sm_103a: tcgen05 + tensor memory + TMA).
//
// Y[m][r] = sum_k w^[r][k] X[m][k]; in the prefill phase the matrix products
// set the time (Appendix B.2), and the
// symmetric formats compute only the integer-code GEMM term of the expansion
// in Appendix B.3 (the min-max grid adds the per-block minimum).
//
// Precision: the dequantised weight s*c is rounded to fp16 (<= 2^-11
// relative, where bf16 would give 2^-8 and miss the 1e-3 output gate) and
// the bf16 activations are converted to fp16 (exact for 2^-17 <= |x| <=
// 65504).  tcgen05.mma kind::f16 takes both operands in fp16 and accumulates
// in fp32 in tensor memory.
//
// Structure: persistent CTAs of 18 warps, one per SM, take output tiles of
// 128 weight rows x BN = 64, 128 or 256 tokens in turn (the row tiles may
// belong to up to four matrices that share X, one launch for a fused q/k/v or
// gate/up projection).  A step is two 64-wide k-blocks (128 codes of a row):
//   warp 0     TMA producer: fp16 activation tiles (128B swizzle), packed
//              code tiles of 256 codes; owner of the tensor-memory allocation;
//   warp 1     issues tcgen05.mma (M=128, N=BN, K=16 per instruction, 8 per
//              step) with the weight operand A in tensor memory and the
//              activations B in shared memory, and commits to the step's
//              "empty" barrier;
//   warps 2-17 dequantise in four groups of four that take every fourth step:
//              each thread owns one weight row of the tile (its tensor-memory
//              lane), reads the step's 128 codes of it from shared memory and
//              their scales from global memory, forms fp16 s*c in the k order
//              of X's columns and writes it to the step's A columns of tensor
//              memory (tcgen05.st; shared memory then carries no
//              generic-proxy stores)
//              (a group whose scale lets s*c reach 65520, checked per scale
//              as |s| 2^(q-1) or |s| (2^q - 1) + |m|, raises SSS_FLAG_RANGE);
//              after a tile's last step the same warps drain its fp32
//              accumulator with tcgen05.ld and store Y (for a fixed token, a
//              warp writes 32 consecutive floats).
// Tensor memory (512 columns): 256 columns of fp32 accumulators, then four A
// stages of 64 columns (lane = row, two k-consecutive halves per 32-bit column).
// Where every CTA has one item only (SOLO; up to 128 tokens per tile), its 256 / BN
// accumulators each take a share of the steps and are added in fp32 at the end: the
// tensor core's sums truncate, so the error grows with the length of the chain
// (q = 2, whose weights are exact in fp16: 5120 x 5120 at 256 tokens 5.1e-6 -> 2.4e-6
// against 64 bits, 4096 x 14336 at 17 3.5e-6 -> 7.7e-7).  With no further item to
// run ahead to, the second accumulator would lie idle.
// What bounds it: at BN = 256 the MMAs (1025 cycles a step; 512 per k-block is
// the pipe's rate), 88 % of cuBLAS's burst rate at 2048 tokens with the
// conversion of X (14336 x 4096 q = 4: 140 us; 192 us when a tile's k-blocks
// each brought their own narrow code and scale tiles); at BN <= 128 the TMA
// unit's rows and the way from L2 to the SM (650-750 cycles a step; the MMAs
// need 512 at BN = 128); at few tokens the launch itself.
// Every mbarrier wait is bounded (about one second of global time); on
// expiry the CTA raises SSS_FLAG_TIMEOUT, all roles leave their loops, and
// the tensor memory is still released.
#include <cuda.h>

#include <string.h>

#include <algorithm>
#include <mutex>

#include "act_q8.cuh"

namespace sss {
namespace {

constexpr int kBM = 128;            // weight rows per tile (MMA M)
constexpr int kBK = 64;             // k per stage (128 bytes of fp16)
constexpr int kThreads = 64 + 32 * 16;  // producer, MMA issuer, 16 dequantising warps
constexpr uint64_t kWaitNs = 1000000000ull;  // bounded waits: 1 s

// ---------------------------------------------------------------------------
// PTX wrappers
// ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count)
               : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// whether the phase has completed, without waiting
__device__ __forceinline__ bool mbar_test_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.test_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

// Bounded wait on a phase parity.  Returns false when the wait gave up,
// either on its own time limit or because another role raised *abort.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          volatile int* abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_ns();
  for (uint32_t it = 1;; ++it) {
    if (mbar_try_wait(bar, parity)) return true;
    if ((it & 255u) == 0) {
      if (*abort) return false;
      if (global_ns() - t0 > kWaitNs) {
        *abort = 1;
        return false;
      }
    }
  }
}

// One lane of the (converged) warp.  The producer and issuer loops run warp-wide
// and elect a lane only around the instruction itself: their counters,
// addresses and descriptors then stay in uniform registers.  Run by one lane
// under divergent control flow, each tcgen05 instruction first moves its
// operands there (45 cycles apiece unloaded, about 200 beside the busy
// dequantising warps), and a k-block's issue took longer than its MMAs.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile(
      "{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(p));
  return p != 0;
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
}

__device__ __forceinline__ void tma_load_2d(const CUtensorMap* map, uint64_t* bar, void* dst,
                                            int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1)
      : "memory");
}

// tcgen05 shared-memory matrix descriptor: K-major operand, 128-byte swizzle,
// 8-row swizzle atoms 1024 bytes apart (stride byte offset), descriptor
// version 1 at bit 46.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((saddr & 0x3FFFFu) >> 4);          // start address
  d |= static_cast<uint64_t>(1) << 16;                           // LBO (unused for SW128 K-major)
  d |= static_cast<uint64_t>(1024 >> 4) << 32;                    // SBO: 1024 B
  d |= static_cast<uint64_t>(1) << 46;                           // version
  d |= static_cast<uint64_t>(2) << 61;                           // 128B swizzle
  return d;
}

// Instruction descriptor, kind::f16: D fp32, A and B fp16, both K-major.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N) {
  return (1u << 4)                                    // D format: F32
         | (0u << 7) | (0u << 10)                     // A, B format: F16
         | (static_cast<uint32_t>(N >> 3) << 17)      // N / 8
         | (static_cast<uint32_t>(M >> 4) << 24);     // M / 16
}

// The four MMAs of one 64-wide k-block (K = 16 each) in one block: A from
// tensor memory at a_tmem + 8 kk, B from the swizzled shared tile whose
// descriptor is b_desc + 2 kk (32 bytes further along k; the start-address
// field counts 16-byte units and does not carry), accumulating into d_tmem
// unless first is set (the tile's first k-block starts from zero).
__device__ __forceinline__ void umma_kblock(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc,
                                            uint32_t idesc, uint32_t first) {
  asm volatile(
      "{\n .reg .pred p;\n setp.eq.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%5], %6, %3, 1;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%7], %8, %3, 1;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], [%9], %10, %3, 1;\n}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(first), "r"(a_tmem + 8), "l"(b_desc + 2),
      "r"(a_tmem + 16), "l"(b_desc + 4), "r"(a_tmem + 24), "l"(b_desc + 6)
      : "memory");
}
// 16 consecutive 32-bit columns of the warp's 32 lanes
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16};\n" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]),
      "r"(r[8]), "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]),
      "r"(r[15])
      : "memory");
}
__device__ __forceinline__ void umma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

// W = 16 or 32 consecutive columns, to be waited for
template <int W>
__device__ __forceinline__ void tmem_ld_async(uint32_t taddr, uint32_t (&r)[W]) {
  if constexpr (W == 16) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
  } else {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
        "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
          "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
          "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
          "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
          "=r"(r[31])
        : "r"(taddr));
  }
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&r)[32]) {
  tmem_ld_async<32>(taddr, r);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// ---------------------------------------------------------------------------
// Dequantisation of 32 codes of one row into 16 fp16 pairs.
//
// Pair p holds the two elements whose fields a single shift brings to bit 0
// of the two 16-bit halves of a code word: q = 4: elements 8w + i and
// 8w + i + 4 (p = 4w + i); q = 2, 3: elements 16w + e and 16w + e + 8
// (p = 8w + e).  The k order inside a k-block is free as long as both
// operands use it, so the conversion of X stores its columns in this order
// (x16_kernel) and no byte permutes are needed here: a shift and one LOP3
// per pair, against a mask, a PRMT and an OR in natural order.
// ---------------------------------------------------------------------------

// Words of sub-chunk i (32 codes) of a thread's 128 codes: lo[] (q = 4: 4
// words, else 2) and for q = 3 its high-bit plane word hi.
template <int Q>
struct Codes128 {
  static constexpr int NW = Q == 4 ? 16 : 8;
  uint32_t lo[NW];
  uint32_t hi[Q == 3 ? 4 : 1];
};

// w: the 4q words of 128 consecutive codes as they lie in memory; q = 3
// keeps its planes per group of G codes.
template <int Q>
__device__ __forceinline__ void order_codes(const uint32_t (&w)[4 * Q], int G, Codes128<Q>& c) {
  if constexpr (Q == 3) {
    if (G == 32) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        c.lo[2 * i] = w[3 * i];
        c.lo[2 * i + 1] = w[3 * i + 1];
        c.hi[i] = w[3 * i + 2];
      }
    } else if (G == 64) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int b = 6 * (i >> 1), h = i & 1;
        c.lo[2 * i] = w[b + 2 * h];
        c.lo[2 * i + 1] = w[b + 2 * h + 1];
        c.hi[i] = w[b + 4 + h];
      }
    } else {
#pragma unroll
      for (int i = 0; i < 8; ++i) c.lo[i] = w[i];
#pragma unroll
      for (int i = 0; i < 4; ++i) c.hi[i] = w[8 + i];
    }
  } else {
#pragma unroll
    for (int i = 0; i < 4 * Q; ++i) c.lo[i] = w[i];
  }
}

// (a & b) | c in one LOP3
__device__ __forceinline__ uint32_t and_or(uint32_t a, uint32_t b, uint32_t c) {
  uint32_t r;
  asm("lop3.b32 %0, %1, %2, %3, 0xEA;" : "=r"(r) : "r"(a), "r"(b), "r"(c));
  return r;
}
// fp16 2^(10 - pos) in both halves, for pos = 0, step, 2 step, ... (step 4 for
// q = 4, else 2)
constexpr int kMagics = 5;

// the high-plane bits of elements 16w .. 16w + 15 (w = half of the plane
// word) spread to every other bit: element 16w + e at bit 2e (e < 8) and
// element 16w + 8 + e at bit 16 + 2e
__device__ __forceinline__ uint32_t spread_high(uint32_t plane, int w) {
  uint32_t x = __byte_perm(plane, 0u, w ? 0x4342u : 0x4140u);
  x = (x | (x << 4)) & 0x0F0F0F0Fu;
  x = (x | (x << 2)) & 0x33333333u;
  x = (x | (x << 1)) & 0x55555555u;
  return x;
}

// The fp16 pairs of sub-chunk i: RN16(s c), or RN16(s u + m) for ASYM.  A
// field u at bit pos of a half, OR-ed into the mantissa of 2^(10 - pos), is
// the fp16 value 2^(10 - pos) + u: it needs no shift of its own while it
// ends below bit 10 (q = 4: pos 0, 4; q = 2: 0 .. 8; q = 3: 0 .. 6 with its
// high bit), so one shift per word serves half of its fields.
// The magic words come in registers (mg, from kernel arguments): as literals
// the compiler splits the mask and the OR, or moves the literal into a
// register each time (208 ALU instructions per 128 codes, 2 issue cycles
// each, against 64 LOP3 and 16 shifts).
template <int Q, bool ASYM>
__device__ __forceinline__ void dequant32(const Codes128<Q>& c, int i, __half2 s2, __half2 m2,
                                          const uint32_t (&mg)[kMagics],
                                          uint32_t (&out)[16]) {
  constexpr int PW = Q == 4 ? 4 : 8;                   // pairs per word
  constexpr int DIRECT = Q == 4 ? 2 : (Q == 2 ? 5 : 4);  // fields taken before the shift
  constexpr int BITS = Q == 4 ? 4 : 2;                 // distance of the fields
#pragma unroll
  for (int w = 0; w < 16 / PW; ++w) {
    const uint32_t v0 = c.lo[i * (16 / PW) + w], v1 = v0 >> (DIRECT * BITS);
    uint32_t h0 = 0u, h1 = 0u;
    if constexpr (Q == 3) {
      const uint32_t hs = spread_high(c.hi[i], w);
      h0 = hs << 2;
      h1 = hs >> (DIRECT * BITS - 2);
    }
#pragma unroll
    for (int e = 0; e < PW; ++e) {
      const int pos = BITS * (e < DIRECT ? e : e - DIRECT);
      const uint32_t field = ((1u << BITS) - 1u) << pos;
      uint32_t mag = and_or(e < DIRECT ? v0 : v1, field | (field << 16), mg[pos / BITS]);
      if constexpr (Q == 3) {
        const uint32_t hb = 4u << pos;
        mag = and_or(e < DIRECT ? h0 : h1, hb | (hb << 16), mag);
      }
      // minus 2^(10 - pos) (+ 2^(q-1) for symmetric codes): exact
      __half2 hv = *reinterpret_cast<const __half2*>(&mag);
      const __half2 bias =
          __float2half2_rn(static_cast<float>((1 << (10 - pos)) + (ASYM ? 0 : 1 << (Q - 1))));
      hv = __hsub2(hv, bias);                             // c (or u) exactly
      hv = ASYM ? __hfma2(hv, s2, m2) : __hmul2(hv, s2);  // RN16(s*c) / RN16(s*u+m)
      out[PW * w + e] = *reinterpret_cast<const uint32_t*>(&hv);
    }
  }
}

// One weight matrix of a call (several share X, e.g. a fused q/k/v
// projection): its row tiles are tiles tile0 .. tile0 + ceil(n / 128) - 1 of
// the grid's x dimension.
struct GemmJob {
  const uint8_t* codes;
  const uint16_t* scales;
  const uint16_t* mins;
  float* y;  // [m][n]
  int64_t n;
  int tile0;
};
struct GemmArgs {
  GemmJob job[kMaxGemmJobs];
  int njobs;
  uint32_t* status;
  int64_t m, k;
  int G;
  uint32_t magic[kMagics];  // dequant32's magic words
  int vec;    // the scales (and mins) of 128 codes can be loaded as one vector
  int stall;  // test hook: the first stage's weight tile is never announced
  // split K: CTA z of nsplit takes k-blocks [z * chunk, ...) and leaves its
  // fp32 tile in part + z * m * np (row tile t at rows 128 t .. 128 t + 127
  // of np = 128 x all row tiles); the last of a tile's splits to finish
  // (counted in cnt, zero on entry) sums them in split order into y
  int nsplit;
  int chunk;  // k-blocks per split, a multiple of kWK
  int rt, mt, items;  // row tiles, token tiles, rt x mt x nsplit
  int64_t np;
  float* part;
  int* cnt;
};

// The activation tile map, and per matrix its code tile map (used with CT).
struct GemmMaps {
  CUtensorMap x;
  CUtensorMap c[kMaxGemmJobs];
};

// A thread owns one weight row and takes 128 codes (two k-blocks) of it at a
// time; a code tile is 128 rows x 256 codes (kWK k-blocks, 32q bytes a row).
// Code tiles this wide matter: the TMA unit moves about one box row per 1.7
// cycles whatever the row's length, so a tile per k-block (32-byte rows, and
// as many 16-byte rows of scales) cost as much as the activation tile and
// set the pace: 640 cycles per k-block at 128 tokens with nothing else to do.
constexpr int kWK = 4;      // k-blocks per code tile
constexpr int kAStages = 4; // A operand steps (two k-blocks) in tensor memory
// A barrier tells a wait for one phase from the next by its parity alone, so
// whoever waits on one has to wait for every phase in turn.  The dequantising
// groups take every fourth step and every other code tile: the A stages are a
// multiple of four and the code tiles an even number, which gives each group
// stages of its own.  The A stages go by step number, of which an item of an odd
// number of steps leaves one out.  Four activation stages (JOINT) go by it too, so
// that a step has one stage for both operands.  Three go step after step and are
// freed by the A stages' barriers: the producer looks at every step's in turn, and
// runs no further ahead than an A stage comes round again (two steps where every
// other number is left out).  (Barriers of their own took a second commit per
// step, 2.8 % of a 256-token tile; the look-ahead rule for four stages as well 15 %
// of down_proj at 512 tokens, where the producer sets the pace.)

// Shared memory: XS activation tiles (1024-aligned for the 128-byte
// swizzle), then with CT the code tiles, then the barriers.
template <int BN, int Q, bool CT, bool SOLO>
struct Smem {
  static constexpr int XS = BN == 256 ? 3 : 4;               // activation stages (steps)
  static constexpr int WS = BN == 256 ? 2 : 4;               // code tiles in flight
  static constexpr int X_BYTES = BN * kBK * 2;               // one k-block: 8, 16 or 32 KB
  static constexpr int W_BYTES = CT ? kBM * 32 * Q : 0;
  static constexpr int W_OFF = XS * 2 * X_BYTES;
  static constexpr int BAR_OFF = W_OFF + WS * W_BYTES;
  static constexpr bool JOINT = XS == kAStages;              // one stage for X and A
  static constexpr int NB = BN == 256 || SOLO ? 1 : 2;       // accumulators, item by item
  static constexpr int PARTS = SOLO ? 256 / BN : 1;          // accumulators of an item
  static constexpr int NBAR = XS + 2 * kAStages + 2 * WS + 2 * NB + 1;
  static constexpr int TOTAL = BAR_OFF + NBAR * 8 + 16 + 1024;  // + align slack
  static constexpr int A_COL = 256;               // first A-stage column in tensor memory
  static_assert(kAStages == 4 && WS % 2 == 0 && XS <= kAStages, "see kAStages");
  static_assert(TOTAL <= 227 * 1024, "shared memory per CTA");
  static_assert(NB * PARTS * BN <= A_COL && A_COL + 64 * kAStages <= 512, "tensor memory");
};
constexpr int kTmemCols = 512;  // one CTA per SM

// The 4q words of codes of tile row `row`, half `h` (128 codes) of a code
// tile in shared memory.  The tile is stored with the swizzle of its row
// length (q = 4: 128 bytes, chunk ^ (row & 7); q = 2: 64 bytes, chunk ^
// ((row >> 1) & 3)), so a quarter-warp's 16-byte loads fall in distinct
// banks; the 96-byte rows of q = 3 are unswizzled (two-way conflicts).
template <int Q>
__device__ __forceinline__ void load_tile_codes(uint32_t tile, int row, int h,
                                                uint32_t (&w)[4 * Q]) {
  const uint32_t base = tile + static_cast<uint32_t>(row * 32 * Q);
  const uint32_t sw = Q == 4 ? (row & 7) : (Q == 2 ? ((row >> 1) & 3) : 0);
#pragma unroll
  for (int c = 0; c < Q; ++c) {
    const uint32_t a = base + 16u * (static_cast<uint32_t>(Q * h + c) ^ sw);
    asm volatile("ld.shared.v4.u32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(w[4 * c]), "=r"(w[4 * c + 1]), "=r"(w[4 * c + 2]), "=r"(w[4 * c + 3])
                 : "r"(a));
  }
}

// The fp16 scales (or mins) of the four 32-code sub-chunks of 128 codes
// whose first group is gi, as u16 pairs; groups past the row's nG read as 0.
__device__ __forceinline__ uint2 load_scales(const uint16_t* __restrict__ row, int64_t gi,
                                             int64_t nG, int G, bool vec) {
  if (G == 32) {
    if (vec) return __ldg(reinterpret_cast<const uint2*>(row + gi));
    uint32_t v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = gi + i < nG ? __ldg(row + gi + i) : 0u;
    return make_uint2(v[0] | (v[1] << 16), v[2] | (v[3] << 16));
  }
  uint32_t a, b;
  if (G == 64) {
    if (vec) {
      const uint32_t v = __ldg(reinterpret_cast<const uint32_t*>(row + gi));
      a = v & 0xFFFFu;
      b = v >> 16;
    } else {
      a = __ldg(row + gi);
      b = gi + 1 < nG ? __ldg(row + gi + 1) : 0u;
    }
  } else {
    a = b = __ldg(row + gi);
  }
  return make_uint2(a | (a << 16), b | (b << 16));
}
__device__ __forceinline__ uint16_t scale_of(const uint2& v, int i) {
  const uint32_t w = (i & 2) ? v.y : v.x;
  return static_cast<uint16_t>((i & 1) ? (w >> 16) : (w & 0xFFFFu));
}

// What an output tile (and K split) of the launch's item list is: items run
// over the row tiles of all matrices first, then token tiles, then splits.
struct Item {
  int jb;               // matrix
  int tx, ty, z;        // row tile (of all matrices), token tile, split
  int n0, m0;           // first row (in its matrix) and token
  int kb_base, nkb;     // its k-blocks: kb_base + kb for kb = 0 .. nkb - 1
  int nsteps;           // of two k-blocks (the last may hold one)
};
__device__ __forceinline__ Item item_of(const GemmArgs& a, int it, int BN) {
  Item w;
  w.tx = it % a.rt;
  const int rest = it / a.rt;
  w.ty = rest % a.mt;
  w.z = rest / a.mt;
  w.jb = 0;
  while (w.jb + 1 < a.njobs && w.tx >= a.job[w.jb + 1].tile0) ++w.jb;
  w.n0 = (w.tx - a.job[w.jb].tile0) * kBM;
  w.m0 = w.ty * BN;
  w.kb_base = w.z * a.chunk;
  w.nkb = min(static_cast<int>(a.k / kBK) - w.kb_base, a.chunk);
  w.nsteps = (w.nkb + 1) / 2;
  return w;
}

// The end of a K split's item, by the 512 dequantising threads: the tile's last
// split to arrive sums the partials in split order (z = 0, 1, ...: the same
// order whichever split is last) into y and leaves the counter at zero.
// Returns false, to every thread, when some thread's ok is false.
__device__ __forceinline__ bool sum_splits(const GemmArgs& a, const Item& e, int BN, bool ok,
                                        volatile int* last) {
  __threadfence();  // this CTA's partial tile, device-wide
  uint32_t bad;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 q, %1, 0;\n bar.red.or.pred p, 1, 512, q;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(bad)
      : "r"(ok ? 0u : 1u)
      : "memory");
  if (bad) return false;
  int* cnt = a.cnt + e.ty * a.rt + e.tx;
  if (threadIdx.x == 64) *last = atomicAdd(cnt, 1) == a.nsplit - 1;
  asm volatile("bar.sync 1, 512;" ::: "memory");
  if (!*last) return true;
  __threadfence();
  // 4 consecutive rows per element (n % 4 == 0, y and the partials 16-byte
  // aligned); four elements per thread at a time, so their loads of a split
  // are in flight together
  const GemmJob& job = a.job[e.jb];
  constexpr int kV = kBM / 4;  // float4 per token of the tile
  constexpr int kE = 4;
  const int64_t mn = a.m * a.np;
  const int64_t g0 = static_cast<int64_t>(e.tx) * kBM;
#pragma unroll 1
  for (int e0 = threadIdx.x - 64; e0 < kV * BN; e0 += kE * 512) {
    float4 acc[kE];
    int64_t off[kE];
    bool in[kE];
#pragma unroll
    for (int j = 0; j < kE; ++j) {
      const int el = e0 + j * 512;
      const int64_t mm = e.m0 + el / kV, rr = static_cast<int64_t>(e.n0) + 4 * (el % kV);
      in[j] = el < kV * BN && mm < a.m && rr < job.n;
      off[j] = in[j] ? mm * a.np + g0 + 4 * (el % kV) : 0;
      acc[j] = in[j] ? __ldcg(reinterpret_cast<const float4*>(a.part + off[j]))
                     : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    for (int z = 1; z < a.nsplit; ++z) {
      float4 v[kE];
#pragma unroll
      for (int j = 0; j < kE; ++j)
        v[j] = in[j] ? __ldcg(reinterpret_cast<const float4*>(a.part + z * mn + off[j]))
                     : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int j = 0; j < kE; ++j) {
        acc[j].x += v[j].x; acc[j].y += v[j].y; acc[j].z += v[j].z; acc[j].w += v[j].w;
      }
    }
#pragma unroll
    for (int j = 0; j < kE; ++j) {
      const int el = e0 + j * 512;
      if (in[j])
        *reinterpret_cast<float4*>(job.y + static_cast<int64_t>(e.m0 + el / kV) * job.n + e.n0 +
                                   4 * (el % kV)) = acc[j];
    }
  }
  if (threadIdx.x == 64) *cnt = 0;
  return true;
}

// Persistent: one CTA per SM takes items blockIdx.x, + gridDim.x, ...  The
// steps of all its items are numbered through, each item starting at an even
// number, so that step P uses A stage P % 4, is dequantised by group P % 4 and
// lies in code tile P / 2.  While an item's last MMAs run and its accumulator
// is drained, the next item's tiles load and its first steps dequantise; with
// up to 128 tokens per tile there are two accumulators, and the next item's
// MMAs run through the drain as well.  (One CTA per item spent about 9000 of
// 27000 cycles at 128 tokens and k = 4096 on its start and end.)
//
// SOLO: no more items than CTAs; the loops over items then end with the first.
//
// CT: the packed codes arrive by TMA (rows of k q / 8 bytes, a multiple of
// 16); otherwise (q = 3 with k an odd multiple of 64) each dequantising
// thread loads its own from global memory one step ahead.
template <int Q, bool ASYM, int BN, bool CT, bool SOLO>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ GemmMaps maps, const __grid_constant__ GemmArgs a) {
  using S = Smem<BN, Q, CT, SOLO>;
  constexpr int XS = S::XS, WS = S::WS, NB = S::NB, PARTS = S::PARTS;
  extern __shared__ unsigned char smem_raw[];
  // 1024-byte alignment for the swizzle atoms
  unsigned char* smem = reinterpret_cast<unsigned char*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint64_t* full_x = reinterpret_cast<uint64_t*>(smem + S::BAR_OFF);
  uint64_t* full_w = full_x + XS;
  uint64_t* empty_w = full_w + WS;
  uint64_t* full_a = empty_w + WS;
  uint64_t* empty = full_a + kAStages;  // of both operands of a step
  uint64_t* done = empty + kAStages;    // an item's MMAs have completed
  uint64_t* acc_free = done + NB;       // its accumulator has been read
  uint64_t* retired = acc_free + NB;    // used when a wait has run out
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(retired + 1);
  volatile int* abort = reinterpret_cast<volatile int*>(tmem_slot + 1);
  volatile int* last = abort + 1;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;

  if (threadIdx.x == 0) {
    for (int s = 0; s < XS; ++s) mbar_init(&full_x[s], 1);
    for (int s = 0; s < kAStages; ++s) {
      mbar_init(&full_a[s], 4);  // the four warps that cover the 128 rows
      mbar_init(&empty[s], 1);
    }
    for (int s = 0; s < WS; ++s) {
      mbar_init(&full_w[s], 1);
      mbar_init(&empty_w[s], 8);  // the warps of its two 128-code halves
    }
    for (int s = 0; s < NB; ++s) {
      mbar_init(&done[s], 1);
      mbar_init(&acc_free[s], 16);
    }
    mbar_init(retired, 1);
    *abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Launched as a programmatic dependent launch of x16_kernel, which releases
  // it only once everything before that kernel has completed.  So the packed
  // weights and scales may be read at once; what x16_kernel writes (X, the
  // split counters), and every write of this kernel, waits for it: the
  // producer before its first activation tile, the other warps before their
  // first epilogue.
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");

  if (warp == 0) {
    // ---------------- TMA producer: activation and code tiles ----------------
    int sx = 0, xn = 0;      // activation stage, and how many steps were issued
    int sw = 0, wn = 0;      // code stage, and how many tiles were issued
    uint32_t phw = 0;
    uint32_t usedx = 0;      // bit s: the parity of activation stage s's next use
    // unless JOINT
    uint32_t used = 0;       // bit s: the parity of A stage s's next use
    uint32_t hist = 0;       // the last steps' A stages and parities, 4 bits each
    uint32_t near = 0;       // bit i: step number P + p - 1 - i is a step, i = 0 .. 3
    int seen = 0;            // steps whose MMAs are known to have completed
    int P = 0;
    bool ok = true;
    for (int it = blockIdx.x; it < a.items && ok; it += gridDim.x) {
      const Item w = item_of(a, it, BN);
      const int nw = CT ? (w.nsteps + 1) / 2 : 0;
      // code tile i of the item: 32q bytes (256 codes) of each row
      auto put_w = [&](int i) -> bool {
        const bool freed = mbar_wait(&empty_w[sw], phw ^ 1u, abort);
        if (!__all_sync(0xffffffffu, freed)) return false;
        if (elect_one()) {
          mbar_arrive_expect_tx(&full_w[sw], S::W_BYTES);
          tma_load_2d(&maps.c[w.jb], &full_w[sw], smem + S::W_OFF + sw * S::W_BYTES,
                      (w.kb_base + i * kWK) * 8 * Q, w.n0);
        }
        __syncwarp();
        if (++sw == WS) {
          sw = 0;
          phw ^= 1u;
        }
        ++wn;
        return true;
      };
      // code tiles run one ahead of the activations: their codes have the
      // dequantisation before them
      ok = nw == 0 || put_w(0);
      if (xn == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
      for (int p = 0; p < w.nsteps && ok; ++p) {
        if (p % 2 == 0 && p / 2 + 1 < nw && !put_w(p / 2 + 1)) {
          ok = false;
          break;
        }
        if constexpr (S::JOINT) {
          // the stage is free once the MMAs that used it last have completed
          const bool freed = mbar_wait(&empty[sx], ((usedx >> sx) & 1u) ^ 1u, abort);
          ok = __all_sync(0xffffffffu, freed);
        } else {
          // the stage is free once the MMAs of XS steps ago have completed; and
          // the last step of this A stage has to be seen before this one can
          // complete the barrier's next phase
          const int ahead = (near & 8u) ? min(XS, __popc(near)) : XS;
          for (; xn - seen >= ahead && ok; ++seen) {
            const uint32_t h = hist >> (4 * (xn - seen - 1));
            const bool freed = mbar_wait(&empty[(h >> 1) & 3u], h & 1u, abort);
            ok = __all_sync(0xffffffffu, freed);
          }
        }
        if (!ok) break;
        if (elect_one()) {
          // (a box past the end of k reads zeros)
          unsigned char* dst = smem + sx * 2 * S::X_BYTES;
          mbar_arrive_expect_tx(&full_x[sx], 2 * S::X_BYTES);
          tma_load_2d(&maps.x, &full_x[sx], dst, (w.kb_base + 2 * p) * kBK,
                      w.m0);
          tma_load_2d(&maps.x, &full_x[sx], dst + S::X_BYTES, (w.kb_base + 2 * p + 1) * kBK,
                      w.m0);
        }
        __syncwarp();
        usedx ^= 1u << sx;
        if (++sx == XS) sx = 0;
        ++xn;
        if constexpr (!S::JOINT) {
          const uint32_t sa = static_cast<uint32_t>(P + p) & 3u;
          hist = (hist << 4) | (sa << 1) | ((used >> sa) & 1u);
          used ^= 1u << sa;
          near = ((near << 1) | 1u) & 15u;
        }
      }
      if (w.nsteps & 1) {  // the step number left out
        if (S::JOINT) sx = (sx + 1) & 3;
        near = (near << 1) & 15u;
      }
      P += (w.nsteps + 1) & ~1;
      if constexpr (SOLO) break;
    }
    if (*abort) {
      // let this CTA's copies still in flight land before the CTA exits (of a
      // stage never used, the phase before its first counts as completed)
      int drain = 0;
      for (int s = 0; s < XS; ++s)
        (void)mbar_wait(&full_x[s], ((usedx >> s) & 1u) ^ 1u, &drain);
      for (int i = max(0, wn - WS); i < wn; ++i)
        (void)mbar_wait(&full_w[i % WS], static_cast<uint32_t>(i / WS) & 1u, &drain);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    // The step loop is unrolled over the A stages, so that their barriers and
    // columns are offsets of uniform registers (the reduction puts the
    // tensor-memory base into one), and the next step's barriers are tried
    // while this step's MMAs issue.
    constexpr uint32_t idesc = make_idesc(kBM, BN);
    const uint32_t tm = __reduce_or_sync(0xffffffffu, tmem);
    const uint64_t bdesc0 = sw128_desc(smem_u32(smem));
    constexpr uint64_t bstep = static_cast<uint64_t>(S::X_BYTES >> 4);
    bool go = true;
    int sx = 0, P = 0, n = 0;  // activation stage, first step and number of the item
    uint32_t phx = 0, used = 0;
    for (int it = blockIdx.x; it < a.items && go; it += gridDim.x, ++n) {
      const Item w = item_of(a, it, BN);
      const int buf = n % NB;
      uint32_t acc = tm + static_cast<uint32_t>(buf * BN);
      const int share = (w.nsteps + PARTS - 1) / PARTS;  // steps per accumulator
      int turn = P;                                      // the next one's first
      // the accumulator's previous item has been drained
      const bool fr = mbar_wait(&acc_free[buf], (static_cast<uint32_t>(n / NB) & 1u) ^ 1u, abort);
      if (!__all_sync(0xffffffffu, fr)) break;
      tc_fence_after();
      bool there = false;
      const int end = P + w.nsteps;
      for (int P0 = P & ~3; P0 < end && go; P0 += kAStages) {
#pragma unroll
        for (int s = 0; s < kAStages; ++s) {
          if (P0 + s < P || P0 + s >= end || !go) continue;
          if (!there) {
            bool t = mbar_wait(&full_a[s], (used >> s) & 1u, abort);
            t = t && mbar_wait(&full_x[S::JOINT ? s : sx], S::JOINT ? (used >> s) & 1u : phx, abort);
            if (!__all_sync(0xffffffffu, t)) {
              go = false;
              continue;
            }
          }
          used ^= 1u << s;
          tc_fence_after();
          const uint64_t bd = bdesc0 + 2 * bstep * (S::JOINT ? s : sx);
          if (!S::JOINT && ++sx == XS) {
            sx = 0;
            phx ^= 1u;
          }
          constexpr int kNext[4] = {1, 2, 3, 0};
          const bool fresh = P0 + s == turn;
          if (PARTS > 1 && fresh) {
            acc += turn == P ? 0u : BN;
            turn += share;
          }
          const bool next = mbar_test_wait(&full_a[kNext[s]], (used >> kNext[s]) & 1u) &&
                            mbar_test_wait(&full_x[S::JOINT ? kNext[s] : sx],
                                           S::JOINT ? (used >> kNext[s]) & 1u : phx);
          if (elect_one()) {
            const uint32_t ta = tm + static_cast<uint32_t>(S::A_COL + 64 * s);
            umma_kblock(acc, ta, bd, idesc, fresh ? 1u : 0u);
            if (2 * (P0 + s - P) + 1 < w.nkb) umma_kblock(acc, ta + 32, bd + bstep, idesc, 0u);
            umma_commit(&empty[s]);  // frees both operands' stages once these MMAs complete
          }
          there = __all_sync(0xffffffffu, next);
        }
      }
      if (elect_one()) umma_commit(&done[buf]);
      __syncwarp();
      P += (w.nsteps + 1) & ~1;
      if constexpr (SOLO) break;
    }
    if (*abort) {  // MMAs still in flight must retire before the CTA's memory goes
      int drain = 0;
      if (elect_one()) umma_commit(retired);
      __syncwarp();
      (void)mbar_wait(retired, 0u, &drain);
    }
  } else {
    // ---------------- dequantise, and the epilogues ----------------
    // a warp may touch tensor-memory lanes 32*(warp % 4) .. +31 only, so
    // thread (warp, lane) owns tile row 32*(warp % 4) + lane; the dequant
    // warps w = warp - 2 form four groups of four (w >> 2), each covering
    // the 128 rows once: group g takes the 128-code steps P with P % 4 = g
    const int quad = warp & 3;
    const int row_i = 32 * quad + lane;
    const int slot = (warp - 2) >> 2;
    const uint32_t lane_base = tmem + (static_cast<uint32_t>(32 * quad) << 16);
    const int lg = a.G == 32 ? 5 : (a.G == 64 ? 6 : 7);
    const int64_t nG = a.k >> lg;
    bool big = false;  // a group whose s*c may leave the fp16 range
    __half2 smax = __float2half2_rn(0.f);  // symmetric grids: the largest |s| seen
    bool ok = true;
    uint32_t mg[kMagics];
#pragma unroll
    for (int i = 0; i < kMagics; ++i) mg[i] = a.magic[i];
    uint32_t used = 0;  // parity of this group's A stage
    // the item at hand and this thread's row of it
    Item w = {};
    int P = 0;           // the item's first step
    const uint16_t *srow = nullptr, *mrow = nullptr;
    bool rok = false;
    uint2 sv_n = make_uint2(0u, 0u), mv_n = make_uint2(0u, 0u);
    uint32_t wn[CT ? 1 : 4 * Q];
    // the scales (and without CT the codes) of the item's step p, one of this
    // group's steps ahead (codes: rows are 8-byte aligned; the last step may
    // hold one k-block only)
    auto fetch = [&](int p) {
      if (p >= w.nsteps || !rok) return;
      const int64_t gi = (static_cast<int64_t>(w.kb_base) * kBK + 128 * static_cast<int64_t>(p)) >> lg;
      sv_n = load_scales(srow, gi, nG, a.G, a.vec != 0);
      if constexpr (ASYM) mv_n = load_scales(mrow, gi, nG, a.G, a.vec != 0);
      if constexpr (!CT) {
        const uint8_t* src = a.job[w.jb].codes + (static_cast<int64_t>(w.n0) + row_i) * (a.k * Q / 8) +
                             (static_cast<int64_t>(w.kb_base) + 2 * static_cast<int64_t>(p)) * (8 * Q);
        const int words = 2 * p + 1 < w.nkb ? 4 * Q : 2 * Q;
#pragma unroll
        for (int i = 0; i < 2 * Q; ++i) {
          const uint2 v = 2 * i < words ? __ldcs(reinterpret_cast<const uint2*>(src) + i)
                                        : make_uint2(0u, 0u);
          wn[2 * i] = v.x;
          wn[2 * i + 1] = v.y;
        }
      }
    };
    auto start_item = [&](int it) {
      w = item_of(a, it, BN);
      const GemmJob& job = a.job[w.jb];
      const int64_t r = static_cast<int64_t>(w.n0) + row_i;
      rok = r < job.n;
      srow = job.scales + (rok ? r : 0) * nG;
      if constexpr (ASYM) mrow = job.mins + (rok ? r : 0) * nG;
      if (!rok) {
        sv_n = mv_n = make_uint2(0u, 0u);
        if constexpr (!CT) {
#pragma unroll
          for (int i = 0; i < 4 * Q; ++i) wn[i] = 0u;
        }
      }
      fetch((slot - P) & 3);
    };
    // dequantise the item's step p (p = nsteps, past the end of an item of an
    // odd number of steps: only its half of the code tile is handed back)
    auto do_step = [&](int p, bool first) {
      const uint2 sv = sv_n, mv = mv_n;
      Codes128<Q> codes;
      {
        uint32_t wv[4 * Q];
        if constexpr (CT) {
          const int t = (P + p) >> 1;  // code tile
          const int ws = t % WS;
          const bool landed = mbar_wait(&full_w[ws], static_cast<uint32_t>(t / WS) & 1u, abort);
          if (!__all_sync(0xffffffffu, landed)) {
            ok = false;
            return;
          }
          load_tile_codes<Q>(smem_u32(smem) + S::W_OFF + ws * S::W_BYTES, row_i, p & 1, wv);
        } else {
#pragma unroll
          for (int i = 0; i < 4 * Q; ++i) wv[i] = wn[i];
        }
        order_codes<Q>(wv, a.G, codes);
      }
      // hands the code tile back: after the codes have been used, since an
      // arrive right behind the loads lets the TMA overwrite rows whose loads
      // are still in flight
      auto release_w = [&]() {
        if constexpr (CT) {
          if (lane == 0) mbar_arrive(&empty_w[((P + p) >> 1) % WS]);
        }
      };
      if (p >= w.nsteps) {  // (no codes were used: nothing to overwrite)
        release_w();
        return;
      }
      fetch(p + 4);
      if constexpr (!ASYM)
        smax = __hmax2(smax, __hmax2(__habs2(*reinterpret_cast<const __half2*>(&sv.x)),
                                     __habs2(*reinterpret_cast<const __half2*>(&sv.y))));
      // (the second k-block of a tile's odd last step is not multiplied)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const __half sh = __ushort_as_half(scale_of(sv, i));
        const __half2 s2 = __halves2half2(sh, sh);
        __half2 m2 = __float2half2_rn(0.f);
        if constexpr (ASYM) {
          const __half mh = __ushort_as_half(scale_of(mv, i));
          m2 = __halves2half2(mh, mh);
          big |= fabsf(__half2float(sh)) * static_cast<float>((1 << Q) - 1) +
                     fabsf(__half2float(mh)) >= 65520.f;
        }
        uint32_t out[16];
        dequant32<Q, ASYM>(codes, i, s2, m2, mg, out);
        if (i == 0) {
          // warp-uniform, since the tensor-memory stores are .sync.aligned:
          // the MMAs that read this stage have completed
          const bool freed = mbar_wait(&empty[slot], used ^ 1u, abort);
          if (!__all_sync(0xffffffffu, freed)) {
            ok = false;
            return;
          }
          used ^= 1u;
          tc_fence_after();
        }
        tmem_st16(lane_base + static_cast<uint32_t>(S::A_COL + 64 * slot + 16 * i), out);
      }
      // the stores, then the arrive the MMA issuer waits on
      asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
      tc_fence_before();
      __syncwarp();
      // (sss_test_set_stall: warp 2 leaves the first stage one arrive short,
      // so the MMA issuer's wait for it runs out)
      if (lane == 0 && !(a.stall && first && p == 0 && warp == 2)) mbar_arrive(&full_a[slot]);
      release_w();
    };

    int n = 0;
    bool begun = false;  // the item's first step of this group is done
    if (static_cast<int>(blockIdx.x) < a.items) start_item(blockIdx.x);
    for (int it = blockIdx.x; it < a.items && ok; it += gridDim.x, ++n) {
      const int pad = (w.nsteps + 1) & ~1;
      for (int p = ((slot - P) & 3) + (begun ? 4 : 0); p < pad && ok; p += 4) do_step(p, n == 0);
      begun = false;
      if (!SOLO && ok && it + static_cast<int>(gridDim.x) < a.items) {
        P += pad;
        start_item(it + gridDim.x);
        const int p = (slot - P) & 3;
        if (p < ((w.nsteps + 1) & ~1)) {
          do_step(p, false);
          begun = true;
        }
      }
      // ---- epilogue of item e = it: a warp may read tensor-memory lanes
      // 32*(warp % 4) .. +31; the four groups take alternate sets of 32 columns
      if (n == 0) asm volatile("griddepcontrol.wait;" ::: "memory");
      const int buf = n % NB;
      const bool fin = ok && mbar_wait(&done[buf], static_cast<uint32_t>(n / NB) & 1u, abort);
      ok = __all_sync(0xffffffffu, fin);  // warp-uniform: tcgen05.ld is .sync.aligned
      const Item e = item_of(a, it, BN);
      const bool split = a.nsplit > 1;
      if (ok) {
        tc_fence_after();
        const GemmJob& job = a.job[e.jb];
        // one split: y; several: this split's partial tile
        const int64_t ld = split ? a.np : job.n;
        float* dst = split ? a.part + e.z * a.m * a.np + static_cast<int64_t>(e.tx) * kBM + row_i
                           : job.y + e.n0 + row_i;
        dst += e.m0 * ld;
        const int mleft = static_cast<int>(a.m - e.m0 < BN ? a.m - e.m0 : BN);
        const bool erok = static_cast<int64_t>(e.n0) + row_i < job.n;
        // everything read: the MMAs may overwrite the accumulator
        auto release = [&]() {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(&acc_free[buf]);
        };
        if constexpr (SOLO) {
          // the groups take BN / 4 columns each, of all accumulators at once
          constexpr int W = BN / 4;
          const int c0 = W * slot;
          const int share = (e.nsteps + PARTS - 1) / PARTS;
          uint32_t v[PARTS][W];
#pragma unroll
          for (int p = 0; p < PARTS; ++p)
            tmem_ld_async<W>(lane_base + static_cast<uint32_t>(p * BN + c0), v[p]);
          asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
          for (int p = 0; p < PARTS; ++p)
#pragma unroll
            for (int c = 0; c < W; ++c) asm volatile("" : "+r"(v[p][c]));  // (not before the wait)
#pragma unroll
          for (int p = 1; p < PARTS; ++p)
            if (p * share < e.nsteps) {  // (the others were not written)
#pragma unroll
              for (int c = 0; c < W; ++c)
                v[0][c] = __float_as_uint(__uint_as_float(v[0][c]) + __uint_as_float(v[p][c]));
            }
          if (erok) {
            float* d = dst + c0 * ld;
#pragma unroll
            for (int c = 0; c < W; ++c) {
              if (c0 + c < mleft) *d = __uint_as_float(v[0][c]);
              d += ld;
            }
          }
        }
        if (!SOLO && 32 * slot >= BN) release();
#pragma unroll 1
        for (int c0 = 32 * slot; !SOLO && c0 < BN; c0 += 128) {
          uint32_t v[32];
          tmem_ld32(lane_base + static_cast<uint32_t>(buf * BN + c0), v);
          if (c0 + 128 >= BN) release();
          if (erok) {
            float* d = dst + c0 * ld;
#pragma unroll
            for (int c = 0; c < 32; ++c) {
              if (c0 + c < mleft) *d = __uint_as_float(v[c]);
              d += ld;
            }
          }
        }
      }
      // (all 16 warps meet here for each item, so that one whose wait ran out
      // leaves no other at the barriers of the sum)
      if (split && !sum_splits(a, e, BN, ok, last)) ok = false;
      if constexpr (SOLO) break;
    }
    if constexpr (!ASYM)
      big = __half2float(__hmax(__low2half(smax), __high2half(smax))) *
                static_cast<float>(1 << (Q - 1)) >= 65520.f;
    if (__any_sync(0xffffffffu, big) && lane == 0 && a.status != nullptr)
      atomicOr(a.status, SSS_FLAG_RANGE);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");  // (a CTA whose wait ran out, too)

  tc_fence_before();
  __syncthreads();
  if (*abort && threadIdx.x == 0 && a.status != nullptr) atomicOr(a.status, SSS_FLAG_TIMEOUT);
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kTmemCols)
                 : "memory");
  }
}

// The fp16 activation operand: bf16 X rounded to fp16 (nearest even), or with
// Q8 the Q8_0 values fl16(fl16(d) q) of its blocks of 32, its columns stored
// in the k order of the dequantised weights (dequant32): of every PERM columns
// (8 for q = 4, 16 for q = 2, 3), position 2i + h holds column i + h PERM/2.  A thread converts 16 columns, so two
// lanes share a Q8_0 block.  The first threads also zero the GEMM's ncnt
// split counters.  HBM- or launch-bound: 2 bytes read, 2 written per value.
template <int PERM, bool Q8>
__global__ void __launch_bounds__(256)
    x16_kernel(const uint16_t* __restrict__ x, __half* __restrict__ y, int64_t nvec,
               int* __restrict__ cnt, int ncnt, uint32_t* __restrict__ status) {
  // programmatic dependent launch: start once the preceding kernel (which
  // may still read the fp16 buffer) has completed, and only then let the GEMM
  // start, which reads the weights before this kernel has ended
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int64_t stride = static_cast<int64_t>(gridDim.x) * blockDim.x;
  const int64_t t0 = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  for (int64_t i = t0; i < ncnt; i += stride) cnt[i] = 0;
  // block-uniform trip count: with Q8 every lane joins the shuffles
  for (int64_t base = static_cast<int64_t>(blockIdx.x) * blockDim.x; base < nvec; base += stride) {
    const int64_t i = base + threadIdx.x;  // columns 16 i .. 16 i + 15 of the flat array
    const bool valid = i < nvec;
    uint32_t w[8];
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const uint4 v = valid ? __ldcs(reinterpret_cast<const uint4*>(x) + 2 * i + c)
                            : make_uint4(0u, 0u, 0u, 0u);
      w[4 * c] = v.x; w[4 * c + 1] = v.y; w[4 * c + 2] = v.z; w[4 * c + 3] = v.w;
    }
    float f[16];
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      f[2 * e] = __uint_as_float(w[e] << 16);
      f[2 * e + 1] = __uint_as_float(w[e] & 0xFFFF0000u);
    }
    if constexpr (Q8) {
      float amax = 0.f;
      unsigned bad = 0, flags = 0;
#pragma unroll
      for (int e = 0; e < 16; ++e) {
        amax = fmaxf(amax, fabsf(f[e]));
        bad |= is_nonfinite(f[e]);
      }
      amax = fmaxf(amax, __shfl_xor_sync(0xffffffffu, amax, 1));
      bad |= __shfl_xor_sync(0xffffffffu, bad, 1);
      uint16_t d16;
      const float d = q8_scale(amax, bad != 0, &d16, &flags);
      const float df = __half2float(__ushort_as_half(d16));
      const float rd = d != 0.f ? __frcp_rn(d) : 0.f;
#pragma unroll
      for (int e = 0; e < 16; ++e)
        f[e] = d != 0.f ? df * static_cast<float>(q8_code(f[e], d, rd)) : 0.f;
      if (valid && (threadIdx.x & 1) == 0 && flags != 0u && status != nullptr)
        atomicOr(status, flags);
    }
    if (valid) {
      uint32_t o[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int ea = PERM == 8 ? 8 * (j >> 2) + (j & 3) : j;
        __half2 h = __floats2half2_rn(f[ea], f[ea + PERM / 2]);
        o[j] = *reinterpret_cast<uint32_t*>(&h);
      }
      reinterpret_cast<uint4*>(y)[2 * i] = make_uint4(o[0], o[1], o[2], o[3]);
      reinterpret_cast<uint4*>(y)[2 * i + 1] = make_uint4(o[4], o[5], o[6], o[7]);
    }
  }
}

// ---------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------

// bytes of the fp16 copy of X, rounded up to 256; SIZE_MAX when m * k * 2
// does not fit in size_t (such a call is rejected before it gets here)
size_t x16_bytes(int64_t m, int64_t k) {
  if (m < 0 || k < 0) return SIZE_MAX;
  const size_t mm = static_cast<size_t>(m), kk = static_cast<size_t>(k);
  if (kk != 0 && mm > (SIZE_MAX - 255) / 2 / kk) return SIZE_MAX;
  return (mm * kk * 2 + 255) / 256 * 256;
}

// How a call runs: tile width, K splits, and k-blocks per split.
struct GemmPlan {
  int bn, nsplit, chunk;
};

// Workspace layout: fp16 X, then (split K) the partial tiles (rows padded to
// whole row tiles, rt of them over all the call's matrices), then the
// per-tile counters.
size_t round256(size_t b) { return (b + 255) / 256 * 256; }
size_t split_bytes(int64_t rt, int64_t m, const GemmPlan& p) {
  if (p.nsplit <= 1) return 0;
  const size_t tiles = static_cast<size_t>(rt) * ((m + p.bn - 1) / p.bn);
  return round256(static_cast<size_t>(p.nsplit) * m * rt * kBM * 4) + round256(tiles * 4);
}

// The plan: for each tile width the K split of least estimated SM cycles (the
// k-blocks of a CTA, its start and end, and the last arrival's sum of the partial
// tiles), then the width of least estimated time in ns (the rounds of items that the
// busiest SM takes, what all items draw together, and a split's cost).  The second
// estimate is fitted to 585 calls at q = 4 (n = 1024 .. 28672, k = 1024 .. 14336, m =
// 17 .. 2048) at every width: off by 3, 5 and 7 % (64, 128 and 256 tokens); the
// width chosen is within 0.2 % of the best one's time in the geometric mean.  (The
// first estimate alone, 290 cycles per k-block for 64 and 128 tokens and 512 for
// 256, took 128-token tiles too often: 14336 x 1024 at 256 tokens 15.6 us against
// 13.1, 20000 x 1024 at 2048 93 against 75.)  Splits end on code-tile boundaries,
// keep at least 8 k-blocks and only fill SMs that the tiles leave idle.
// rt: the row tiles of all the call's matrices; ws: the bytes the partial tiles
// must fit in.
GemmPlan plan_gemm(int64_t rt, int64_t k, int64_t m, size_t ws) {
  struct Width {
    int bn;
    int64_t cycles, drain;  // per k-block, per item
    int64_t start, item, kblock, load, split;  // ns
  };
  constexpr Width kWidths[] = {{64, 288, 600, 0, 1100, 153, 20, 2100},
                               {128, 296, 600, 40, 1830, 138, 49, 2500},
                               {256, 512, 2500, 170, 3200, 199, 97, 3200}};
  const int64_t sms = device_sm_count();
  const int64_t nkb = k / kBK;
  GemmPlan best{128, 1, static_cast<int>((nkb + kWK - 1) / kWK * kWK)};
  int64_t best_ns = INT64_MAX;
  for (const Width& w : kWidths) {
    if (w.bn > 64 && m <= w.bn / 2) break;
    const int64_t tiles = rt * ((m + w.bn - 1) / w.bn);
    GemmPlan plan = best;
    int64_t best_cycles = INT64_MAX;
    for (int64_t split = 1; split <= 32; ++split) {
      const int64_t chunk = ((nkb + split - 1) / split + kWK - 1) / kWK * kWK;
      if (split > 1 &&
          (chunk < 8 || (nkb + chunk - 1) / chunk != split || tiles * split > sms))
        continue;
      const GemmPlan p{w.bn, static_cast<int>(split), static_cast<int>(chunk)};
      if (split > 1 &&
          (x16_bytes(m, k) > ws || x16_bytes(m, k) + split_bytes(rt, m, p) > ws))
        continue;
      const int64_t rounds = (tiles * split + sms - 1) / sms;
      const int64_t sum = split > 1 ? 500 + split * m * rt * kBM * 4 / 1000 : 0;
      const int64_t cycles = rounds * (std::min(chunk, nkb) * w.cycles + w.drain) + sum;
      if (cycles < best_cycles) {
        best_cycles = cycles;
        plan = p;
      }
    }
    const int64_t items = tiles * plan.nsplit, kbs = std::min<int64_t>(plan.chunk, nkb);
    const int64_t rounds = (items + sms - 1) / sms;
    const int64_t sum = plan.nsplit > 1 ? w.split + 6 * plan.nsplit * std::min<int64_t>(m, w.bn) : 0;
    const int64_t ns =
        w.start + rounds * (kbs * w.kblock + w.item) + items * kbs * w.load / sms + sum;
    if (ns < best_ns) {
      best_ns = ns;
      best = plan;
    }
  }
  return best;
}

int64_t row_tiles(const sss_qtensor_t* const* ts, int count) {
  int64_t rt = 0;
  for (int j = 0; j < count; ++j) rt += (ts[j]->n + kBM - 1) / kBM;
  return rt;
}

struct GemmCall {
  const sss_qtensor_t* const* ts;
  float* const* ys;
  int count;
  const __half* x16;
  int64_t m;
  uint32_t* status;
  cudaStream_t stream;
  GemmPlan plan;
  float* part;
  int* cnt;
};

template <int Q, bool ASYM, int BN, bool CT, bool SOLO>
cudaError_t run_gemm(const GemmCall& c) {
  using S = Smem<BN, Q, CT, SOLO>;
  const sss_qtensor_t& t0 = *c.ts[0];  // k, q, group and grid are those of every matrix
  EncodeTiledFn enc = tensor_map_encoder();
  if (enc == nullptr) return cudaErrorNotSupported;
  GemmMaps maps;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(t0.k), static_cast<cuuint64_t>(c.m)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(t0.k) * 2};
  const cuuint32_t box[2] = {kBK, BN};
  const cuuint32_t estr[2] = {1, 1};
  CUresult cr = enc(&maps.x, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<__half*>(c.x16), dims,
                    strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                    CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                    CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (cr != CUDA_SUCCESS) return cudaErrorInvalidValue;
  GemmArgs a;
  memset(&a, 0, sizeof a);
  const int64_t nG = t0.k / t0.group;
  const int per = t0.group >= 128 ? 1 : 128 / t0.group;  // groups of 128 codes
  bool vec = nG % per == 0;
  int64_t tile0 = 0;
  for (int j = 0; j < kMaxGemmJobs; ++j) {
    maps.c[j] = maps.x;  // a placeholder where there is no code map
    if (j >= c.count) continue;
    const sss_qtensor_t& t = *c.ts[j];
    if constexpr (CT) {
      // packed codes [n][k q / 8] bytes: a tile is 32q bytes of 128 rows;
      // bytes past the row and rows past n read as zero
      const cuuint64_t cd[2] = {static_cast<cuuint64_t>(t.k * Q / 8), static_cast<cuuint64_t>(t.n)};
      const cuuint64_t cs[1] = {static_cast<cuuint64_t>(t.k * Q / 8)};
      const cuuint32_t cb[2] = {static_cast<cuuint32_t>(32 * Q), kBM};
      cr = enc(&maps.c[j], CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, t.codes, cd, cs, cb, estr,
               CU_TENSOR_MAP_INTERLEAVE_NONE,
               Q == 4   ? CU_TENSOR_MAP_SWIZZLE_128B
               : Q == 2 ? CU_TENSOR_MAP_SWIZZLE_64B
                        : CU_TENSOR_MAP_SWIZZLE_NONE,
               CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
      if (cr != CUDA_SUCCESS) return cudaErrorInvalidValue;
    }
    vec = vec && reinterpret_cast<uintptr_t>(t.scales) % (2 * per) == 0 &&
          (!ASYM || reinterpret_cast<uintptr_t>(t.mins) % (2 * per) == 0);
    a.job[j].codes = t.codes;
    a.job[j].scales = t.scales;
    a.job[j].mins = t.mins;
    a.job[j].y = c.ys[j];
    a.job[j].n = t.n;
    a.job[j].tile0 = tile0;
    tile0 += (t.n + kBM - 1) / kBM;
  }
  auto kern = gemm_kernel<Q, ASYM, BN, CT, SOLO>;
  cudaError_t e = ensure_smem(kern, S::TOTAL);
  if (e != cudaSuccess) return e;
  a.njobs = c.count;
  a.status = c.status;
  a.m = c.m;
  a.k = t0.k;
  a.G = t0.group;
  a.vec = vec ? 1 : 0;
  for (int i = 0; i < kMagics; ++i) {
    const int pos = (Q == 4 ? 4 : 2) * i;
    const uint32_t h = pos <= 10 ? static_cast<uint32_t>(25 - pos) << 10 : 0u;
    a.magic[i] = h | (h << 16);
  }
  a.stall = (test_stall_mask() & SSS_TEST_STALL_GEMM) ? 1 : 0;
  a.nsplit = c.plan.nsplit;
  a.chunk = c.plan.chunk;
  a.np = tile0 * kBM;
  a.part = c.part;
  a.cnt = c.cnt;
  const int64_t mt = (c.m + BN - 1) / BN;
  const int64_t items = tile0 * mt * c.plan.nsplit;
  if (items > INT32_MAX - 4096) return cudaErrorNotSupported;
  a.rt = static_cast<int>(tile0);
  a.mt = static_cast<int>(mt);
  a.items = static_cast<int>(items);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(std::min<int64_t>(items, device_sm_count())), 1, 1);
  cfg.blockDim = dim3(kThreads, 1, 1);
  cfg.dynamicSmemBytes = S::TOTAL;
  cfg.stream = c.stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, maps, a);
}

template <int Q, bool ASYM, bool CT>
cudaError_t gemm_bn(const GemmCall& c) {
  const int64_t items = row_tiles(c.ts, c.count) * ((c.m + c.plan.bn - 1) / c.plan.bn) * c.plan.nsplit;
  const bool solo = items <= device_sm_count();
  switch (c.plan.bn) {
    case 64: return solo ? run_gemm<Q, ASYM, 64, CT, true>(c) : run_gemm<Q, ASYM, 64, CT, false>(c);
    case 128: return solo ? run_gemm<Q, ASYM, 128, CT, true>(c) : run_gemm<Q, ASYM, 128, CT, false>(c);
    default: return run_gemm<Q, ASYM, 256, CT, false>(c);
  }
}

template <int Q, bool ASYM>
cudaError_t gemm_ct(const GemmCall& c) {
  // code rows a multiple of 16 bytes, as a tensor map needs (q = 2 and 4:
  // always, since k % 64 == 0)
  if constexpr (Q == 3) {
    if (c.ts[0]->k % 128 != 0) return gemm_bn<Q, ASYM, false>(c);
  }
  return gemm_bn<Q, ASYM, true>(c);
}

template <int Q>
cudaError_t gemm_grid(const GemmCall& c) {
  if (c.ts[0]->grid == SSS_GRID_ASYM) return gemm_ct<Q, true>(c);
  return gemm_ct<Q, false>(c);
}

// X to the fp16 operand at x16, and the ncnt split counters at cnt to zero
template <int PERM, bool Q8>
cudaError_t run_x16(const uint16_t* x, __half* x16, int64_t m, int64_t k, int* cnt, int ncnt,
                    uint32_t* status, cudaStream_t stream) {
  const int64_t nvec = m * k / 16;
  const int64_t want = (nvec + 255) / 256;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(std::max<int64_t>(
                         1, std::min<int64_t>(want, static_cast<int64_t>(device_sm_count()) * 8))),
                     1, 1);
  cfg.blockDim = dim3(256, 1, 1);
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, x16_kernel<PERM, Q8>, x, x16, nvec, cnt, ncnt, status);
}

}  // namespace

// the workspace that lets the call take its preferred plan (with split K
// where it helps); x16_bytes alone is enough to run it unsplit
size_t gemm_multi_workspace_bytes(const sss_qtensor_t* const* ts, int count, int64_t m) {
  const size_t x = x16_bytes(m, ts[0]->k);
  if (x == SIZE_MAX) return SIZE_MAX;
  const int64_t rt = row_tiles(ts, count);
  return x + split_bytes(rt, m, plan_gemm(rt, ts[0]->k, m, SIZE_MAX));
}
size_t gemm_workspace_bytes(const sss_qtensor_t& t, int64_t m) {
  const sss_qtensor_t* one[1] = {&t};
  return gemm_multi_workspace_bytes(one, 1, m);
}
size_t gemm_workspace_min_bytes(const sss_qtensor_t& t, int64_t m) { return x16_bytes(m, t.k); }

cudaError_t launch_gemm_multi(const sss_qtensor_t* const* ts, float* const* ys, int count,
                              const uint16_t* x, int64_t m, void* workspace, size_t ws_bytes,
                              uint32_t* status, cudaStream_t stream, bool act_q8) {
  if (count < 1 || count > kMaxGemmJobs) return cudaErrorInvalidValue;
  const int64_t k = ts[0]->k;
  const int q = ts[0]->q;
  __half* x16 = static_cast<__half*>(workspace);
  const int64_t rt = row_tiles(ts, count);
  const GemmPlan plan = plan_gemm(rt, k, m, ws_bytes);
  float* part = nullptr;
  int* cnt = nullptr;
  int ncnt = 0;
  if (plan.nsplit > 1) {
    unsigned char* p = static_cast<unsigned char*>(workspace) + x16_bytes(m, k);
    part = reinterpret_cast<float*>(p);
    cnt = reinterpret_cast<int*>(p + round256(static_cast<size_t>(plan.nsplit) * m * rt * kBM * 4));
    ncnt = static_cast<int>(rt * ((m + plan.bn - 1) / plan.bn));
  }
  cudaError_t e;
  if (q == 4)
    e = act_q8 ? run_x16<8, true>(x, x16, m, k, cnt, ncnt, status, stream)
               : run_x16<8, false>(x, x16, m, k, cnt, ncnt, status, stream);
  else
    e = act_q8 ? run_x16<16, true>(x, x16, m, k, cnt, ncnt, status, stream)
               : run_x16<16, false>(x, x16, m, k, cnt, ncnt, status, stream);
  if (e != cudaSuccess) return e;
  const GemmCall c{ts, ys, count, x16, m, status, stream, plan, part, cnt};
  switch (q) {
    case 2: return gemm_grid<2>(c);
    case 3: return gemm_grid<3>(c);
    case 4: return gemm_grid<4>(c);
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_gemm(const sss_qtensor_t& t, const uint16_t* x, int64_t m, float* y,
                        void* workspace, size_t ws_bytes, uint32_t* status, cudaStream_t stream,
                        bool act_q8) {
  const sss_qtensor_t* one[1] = {&t};
  float* ys[1] = {y};
  return launch_gemm_multi(one, ys, 1, x, m, workspace, ws_bytes, status, stream, act_q8);
}

}  // namespace sss
