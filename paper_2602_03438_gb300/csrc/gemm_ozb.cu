// Batched complex GEMM with FP64-class accuracy on the FP16 tensor cores (tcgen05
// kind::f16, sm_103a) from byte digits: the product engine of the mixed-precision RGF.
//
//   D = alpha op(A) op(B) + beta C,   op in {N, H},  n x n blocks, 16 <= n <= 512
//
// Error-free slicing in the manner of Ozaki et al.: every row of op(A) and column of op(B)
// gets a power-of-two scale 2^e (|x| < 2^(e-1) for its real and imaginary parts), and
// X = rint(x 2^(8 ND - e)) is cut into ND balanced base-2^8 digits, X = sum_q d_q
// 2^(8 (ND - 1 - q)), |d_q| <= 128: exact in FP16.  The slice products with s + t = g < ND are
// summed into one FP32 accumulator per g; the rest is below the result's accuracy.
//  * ND = 7 (the FP64-class product): 28 slice products.  Against 8 digits of 7 bits
//    (36 products) the entries' rounding is the same (|X| <= 2^55) and what the dropped
//    products leave out is about the same: 6 products of digits up to 128 at 2^-72 against
//    7 of digits up to 64 at 2^-70.
//  * ND = 5 (corrections): 15 slice products, error ~2^-39 of the row x column norms.
// Exactness: over a pass of 128 complex terms one slice product's sum stays within
// 2 128 2^14 = 2^22, so an accumulator is exact (2^24) for up to 4 of them.  Groups of 5
// and more: g = 4 of ND = 7 puts one of its five into a spare accumulator; the last two
// groups may round above 2^24, at 2^-56 and 2^-64 of the scales, far below what the dropped
// products leave out.  Larger n runs in passes, each drained into 64-bit integers that keep
// every bit (they may wrap once: the sign that a sum had is kept beside it).  Error against 128-bit
// sums, rms of the row x column norms, 8 digits of 7 bits before and now: normal entries n =
// 128 2.71e-17 2.55e-17, 512 1.77e-17 1.63e-17; entries decaying from the diagonal 128
// 1.26e-16 1.18e-16, 512 8.3e-17 8.0e-17; smaller at every size measured from 16 to 512.
//
// Layout: digits of op(A) are made by a pre-pass as shared-memory images in global memory,
// [unit][row tile][chunk of 16 k][real, imaginary][digit], each plane 128 rows of 16 FP16
// (32-byte swizzle); the digits of op(B) are made inside the kernel.  Real and imaginary
// parts are separate planes (B: real, imaginary, negated imaginary): with A_s fixed,
//   re += Ar_s Br, re += Ai_s (-Bi);  im += Ar_s Bi, im += Ai_s Br
// each over all of B's digit planes t < ND - s as one wide instruction.
//
// One persistent CTA per SM walks (unit, row tile, column tile) in that order, so that the
// column tiles that share an A image run side by side and read it from L2.  Warps 0-7
// drain the accumulators and store D, 8-11 make B's digits, 12 copies A's images, 13
// issues the MMAs.  All accumulators of a 128 x 32 tile fill the 512 TMEM columns, so the
// next tile's MMAs wait for the drain: it only combines the groups into 64-bit integers in
// registers; conversion, C and the stores (through shared memory, so that they are whole
// 128-byte lines) overlap the next MMAs.  A pass's real accumulators are complete, drained
// and refilled ahead of its imaginary ones, so that half of a drain overlaps MMAs too.
//
// What bounds it (n = 128): shared-memory bandwidth.  A tile's MMAs take 14.3 k clocks of the
// tensor pipe, but their operands are read from shared memory for 14 k, A's images and B's
// digits are written there for 5 k and the stores pass through it for 2 k; with the part of
// the drain (256 KB of TMEM, 5 k clocks) that nothing overlaps a tile takes 26 k.  Measured
// per 1024 units of n = 128 with C, pre-pass included (HBM bound, 143 us): 500 us, against
// 702 us for 8 digits of 7 bits in BF16 with the drain through shared memory; 16 units of
// n = 512: 408 against 955 us.  On the way (us per 1024 units of 128): issuing from one
// lane's branch 620 (each MMA's descriptors pass between the register files), a 64-bit FP
// conversion per output in place of the integer one 572, spilled registers for want of the
// register split 624, eight producer warps 635, one drain of re and im together and three
// waits per chunk 535.  A planes kept in the collector for two instructions each: no faster.
#include <cuda_fp16.h>

#include <type_traits>

#include "negf_internal.cuh"

namespace negf {

namespace {

constexpr int TM = 128;                  // rows per tile
constexpr int KC = 16;                   // complex k per chunk: one 16-deep MMA per part
constexpr int PASS = 8;                  // chunks per exact pass (128 complex k)
constexpr uint32_t A_PL = TM * 32;       // one digit plane of an A part: 128 rows of 32 bytes
constexpr int MAX_LIST = 2048;           // units of a mask that a CTA lists
constexpr unsigned long long kWaitNs = 1000000000ull;   // 1 s

// ND digits, tiles of TNC complex columns
template <int ND, int TNC>
struct Cfg {
  static constexpr uint32_t A_PART = ND * A_PL;          // a chunk's real or imaginary planes (28 KB)
  static constexpr uint32_t B_PL = TNC * 32;             // one digit plane of a B part
  static constexpr uint32_t B_CHUNK = 3 * ND * B_PL;     // real, imaginary, negated imaginary planes (21 KB)
  static constexpr uint32_t OFF_B = 2 * A_PART;          // of a stage: both A parts, then B
  static constexpr uint32_t STAGE = OFF_B + B_CHUNK;
  static constexpr int NSTG = ND == 7 ? 2 : 3;           // ring stages, one chunk each
  static constexpr int SPLIT = ND == 7 ? 4 : -1;         // the group with a spare accumulator
  static constexpr uint32_t COL_IM = ND * TNC;           // TMEM columns: re groups, im groups, spares
  static constexpr uint32_t COL_SP = 2 * ND * TNC;
  static constexpr uint32_t TMEM_COLS = TNC == 32 ? 512 : 256;
  static constexpr uint32_t OFF_ST = NSTG * STAGE;       // per epilogue warp: 32 rows of 128 bytes
  static constexpr uint32_t OFF_BAR = OFF_ST + 8 * 4096;
  static constexpr uint32_t OFF_LIST = OFF_BAR + 256;
  static constexpr uint32_t SMEM = OFF_LIST + 2 * MAX_LIST + 1024;
};
constexpr int NT = 512;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return static_cast<uint32_t>(__cvta_generic_to_shared(p)); }

// K-major rows of 32 bytes, 32-byte swizzle: 8-row atoms of 256 B, 16-byte chunk XOR (row>>2)&1
__device__ __forceinline__ uint32_t sw32(int r, int c) {   // c = FP16 column in [0, 16)
  return (uint32_t)((r >> 3) * 256 + (r & 7) * 32 + ((((c >> 3) ^ ((r & 7) >> 2)) & 1) << 4) + (c & 7) * 2);
}
__device__ __forceinline__ uint64_t sdesc32(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);   // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused, swizzled K-major)
  d |= (uint64_t)(256 >> 4) << 32;           // stride byte offset: 8-row groups
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)6 << 61;                    // 32-byte swizzle
  return d;
}
// kind::f16: FP16 A and B (K-major), FP32 D, M = 128, N columns
__device__ __forceinline__ constexpr uint32_t idesc(int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
// bounded wait: false after kWaitNs of GPU time (the caller records the timeout)
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  unsigned long long t0 = 0, t;
  for (int it = 0;; ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (it == 0) t0 = t;
    if (t - t0 > kWaitNs) return false;
  }
}
__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_g2s(uint32_t dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(dst),
               "l"(src), "r"(bytes), "r"(smem_u32(bar))
               : "memory");
}
__device__ __forceinline__ void prefetch_l2(const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar, uint32_t el) {
  asm volatile("{\n .reg .pred e;\n setp.ne.b32 e, %1, 0;\n"
               " @e tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n}\n" ::"r"(smem_u32(bar)),
               "r"(el)
               : "memory");
}
// the A collector: FILL reads A and keeps it for LAST, which drops it; ONCE keeps nothing
enum Collect { FILL, LAST, ONCE };
template <int C>
__device__ __forceinline__ void mma(uint32_t d, uint64_t a, uint64_t b, uint32_t id, uint32_t acc, uint32_t el) {
#define NEGF_MMA(Q)                                                                                              \
  asm volatile("{\n .reg .pred p, e;\n setp.ne.b32 p, %4, 0;\n setp.ne.b32 e, %5, 0;\n"                          \
               " @e tcgen05.mma.cta_group::1.kind::f16.collector::a::" Q " [%0], %1, %2, %3, p;\n}\n" ::"r"(d),  \
               "l"(a), "l"(b), "r"(id), "r"(acc), "r"(el)                                                        \
               : "memory")
  if (C == FILL) NEGF_MMA("fill");
  else if (C == LAST) NEGF_MMA("lastuse");
  else NEGF_MMA("discard");
#undef NEGF_MMA
}
// 1 in the one lane that issues for the warp
__device__ __forceinline__ uint32_t elect_one() {
  uint32_t e;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(e));
  return e;
}

// One A part (its ND digit planes at `da`) against one set of B planes: the product goes to
// the groups' columns from c on (spare accumulator at sp).  first: these MMAs initialise the
// accumulators.  Rolled loops: a pass's unrolled MMAs are some 25 KB of straight-line code,
// whose fetch held the issuing warp for a quarter of a tile's time.
template <int ND, int TNC>
__device__ __forceinline__ void part_mmas(uint32_t c, uint32_t sp, uint64_t a, uint64_t b, bool first, uint32_t el) {
  using T = Cfg<ND, TNC>;
  const uint32_t acc0 = first ? 0u : 1u;
  constexpr uint32_t STEP = A_PL >> 4, NSTEP = (uint32_t)(TNC >> 3) << 17;
  uint32_t id = idesc(ND * TNC), acc = acc0;
  constexpr int S1 = T::SPLIT > 0 ? T::SPLIT : ND;
#pragma unroll 1
  for (int s = 0; s < S1; ++s) {
    mma<ONCE>(c, a, b, id, acc, el);
    acc = 1u;
    a += STEP;
    c += TNC;
    id -= NSTEP;
  }
  if (T::SPLIT > 0) {   // the split digit: its product with t = 0 goes to the spare accumulators
    mma<FILL>(sp, a, b, idesc(TNC), acc0, el);
    mma<LAST>(c + TNC, a, b + (T::B_PL >> 4), id - NSTEP, 1u, el);
#pragma unroll 1
    for (int s = S1 + 1; s < ND; ++s) {
      a += STEP;
      c += TNC;
      id -= NSTEP;
      mma<ONCE>(c, a, b, id, 1u, el);
    }
  }
}

#define TC_LD4(taddr, r)                                                                          \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"                         \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])                                    \
               : "r"(taddr))

// ---------------------------------------------------------------------------
// digits
// ---------------------------------------------------------------------------
// the high word of |x| orders like the value and carries its exponent: scales from integer
// maxima.  e with |x| < 2^(e - 1) for the largest word (0 for an all-zero vector;
// kNonFiniteScale where it is an infinity's or a NaN's, whose digits come out as zeros)
__device__ __forceinline__ unsigned int abs_hi(double x) { return (unsigned int)__double2hiint(x) & 0x7FFFFFFFu; }
__device__ __forceinline__ int scale_exp_hi(unsigned int h) {
  if (h == 0) return 0;
  if (h >= 0x7FF00000u) return kNonFiniteScale;
  const int ex = (int)(h >> 20);
  return (ex == 0 ? 1 : ex) - 1021;
}

// x with its sign flipped by `mask` (0 or the sign bit): a negation chosen at run time would
// be an FP64 instruction
__device__ __forceinline__ double flip(double x, int mask) {
  return __hiloint2double(__double2hiint(x) ^ mask, __double2loint(x));
}
// conj(x): -x would be an FP64 instruction (1024 products of n = 128 with B^H: 402 -> 389 us)
__device__ __forceinline__ zc conj_bits(zc x) { return zmake(x.x, flip(x.y, (int)0x80000000)); }

// 128 in each of the ND - 1 low bytes
template <int ND>
constexpr unsigned long long kByteBias = (0x8080808080808080ull >> (8 * (9 - ND)));

// Y = X + kByteBias with X = rint(x 2^(8 ND - e)): byte k of Y, minus 128, is the digit of
// weight 2^(8k), and Y >> 8 (ND - 1) the top one (the carries of one addition balance all)
template <int ND>
__device__ __forceinline__ long long biased_bytes(double x, int e) {
  const int hi = __double2hiint(x);
  const int ex = (hi >> 20) & 0x7FF;
  const unsigned long long m =
      ((unsigned long long)(unsigned)((hi & 0xFFFFF) | 0x100000) << 32) | (unsigned)__double2loint(x);
  // X = m 2^(ex - 1075 + 8 ND - e) rounded: (m << 3) >> s with s >= 1, because |x| < 2^(e-1)
  const int s = min(1078 - 8 * ND + e - ex, 63);
  long long X = (long long)((((m << 3) >> (s - 1)) + 1) >> 1);
  if (ex == 0) X = 0;
  if (hi < 0) X = -X;
  return X + (long long)kByteBias<ND>;
}
// digit plane q of two values as FP16 pairs: 1024 + byte as FP16 bits, minus 1152
template <int ND>
__device__ __forceinline__ unsigned int digit_pair(long long y0, long long y1, int q) {
  unsigned int u;
  if (q == 0) {
    const int t0 = ND == 7 ? (int)(y0 >> 32) >> 16 : (int)(y0 >> 32), t1 = ND == 7 ? (int)(y1 >> 32) >> 16 : (int)(y1 >> 32);
    u = (unsigned)(0x6480 + t0) | ((unsigned)(0x6480 + t1) << 16);
  } else {
    const int k = ND - 1 - q;
    const unsigned int w0 = k < 4 ? (unsigned)y0 : (unsigned)(y0 >> 32), w1 = k < 4 ? (unsigned)y1 : (unsigned)(y1 >> 32);
    const unsigned int sel = (unsigned)((k & 3) | (k & 3) << 4 | (4 + (k & 3)) << 8 | (4 + (k & 3)) << 12);
    u = (__byte_perm(w0, w1, sel) & 0x00FF00FFu) | 0x64006400u;
  }
  const __half2 v = __hsub2(*reinterpret_cast<const __half2*>(&u), __half2half2(__ushort_as_half(0x6480)));
  return *reinterpret_cast<const unsigned int*>(&v);
}
static_assert((0x8080808080808080ull >> 16) == 0x0000808080808080ull, "six low bytes for seven digits");

struct ImgArgs {
  unsigned char* a;   // [unit][tiles_m][chunks] x (real, imaginary) x ND planes
  int* ea;            // [unit][n] row scales of op(A)
  int* eb;            // [unit][n] column scales of op(B)
  int tiles_m, tiles_n, chunks;
};

// operands in the plain layout as a compact argument (the general BMat's fields cost the
// pre-pass registers), or as they are
struct Plain {
  const zc* p;
  long long us;
  __device__ const zc* at(int u) const { return p + (long long)u * us; }
};
struct PreArgs {
  Plain A, B;
  int opA, opB, n;
  const int* active;
};

// ---------------------------------------------------------------------------
// pre-pass: blocks of 32 rows of op(A) (scales and digit images), then blocks of 32 columns
// of op(B) (scales); HOLD: a row's entries stay in registers between scale and digits
// ---------------------------------------------------------------------------
constexpr int PRE = 32;
template <int ND, bool HOLD, class ARGS>
__global__ void __launch_bounds__(256) ozb_prepass_kernel(ARGS g, ImgArgs im, int a_blocks) {
  pdl_begin();
  const int u = blockIdx.y;
  if (g.active && !g.active[u]) return;
  const int n = g.n, tid = threadIdx.x;
  if ((int)blockIdx.x >= a_blocks) {
    const int c0 = ((int)blockIdx.x - a_blocks) * PRE;
    const zc* __restrict__ B = g.B.at(u);
    int* out = im.eb + (size_t)u * n;
    const int warp = tid >> 5, lane = tid & 31;
    if (g.opB == OP_H) {   // rows of B, a warp for four of them side by side
      unsigned int v[PRE / 8] = {};
#pragma unroll 2
      for (int k = lane; k < n; k += 32) {
#pragma unroll
        for (int q = 0; q < PRE / 8; ++q) {
          const int c = c0 + warp + 8 * q;
          const zc x = c < n ? B[(size_t)c * n + k] : zmake(0.0, 0.0);
          v[q] = max(v[q], max(abs_hi(x.x), abs_hi(x.y)));
        }
      }
#pragma unroll
      for (int q = 0; q < PRE / 8; ++q) {
        const int c = c0 + warp + 8 * q;
        v[q] = __reduce_max_sync(0xffffffffu, v[q]);
        if (lane == 0 && c < n) out[c] = scale_exp_hi(v[q]);
      }
    } else {
      __shared__ unsigned int part[8][PRE];
      const int c = c0 + lane;
      unsigned int v = 0;
      if (c < n) {
#pragma unroll 8
        for (int k = warp; k < n; k += 8) {
          const zc x = B[(size_t)k * n + c];
          v = max(v, max(abs_hi(x.x), abs_hi(x.y)));
        }
      }
      part[warp][lane] = v;
      __syncthreads();
      if (warp == 0 && c < n) {
#pragma unroll
        for (int w = 1; w < 8; ++w) v = max(v, part[w][lane]);
        out[c] = scale_exp_hi(v);
      }
    }
    return;
  }
  // eight threads per row, thread `sub` at k = 16 c + 2 sub, + 1 of every chunk c
  const zc* __restrict__ A = g.A.at(u);
  const int sub = tid & 7, gm = blockIdx.x * PRE + (tid >> 3), tm = gm / TM, am = gm - tm * TM;
  const int chunks = im.chunks;
  auto load = [&](int c, int h) {
    const int gk = c * KC + 2 * sub + h;
    zc x = zmake(0.0, 0.0);
    if (gm < n && gk < n) x = (g.opA == OP_N) ? A[(size_t)gm * n + gk] : conj_bits(A[(size_t)gk * n + gm]);
    return x;
  };
  constexpr int H = HOLD ? PASS : 1;
  zc v[H][2];
  unsigned int mh = 0;
  if (HOLD) {
#pragma unroll
    for (int c = 0; c < H; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) v[c][h] = (c < chunks) ? load(c, h) : zmake(0.0, 0.0);
#pragma unroll
    for (int c = 0; c < H; ++c)
#pragma unroll
      for (int h = 0; h < 2; ++h) mh = max(mh, max(abs_hi(v[c][h].x), abs_hi(v[c][h].y)));
  } else {
#pragma unroll 4
    for (int c = 0; c < chunks; ++c) {
      const zc x = load(c, 0), y = load(c, 1);
      mh = max(max(mh, max(abs_hi(x.x), abs_hi(x.y))), max(abs_hi(y.x), abs_hi(y.y)));
    }
  }
#pragma unroll
  for (int off = 1; off < 8; off <<= 1) mh = max(mh, __shfl_xor_sync(0xffffffffu, mh, off));
  const int e = scale_exp_hi(mh);
  if (gm >= n) return;   // rows past n keep what the image holds: they reach no stored entry
  if (sub == 0) im.ea[(size_t)u * n + gm] = e;
  unsigned char* row = im.a + (size_t)(u * im.tiles_m + tm) * chunks * (2 * ND * A_PL) + sw32(am, 2 * sub);
  auto emit = [&](int c, zc x, zc y) {
    unsigned char* img = row + (size_t)c * (2 * ND * A_PL);
    const long long r0 = biased_bytes<ND>(x.x, e), r1 = biased_bytes<ND>(y.x, e);
    const long long i0 = biased_bytes<ND>(x.y, e), i1 = biased_bytes<ND>(y.y, e);
#pragma unroll
    for (int q = 0; q < ND; ++q) {
      *reinterpret_cast<unsigned int*>(img + q * A_PL) = digit_pair<ND>(r0, r1, q);
      *reinterpret_cast<unsigned int*>(img + (ND + q) * A_PL) = digit_pair<ND>(i0, i1, q);
    }
  };
  if (HOLD) {
#pragma unroll
    for (int c = 0; c < H; ++c)
      if (c < chunks) emit(c, v[c][0], v[c][1]);
  } else {
#pragma unroll 2
    for (int c = 0; c < chunks; ++c) emit(c, load(c, 0), load(c, 1));
  }
}

// ---------------------------------------------------------------------------
// the product
// ---------------------------------------------------------------------------
// one output's group sums of a pass (column j of the loaded registers) as a 64-bit integer in units
// of 2^-56 (ND = 7; the last group's low byte rounded off, 2^-57 where the dropped products
// leave out some 2^-54) or 2^-48 (ND = 5) of the scales: below 2^62
template <int ND>
__device__ __forceinline__ long long combine(const uint32_t (&g)[8][4], int j) {
  auto G = [&](int d) { return __float2int_rn(__uint_as_float(g[d][j])); };
  const int top = G(0) * 256 + G(1);
  if (ND == 7) {
    long long w = (long long)G(2) * (1 << 24);
    w += (long long)G(3) * (1 << 16);
    w += (long long)(G(4) + G(7)) * 256;
    w += G(5) + ((G(6) + 128) >> 8);
    return w + ((long long)top << 32);
  }
  long long w = (long long)G(2) * (1 << 16);
  w += (long long)G(3) * 256 + G(4);
  return w + (long long)top * (1 << 24);
}

// v 2^p as a double (0 for v = 0 or below the normal range), |v| < 2^63 and p <= kMaxExp, built in
// integers: a 64-bit conversion is an FP64-pipe instruction, and a tile's 8192 of them held
// that pipe for a third of the tile's time
constexpr int kMaxExp = 960;   // no result is past the range of a double up to here
__device__ __forceinline__ double ldexp_int(long long v, int p) {
  const int sg = (int)(v >> 32) & (int)0x80000000;
  const unsigned long long a = v < 0 ? 0ull - (unsigned long long)v : (unsigned long long)v;
  const int lz = __clzll((long long)a);
  const unsigned long long m = a << (lz & 63);                     // leading bit at 63
  const unsigned long long r = (m >> 11) + ((m >> 10) & 1ull);     // 53 bits, rounded (a carry moves the exponent)
  const int e = 1085 - lz + p;                                     // exponent field - 1: the leading bit adds 1
  if (lz == 64 || e < 0) return 0.0;
  return __hiloint2double((int)(r >> 32) + (e << 20) + sg, (int)(unsigned)r);
}
// the same for any p: infinity past the range, NaN where p holds a kNonFiniteScale
// other_sign: v stands 2^64 off, to the side of its sign
__device__ __forceinline__ double ldexp_any(long long v, bool other_sign, int p) {
  if (p > kNonFiniteScale / 2) return NAN;
  const int down = p > kMaxExp ? p - kMaxExp : 0;   // (up to 1200)
  double x;
  if (other_sign) {   // 2^63 <= |value| < 2^64
    const bool neg = v >= 0;
    const unsigned long long a = neg ? 0ull - (unsigned long long)v : (unsigned long long)v;
    x = flip(ldexp_int((long long)((a >> 1) | (a & 1)), p - down + 1), neg ? (int)0x80000000 : 0);
  } else {
    x = ldexp_int(v, p - down);
  }
  for (int d = down; d > 0; d -= 600) x *= __hiloint2double((1023 + min(d, 600)) << 20, 0);
  return x;
}
// UAB: alpha = +-1, beta in {0, +-1}; MASK: g.active may be given (its registers cost the others 3%)
template <int ND, int TNC, bool UAB, bool MASK>
__global__ void __launch_bounds__(NT, 1) ozb_product_kernel(GemmArgs g, ImgArgs im, int* err) {
  using T = Cfg<ND, TNC>;
  constexpr int NSTG = T::NSTG;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + T::OFF_BAR);
  // full[s]: a chunk's A images (one expect_tx) and B digits (four warps); emptyR[s], emptyI[s]:
  // its real and imaginary A planes are read (with the imaginary ones, B too)
  uint64_t *full = bars, *emptyR = full + NSTG, *emptyI = emptyR + NSTG;
  uint64_t *doneR = emptyI + NSTG, *doneI = doneR + 1;   // a pass's re, im accumulators are complete
  uint64_t *freeR = doneI + 1, *freeI = freeR + 1;       // ... are drained
  uint64_t* fin = freeI + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(fin + 1);
  __shared__ volatile int s_fail;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = g.n, chunks = im.chunks;
  const int per_unit = im.tiles_m * im.tiles_n;
  uint16_t* list = reinterpret_cast<uint16_t*>(base + T::OFF_LIST);
  __shared__ int s_warp[NT / 32];

  if (tid == 0) {
    for (int i = 0; i < NSTG; ++i) {
      mbar_init(&full[i], 5);
      mbar_init(&emptyR[i], 1);
      mbar_init(&emptyI[i], 1);
    }
    mbar_init(doneR, 1);
    mbar_init(doneI, 1);
    mbar_init(freeR, 8);
    mbar_init(freeI, 8);
    mbar_init(fin, 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(T::TMEM_COLS)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  pdl_begin();
  // Under a mask the tiles are those of the units set, in the order of their numbers: every CTA
  // makes the same list.  (Walking all units and skipping gave a CTA up to twice the mean: 384
  // units of n = 128, 135 of them set, 67 -> 56 us.)
  const bool listed = MASK && g.active && g.units <= MAX_LIST;
  int count = g.units;
  if (listed) {
    count = 0;
    for (int u0 = 0; u0 < g.units; u0 += NT) {
      const bool set = u0 + tid < g.units && g.active[u0 + tid];
      const unsigned int m = __ballot_sync(0xffffffffu, set);
      if (lane == 0) s_warp[warp] = __popc(m);
      __syncthreads();
      int before = count;
#pragma unroll
      for (int w = 0; w < NT / 32; ++w) {
        const int k = s_warp[w];
        before += w < warp ? k : 0;
        count += k;
      }
      if (set) list[before + __popc(m & ((1u << lane) - 1u))] = (uint16_t)(u0 + tid);
      __syncthreads();
    }
  }
  const long long ntiles = (long long)count * per_unit;
  const uint32_t tmem = *tmem_slot;
  const uint32_t lbase = smem_u32(base);
  // a tile's unit, row tile and column tile; every role walks the same tiles
  auto tile_at = [&](long long i, int& u, int& tm, int& tn) {
    u = (int)(i / per_unit);
    const int r = (int)(i - (long long)u * per_unit);
    tm = r / im.tiles_n;
    tn = r - tm * im.tiles_n;
    if (listed) {
      u = list[u];
      return true;
    }
    return !(MASK && g.active && !g.active[u]);
  };

  // registers move between the warpgroups (each role's branch begins with its share):
  // 2 x 192 + 72 + 56 = 512, the launch's 4 x 128 per lane
  if (warp >= 12) {
   asm volatile("setmaxnreg.dec.sync.aligned.u32 56;");
   if (warp == 12) {
    // ---------------- A: each chunk's real and imaginary planes into its stage.  The tiles of
    // one image take turns prefetching it into L2, PF chunks ahead.
    if (lane == 0) {
      constexpr int PF = 3;
      int st = 0, issued = 0;
      uint32_t ph = 0;   // parity of the stage's last release
      bool filled = false;
      for (long long i = blockIdx.x; i < ntiles && !s_fail; i += gridDim.x) {
        int u, tm, tn;
        if (!tile_at(i, u, tm, tn)) continue;
        const unsigned char* img = im.a + (size_t)(u * im.tiles_m + tm) * chunks * (2 * T::A_PART);
        for (int c = 0; c < chunks; ++c) {
          const unsigned char* src = img + (size_t)c * (2 * T::A_PART);
          const uint32_t dst = lbase + st * T::STAGE;
          if (filled && !mbar_wait(&emptyR[st], ph ^ 1)) { s_fail = 1; break; }
          mbar_expect_tx(&full[st], 2 * T::A_PART);
          bulk_g2s(dst, src, T::A_PART, &full[st]);
          if (filled && !mbar_wait(&emptyI[st], ph ^ 1)) s_fail = 1;   // (the copy completes the stage's count)
          bulk_g2s(dst + T::A_PART, src + T::A_PART, T::A_PART, &full[st]);
          ++issued;
          if (s_fail) break;
          const int cp = c + PF;
          if (cp < chunks && cp % im.tiles_n == tn) prefetch_l2(src + (size_t)PF * (2 * T::A_PART), 2 * T::A_PART);
          if (++st == NSTG) { st = 0; ph ^= 1; filled = true; }
        }
      }
      if (s_fail) {   // a timeout: let the copies in flight land before the CTA ends
        for (int m = max(0, issued - NSTG); m < issued; ++m) mbar_wait(&full[m % NSTG], (m / NSTG) & 1);
      }
    }
   } else if (warp == 13) {
    // ---------------- MMA issue: the whole warp walks the loops, so that descriptors stay in
    // uniform registers (issued from one lane's branch, every MMA took ~100 clocks of moves
    // between register files), and one elected lane issues
    const uint32_t el = elect_one();
    {
      const uint32_t re = tmem, imc = tmem + T::COL_IM, spr = tmem + T::COL_SP, spi = spr + TNC;
      int st = 0;
      uint32_t ph = 0, passes = 0;
      for (long long i = blockIdx.x; i < ntiles && !s_fail; i += gridDim.x) {
        int u, tm, tn;
        if (!tile_at(i, u, tm, tn)) continue;
        for (int c0 = 0; c0 < chunks && !s_fail; c0 += PASS) {
          const int c1 = min(c0 + PASS, chunks);
          for (int c = c0; c < c1; ++c) {
            if (!mbar_wait(&full[st], ph)) { s_fail = 1; break; }
            const uint32_t sa = lbase + st * T::STAGE;
            const uint64_t ar = sdesc32(sa), ai = sdesc32(sa + T::A_PART), br = sdesc32(sa + T::OFF_B);
            const uint64_t bi = br + ((ND * T::B_PL) >> 4), nbi = br + ((2 * ND * T::B_PL) >> 4);
            const bool first = c == c0, last = c == c1 - 1;
            // all of re, then all of im: the drain of one overlaps the MMAs of the other
            if (first && passes > 0 && !mbar_wait(freeR, (passes - 1) & 1)) { s_fail = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            part_mmas<ND, TNC>(re, spr, ar, br, first, el);
            part_mmas<ND, TNC>(re, spr, ai, nbi, false, el);
            if (last) mma_commit(doneR, el);
            if (first && passes > 0 && !mbar_wait(freeI, (passes - 1) & 1)) { s_fail = 1; break; }
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            part_mmas<ND, TNC>(imc, spi, ar, bi, first, el);
            mma_commit(&emptyR[st], el);
            part_mmas<ND, TNC>(imc, spi, ai, br, false, el);
            mma_commit(&emptyI[st], el);
            if (last) mma_commit(doneI, el);
            if (++st == NSTG) { st = 0; ph ^= 1; }
          }
          if (s_fail) break;
          ++passes;
        }
      }
      if (s_fail) {   // a timeout: wait for the MMAs in flight
        mma_commit(fin, el);
        mbar_wait(fin, 0);
      }
    }
   }
  } else if (warp >= 8) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 72;");
    // ---------------- B digits: TPC threads per column, KPT consecutive complex k each; the
    // next chunk (of this tile or the next) is loaded while this one is cut
    constexpr int TPC = 128 / TNC, KPT = KC / TPC;
    const int tb = tid - 256, bn = tb / TPC, k0 = (tb % TPC) * KPT;
    const uint32_t off = sw32(bn, k0);
    long long i = blockIdx.x;
    int u = 0, tm = 0, tn = 0, c = 0;
    auto skip_on = [&]() {
      while (i < ntiles && !tile_at(i, u, tm, tn)) i += gridDim.x;
    };
    auto load = [&](zc* v, int& eb) {
      const int gn = tn * TNC + bn;
      const zc* B = g.B.at(u);
      eb = (gn < n) ? im.eb[(size_t)u * n + gn] : 0;
#pragma unroll
      for (int h = 0; h < KPT; ++h) {
        const int gk = c * KC + k0 + h;
        v[h] = zmake(0.0, 0.0);
        if (gn < n && gk < n) v[h] = (g.opB == OP_N) ? B[(size_t)gk * n + gn] : conj_bits(B[(size_t)gn * n + gk]);
      }
    };
    auto advance = [&]() {
      if (++c == chunks) {
        c = 0;
        i += gridDim.x;
        skip_on();
      }
    };
    skip_on();
    zc nx[KPT];
    int eb_nx = 0;
    if (i < ntiles) load(nx, eb_nx);
    int st = 0;
    uint32_t ph = 0;
    bool filled = false;
    while (i < ntiles && !s_fail) {
      zc v[KPT];
      const int eb = eb_nx;
#pragma unroll
      for (int h = 0; h < KPT; ++h) v[h] = nx[h];
      advance();
      if (i < ntiles) load(nx, eb_nx);
      long long yr[KPT], yi[KPT];
#pragma unroll
      for (int h = 0; h < KPT; ++h) {
        yr[h] = biased_bytes<ND>(v[h].x, eb);
        yi[h] = biased_bytes<ND>(v[h].y, eb);
      }
      if (filled && !mbar_wait(&emptyI[st], ph ^ 1)) { s_fail = 1; break; }
      unsigned char* P = base + st * T::STAGE + T::OFF_B + off;
#pragma unroll
      for (int q = 0; q < ND; ++q) {
        const unsigned int r0 = digit_pair<ND>(yr[0], yr[1], q), i0 = digit_pair<ND>(yi[0], yi[1], q);
        unsigned char* Q = P + q * T::B_PL;
        constexpr unsigned int NEG = 0x80008000u;
        if (KPT == 4) {
          const unsigned int r1 = digit_pair<ND>(yr[KPT - 2], yr[KPT - 1], q), i1 = digit_pair<ND>(yi[KPT - 2], yi[KPT - 1], q);
          *reinterpret_cast<uint2*>(Q) = make_uint2(r0, r1);
          *reinterpret_cast<uint2*>(Q + ND * T::B_PL) = make_uint2(i0, i1);
          *reinterpret_cast<uint2*>(Q + 2 * ND * T::B_PL) = make_uint2(i0 ^ NEG, i1 ^ NEG);
        } else {
          *reinterpret_cast<unsigned int*>(Q) = r0;
          *reinterpret_cast<unsigned int*>(Q + ND * T::B_PL) = i0;
          *reinterpret_cast<unsigned int*>(Q + 2 * ND * T::B_PL) = i0 ^ NEG;
        }
      }
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&full[st]);
      if (++st == NSTG) { st = 0; ph ^= 1; filled = true; }
    }
  } else {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 192;");
    // ---------------- drain and store: TMEM lanes 32 (warp % 4) .., TNC / 2 complex columns
    constexpr int CW = TNC / 2;                 // complex columns per thread
    const int quad = warp & 3, cb = (warp >> 2) * CW;
    const uint32_t lane_base = tmem + ((uint32_t)(32 * quad) << 16);
    unsigned char* stg = base + T::OFF_ST + warp * 4096;
    uint32_t passes = 0;
    for (long long i = blockIdx.x; i < ntiles && !s_fail; i += gridDim.x) {
      int u, tm, tn;
      if (!tile_at(i, u, tm, tn)) continue;
      const int m0 = tm * TM + 32 * quad, n0 = tn * TNC + cb;
      // the scales, long before they are used
      const int er = (m0 + lane < n) ? im.ea[(size_t)u * n + m0 + lane] - (ND == 7 ? 56 : 48) : 0;
      int ebj[CW / 8];   // lane j holds column j's
#pragma unroll
      for (int h = 0; h < CW / 8; ++h) {
        const int gcol = n0 + 8 * h + (lane & 7);
        ebj[h] = gcol < n ? im.eb[(size_t)u * n + gcol] : 0;
      }
      // The passes' sums wrap: each is below 2^62 and four below 2^64.  Bit j of wrapped (CW + j for the
      // imaginary part) says that column j's stands 2^64 off, to the side of its sign.
      long long vr[CW], vi[CW];
      uint32_t wrapped = 0;
      // one pass: the first, or a later one, whose sums may wrap (each in code of its own: the check's
      // instructions in every pass cost 2% of a product of one)
      auto drain = [&](auto first) {
        bool ok = true;
#pragma unroll
        for (int part = 0; part < 2; ++part) {
          ok = __all_sync(0xffffffffu, mbar_wait(part ? doneI : doneR, passes & 1));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          // steps of 4 complex columns; the next step's loads fly while this step's groups are
          // combined
          uint32_t w[2][8][4];
          auto fetch = [&](int cc, uint32_t (&x)[8][4]) {
#pragma unroll
            for (int d = 0; d < ND; ++d) TC_LD4(lane_base + (uint32_t)(part * T::COL_IM + d * TNC + cb + 4 * cc), x[d]);
            if (ND == 7) TC_LD4(lane_base + (uint32_t)(T::COL_SP + part * TNC + cb + 4 * cc), x[7]);
          };
          fetch(0, w[0]);
#pragma unroll
          for (int cc = 0; cc < CW / 4; ++cc) {
            asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
            if (cc + 1 < CW / 4) fetch(cc + 1, w[(cc + 1) & 1]);
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const long long v = combine<ND>(w[cc & 1], j);
              long long& o = part ? vi[4 * cc + j] : vr[4 * cc + j];
              if (decltype(first)::value) {
                o = v;
              } else if (ND < 7) {
                o += v;
              } else {
                const long long t = (long long)((unsigned long long)o + (unsigned long long)v);
                wrapped ^= ((uint32_t)(((o ^ t) & (v ^ t)) >> 32) >> 31) << (part * CW + 4 * cc + j);
                o = t;
              }
            }
          }
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(part ? freeI : freeR);
        }
        if (!ok) s_fail = 1;
        ++passes;
        return ok;
      };
      bool ok = drain(std::true_type());
      for (int c0 = PASS; ok && c0 < chunks; c0 += PASS) ok = drain(std::false_type());
      if (!ok) break;
      // rows of this lane -> doubles -> shared memory, then 8 lanes per row: whole lines
      zc* D = g.D.at(u);
      const zc* Cm = (g.C.p && !(UAB && g.beta.x == 0.0)) ? g.C.at(u) : nullptr;
      const int j = lane & 7, r4 = lane >> 3;
      const int neg_a = g.alpha.x < 0.0 ? (int)0x80000000 : 0, neg_b = g.beta.x < 0.0 ? (int)0x80000000 : 0;
      int eb_max = ebj[0];
#pragma unroll
      for (int h = 1; h < CW / 8; ++h) eb_max = max(eb_max, ebj[h]);
      if (__reduce_max_sync(0xffffffffu, er) + __reduce_max_sync(0xffffffffu, eb_max) > kMaxExp ||
          __any_sync(0xffffffffu, wrapped != 0)) {
        // results near the end of the range or past it, or past 64 bits: the integers through shared memory, each
        // converted with its own check (in the path below that check cost 2% of the product)
#pragma unroll
        for (int h = 0; h < CW / 8; ++h) {
#pragma unroll
          for (int q = 0; q < 8; ++q)
            *reinterpret_cast<longlong2*>(stg + lane * 128 + ((q ^ (lane & 7)) << 4)) = make_longlong2(vr[8 * h + q], vi[8 * h + q]);
          __syncwarp();
          const int gcol = n0 + 8 * h + j;
#pragma unroll 1
          for (int k = 0; k < 8; ++k) {
            const int rl = 4 * k + r4, row = m0 + rl;
            const int p = __shfl_sync(0xffffffffu, er, rl) + __shfl_sync(0xffffffffu, ebj[h], j);
            const longlong2 x = *reinterpret_cast<const longlong2*>(stg + rl * 128 + ((j ^ (rl & 7)) << 4));
            const uint32_t off = __shfl_sync(0xffffffffu, wrapped, rl) >> (8 * h + j);
            if (row >= n || gcol >= n) continue;
            const zc acc = zmake(ldexp_any(x.x, off & 1, p), ldexp_any(x.y, (off >> CW) & 1, p));
            const zc c = Cm ? Cm[(size_t)row * n + gcol] : zmake(0.0, 0.0);
            zc v = UAB ? zmake(flip(acc.x, neg_a), flip(acc.y, neg_a)) : zmul(g.alpha, acc);
            if (Cm) v = zadd(v, UAB ? zmake(flip(c.x, neg_b), flip(c.y, neg_b)) : zmul(g.beta, c));
            if (g.plus_identity && row == gcol) v.x += 1.0;
            D[(size_t)row * n + gcol] = v;
          }
          __syncwarp();
        }
        continue;
      }
#pragma unroll
      for (int h = 0; h < CW / 8; ++h) {
        if (n0 + 8 * h >= n) break;
        const int gcol = n0 + 8 * h + j;
        zc cv[8];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int row = m0 + 4 * k + r4;
          cv[k] = (Cm && row < n && gcol < n) ? Cm[(size_t)row * n + gcol] : zmake(0.0, 0.0);
        }
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          const int p = er + __shfl_sync(0xffffffffu, ebj[h], q);
          const zc v = zmake(ldexp_int(vr[8 * h + q], p), ldexp_int(vi[8 * h + q], p));
          *reinterpret_cast<zc*>(stg + lane * 128 + ((q ^ (lane & 7)) << 4)) = v;
        }
        __syncwarp();
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const int rl = 4 * k + r4, row = m0 + rl;
          const zc acc = *reinterpret_cast<const zc*>(stg + rl * 128 + ((j ^ (rl & 7)) << 4));
          zc v;
          if (UAB) {
            v = zmake(flip(acc.x, neg_a), flip(acc.y, neg_a));
            if (Cm) v = zadd(v, zmake(flip(cv[k].x, neg_b), flip(cv[k].y, neg_b)));
          } else {
            v = zmul(g.alpha, acc);
            if (Cm) v = zadd(v, zmul(g.beta, cv[k]));
          }
          if (g.plus_identity) {
            if (row == gcol) v.x += 1.0;
          }
          if (row < n && gcol < n) D[(size_t)row * n + gcol] = v;
        }
        __syncwarp();
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (s_fail && tid == 0) raise_error(err, NEGF_ERR_TIMEOUT);
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(T::TMEM_COLS) : "memory");
  }
}

int g_sms[kMaxDevices];   // multiprocessors per device (set with the kernels' attributes)

template <int ND, int TNC>
cudaError_t launch(const GemmArgs& g, void* scratch, int* err, cudaStream_t s, int slot) {
  using T = Cfg<ND, TNC>;
  cudaError_t e = once_per_device(slot, [](int d) {
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    cudaError_t r = cudaFuncSetAttribute(ozb_product_kernel<ND, TNC, true, false>, smem, (int)T::SMEM);
    if (r == cudaSuccess) r = cudaFuncSetAttribute(ozb_product_kernel<ND, TNC, true, true>, smem, (int)T::SMEM);
    if (r == cudaSuccess) r = cudaFuncSetAttribute(ozb_product_kernel<ND, TNC, false, true>, smem, (int)T::SMEM);
    if (r == cudaSuccess) r = cudaDeviceGetAttribute(&g_sms[d], cudaDevAttrMultiProcessorCount, d);
    return r;
  });
  if (e != cudaSuccess) return e;
  int dev = 0;
  if ((e = cudaGetDevice(&dev)) != cudaSuccess) return e;
  const int n = g.n;
  ImgArgs im;
  im.chunks = (n + KC - 1) / KC;
  im.tiles_m = (n + TM - 1) / TM;
  im.tiles_n = (n + TNC - 1) / TNC;
  unsigned char* p = (unsigned char*)scratch;
  im.ea = (int*)p;
  im.eb = im.ea + (size_t)n * g.units;
  p += (sizeof(int) * 2 * (size_t)n * g.units + 1023) & ~(size_t)1023;
  im.a = p;
  const int blocks = (n + PRE - 1) / PRE, ab = g.reuse_a ? 0 : blocks;
  const dim3 pre(ab + blocks, g.units);
  if (g.A.plain() && g.B.plain()) {
    PreArgs a{Plain{g.A.p, g.A.us}, Plain{g.B.p, g.B.us}, g.opA, g.opB, n, g.active};
    if (im.chunks <= PASS) e = launch_pdl(ozb_prepass_kernel<ND, true, PreArgs>, pre, 256, 0, s, a, im, ab);
    else e = launch_pdl(ozb_prepass_kernel<ND, false, PreArgs>, pre, 256, 0, s, a, im, ab);
  } else {
    if (im.chunks <= PASS) e = launch_pdl(ozb_prepass_kernel<ND, true, GemmArgs>, pre, 256, 0, s, g, im, ab);
    else e = launch_pdl(ozb_prepass_kernel<ND, false, GemmArgs>, pre, 256, 0, s, g, im, ab);
  }
  if (e != cudaSuccess) return e;
  const bool uab = (g.alpha.y == 0.0 && (g.alpha.x == 1.0 || g.alpha.x == -1.0)) &&
                   (!g.C.p || (g.beta.y == 0.0 && (g.beta.x == 0.0 || g.beta.x == 1.0 || g.beta.x == -1.0)));
  const long long tiles = (long long)g.units * im.tiles_m * im.tiles_n;
  const int grid = (int)(tiles < g_sms[dev] ? tiles : g_sms[dev]);
  auto* k = !uab ? ozb_product_kernel<ND, TNC, false, true>
            : g.active ? ozb_product_kernel<ND, TNC, true, true> : ozb_product_kernel<ND, TNC, true, false>;
  return launch_pdl(k, grid, NT, T::SMEM, s, g, im, err);
}

}  // namespace

bool oz_supported(int n) { return n >= 16 && n <= 512; }

// Workspace of a product, as negotiated with callers through their workspace sizes: scales
// and images (8 planes per part; the 7 used take less)
size_t ozt_scratch_bytes(int n, int units) {
  const size_t tm = (size_t)(n + TM - 1) / TM;
  const size_t scales = (sizeof(int) * 2 * (size_t)n * units + 1023) & ~(size_t)1023;
  const size_t chunks = (size_t)(n + KC - 1) / KC;
  const size_t half = (size_t)(n + 7) / 8 * (8 * A_PL), full = chunks * (16 * A_PL);
  return scales + (size_t)units * tm * (full > half ? full : half);
}

bool oz_variant_supported(int n, int variant) {
  if (!oz_supported(n)) return false;
  switch (variant) {
    case OZ_DEFAULT: case OZ_FULL: return true;
    case OZ_HALF: case OZ_PERSISTENT: return n <= 128;
    default: return false;
  }
}

// Tiles of 32 complex columns, or of 16 where those take less time: a 16-column tile takes
// about five eighths of a 32-column one (n = 128, 1024 units: 682 us with 8 of them against
// 534 us with 4), so they win where they fit in the same number of rounds of the SMs (n =
// 128, 4 units: 28 against 34 us) or leave out a padded half tile (n = 16, 1024 units: 56
// against 76 us; n = 48, 100 units: 28 against 37 us)
template <int ND>
static cudaError_t run(const GemmArgs& g, void* scratch, int* err, cudaStream_t s, int variant, int slot32, int slot16) {
  if (g.units <= 0 || g.n <= 0) return cudaSuccess;
  if (!scratch || !oz_variant_supported(g.n, variant)) return cudaErrorInvalidValue;
  bool narrow = variant == OZ_HALF;
  if (variant == OZ_DEFAULT) {
    const long long rows = (long long)g.units * ((g.n + TM - 1) / TM);
    const long long r16 = (rows * ((g.n + 15) / 16) + kSms - 1) / kSms, r32 = (rows * ((g.n + 31) / 32) + kSms - 1) / kSms;
    narrow = 5 * r16 < 8 * r32;
  }
  return narrow ? launch<ND, 16>(g, scratch, err, s, slot16) : launch<ND, 32>(g, scratch, err, s, slot32);
}

cudaError_t zgemm_ozt_variant(const GemmArgs& g, void* scratch, int* err, cudaStream_t s, int variant) {
  return run<7>(g, scratch, err, s, variant, INIT_OZB, INIT_OZB16);
}
cudaError_t zgemm_ozt_lo(const GemmArgs& g, void* scratch, int* err, cudaStream_t s) {
  return run<5>(g, scratch, err, s, OZ_DEFAULT, INIT_OZB_LO, INIT_OZB16_LO);
}

}  // namespace negf

extern "C" int32_t negf_sliced_digits(void) { return 7; }
