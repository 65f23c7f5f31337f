// Batched complex GEMM with FP64-class accuracy on the BF16 tensor cores
// (tcgen05 kind::f16, sm_103a) for callers with little scratch: all digits are made inside
// the kernel, and only the row and column scales pass through memory.  The sweeps'
// product is the byte-digit kernel of gemm_ozb.cu.
//
//   D = alpha op(A) op(B) + beta C,   op in {N, H},  n x n blocks, one unit per grid z.
//
// Why: FP32 accumulation on the tensor cores truncates, so a compensated TF32
// split stays at ~1e-6 relative per 128-wide product, and the near-resonant
// blocks of the RGF at eta = 1e-6 amplify that by ~1e4.  Integer-valued operands,
// however, accumulate exactly as long as every partial sum stays below 2^24.
//
// Scheme (error-free slicing in the manner of Ozaki et al.), with NS digits per value
// (NEGF_OZ_DIGITS, 6..8; 8 by default):
//  * every row m of op(A') and column j of op(B') gets a power-of-two scale 2^e
//    with all its entries below 2^(e-1) (A' = [Re A | Im A], B' = [[Re B, Im B],
//    [-Im B, Re B]] as in the TF32 kernel);
//  * each real entry x becomes X = rint(x 2^(7 NS - e)) (|X| <= 2^(7 NS - 1)) and is
//    cut into balanced base-2^7 digits d1..dNS with |d| <= 64:
//    X = sum d_s 2^(7(NS-s)), all exact in BF16;
//  * the slice products A_s B_t with s + t = d <= NS + 1 (NS (NS + 1) / 2 pairs: 36
//    for NS = 8) are summed into one FP32 accumulator per d (NS accumulators in TMEM).
//    With K = 2n real terms the largest group sum is NS * 64 * 64 * 2n < 2^24 for
//    n <= 256: exact;
//  * the epilogue forms sum_d G_d 2^(7(NS+1-d)) as two exact int64 halves, converts
//    each exactly to a double, scales it by 2^(e_A + e_B - 7 (NS + 1)) with an integer
//    addition to its exponent field, and adds the two (GB300's FP64 pipe is narrow:
//    the recombination stays in the integer units but for that one addition).
// The error is ~2^(1 - 7 NS) of |row of A| |column of B| (truncation of the digits and
// of the pairs with s + t > NS + 1; 2^-55 for NS = 8): FP64-class for the RGF
// tolerances.  (Rows and columns keep their own scales; entries far below their
// row's or column's largest entry keep an absolute, not a relative, accuracy.)
//
// Tile: 128 rows x 32 complex columns (N = 64 real: 32 real parts, 32 imaginary
// parts; NS accumulators x 64 columns in a 512-column TMEM allocation), K chunks of 16
// complex (32 real = 64-byte rows, 64B swizzle), two shared-memory stages.
#include <stdlib.h>

#include "negf_internal.cuh"

namespace negf {

namespace {

constexpr int TM = 128;                 // rows per tile
constexpr int TNC = 32;                 // complex columns per tile
constexpr int NR = 2 * TNC;             // real MMA columns (64)
constexpr int KC = 16;                  // complex K per chunk
#ifndef NEGF_OZ_DIGITS
#define NEGF_OZ_DIGITS 8
#endif
constexpr int NS = NEGF_OZ_DIGITS;      // digits per value
constexpr int NG = NS;                  // scale groups d = 2..NS+1
constexpr int HSPLIT = 4;               // groups [0, HSPLIT) and [HSPLIT, NG) recombine separately
static_assert(NS >= 4 && NS <= 8, "4 to 8 digits: the group sums and the halves stay exact");
constexpr int NT = 256;
constexpr int kCluster = 4;            // column tiles sharing one A tile's digits
constexpr uint32_t ROWB = 64;                            // bytes per smem row (32 bf16)
constexpr uint32_t A_SLICE = TM * ROWB;                  // 8 KB
constexpr uint32_t B_SLICE = NR * ROWB;                  // 4 KB
constexpr uint32_t STAGE = NS * (A_SLICE + B_SLICE);     // 96 KB for NS = 8
constexpr uint32_t SMEM_BYTES = 2 * STAGE + 1024 + 64;
constexpr unsigned long long kWaitNs = 1000000000ull;   // 1 s

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// K-major, 64-byte swizzle: 8-row atoms of 512 B; 16-byte chunk index XOR (row>>1)&3
__device__ __forceinline__ uint32_t sw64(int r, int c) {   // c = bf16 column in [0, 32)
  return (uint32_t)((r >> 3) * 512 + (r & 7) * 64 + ((((c >> 3) ^ ((r & 7) >> 1)) & 3) << 4) + (c & 7) * 2);
}

__device__ __forceinline__ uint64_t sdesc64(uint32_t saddr) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr & 0x3FFFF) >> 4);   // start address
  d |= (uint64_t)1 << 16;                    // leading byte offset (unused, swizzled K-major)
  d |= (uint64_t)(512 >> 4) << 32;           // stride byte offset: 8-row groups
  d |= (uint64_t)1 << 46;                    // descriptor version
  d |= (uint64_t)4 << 61;                    // 64-byte swizzle
  return d;
}

// kind::f16 with BF16 A/B, FP32 D, both K-major, M = 128, N = 64
constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(NR >> 3) << 17) | ((uint32_t)(TM >> 4) << 24);

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
// acquire at cluster scope: the phase was completed by arrivals from other members
__device__ __forceinline__ bool mbar_try_wait_cluster(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ bool mbar_wait_cluster(uint64_t* bar, uint32_t parity) {
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (;;) {
    if (mbar_try_wait_cluster(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > kWaitNs) return false;
  }
}
// arrive (release, cluster scope) on an mbarrier of another member (shared::cluster address)
__device__ __forceinline__ void mbar_arrive_remote(uint32_t cluster_addr) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_addr) : "memory");
}
// bounded wait: gives up after `limit_ns` of GPU time (the caller records the timeout)
__device__ __forceinline__ bool mbar_wait_ns(uint64_t* bar, uint32_t parity, unsigned long long limit_ns) {
  unsigned long long t0, t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t0));
  for (;;) {
    if (mbar_try_wait(bar, parity)) return true;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    if (t - t0 > limit_ns) return false;
  }
}
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) { return mbar_wait_ns(bar, parity, kWaitNs); }
__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
// shared::cluster address of the same shared::cta offset in member `rank`
__device__ __forceinline__ uint32_t mapa_shared(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster_v2(uint32_t addr, uint32_t a, uint32_t b) {
  asm volatile("st.shared::cluster.v2.b32 [%0], {%1, %2};" ::"r"(addr), "r"(a), "r"(b) : "memory");
}
__device__ __forceinline__ void st_cluster_v4(uint32_t addr, uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
  asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(a), "r"(b), "r"(c), "r"(d)
               : "memory");
}
// all threads of all member CTAs
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t a, uint64_t b, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(a), "l"(b), "r"(IDESC), "r"(acc)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(bar))
               : "memory");
}

#define TC_LD8(taddr, r)                                                                          \
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"          \
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), \
                 "=r"(r[7])                                                                       \
               : "r"(taddr))

// The high word of |x| (sign cleared): for non-negative doubles it orders like the value
// and carries its exponent field, so the largest entry's scale comes from integer maxima
// (GB300's FP64 pipe is narrow; fabs/fmax per entry held the pre-pass on it).
__device__ __forceinline__ unsigned int abs_hi(double x) { return (unsigned int)__double2hiint(x) & 0x7FFFFFFFu; }
// scale exponent e with |x| < 2^(e-1) for the largest |entry|, from its abs_hi word, so that
// the top digit stays within 64: exponent field - 1021 for a normal maximum, 0 for an
// all-zero vector, -1021 for a subnormal maximum, kNonFiniteScale for an infinity or a NaN (whose
// digits come out as zeros)
__device__ __forceinline__ int scale_exp_hi(unsigned int h) {
  if (h == 0) return 0;
  if (h >= 0x7FF00000u) return kNonFiniteScale;
  const int ex = (int)(h >> 20);
  return (ex == 0 ? 1 : ex) - 1021;
}

// sum of 64 in each of the NS - 1 low 7-bit fields (the balancing constant below)
__host__ __device__ constexpr unsigned long long balance_constant(int fields) {
  return fields == 0 ? 0ull : (64ull << (7 * (fields - 1))) + balance_constant(fields - 1);
}
constexpr unsigned long long kBalance = balance_constant(NS - 1);

// digits of x at scale 2^e (|x| < 2^(e-1)): X = rint(|x| 2^(7 NS - e)) <= 2^(7 NS - 1) is cut
// into balanced base-2^7 digits (|d| <= 64), d[0] the most significant, and the sign of
// x is applied to every digit.  Adding 64 to each of the NS - 1 low fields lets binary
// carries do the balancing: field k of Y = X + 64 sum_k 2^(7k) is f_k + c_(k-1) + 64
// mod 128 with carry c_k = [f_k + c_(k-1) >= 64], so d_k = field_k(Y) - 64, and the top
// digit is Y >> 7 (NS - 1) = f_(NS-1) + c_(NS-2)
__device__ __forceinline__ void digits(double x, int e, int d[NS]) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int ex = (int)((bits >> 52) & 0x7FF);
  unsigned long long X = 0;
  if (ex != 0) {
    const unsigned long long mant = (bits & ((1ull << 52) - 1)) | (1ull << 52);
    const int rs = 1075 - 7 * NS + e - ex;   // >= -2 because |x| < 2^(e-1)
    if (rs <= 0) X = mant << (-rs);
    else if (rs < 64) X = (mant + (1ull << (rs - 1))) >> rs;
  }
  const unsigned long long Y = X + kBalance;
  const unsigned int lo = (unsigned int)Y, hi = (unsigned int)(Y >> 32);
#pragma unroll
  for (int k = 0; k < NS - 1; ++k) {
    const int sh = 7 * k;
    unsigned int f;
    if (sh + 7 <= 32) f = (lo >> sh) & 127u;
    else if (sh >= 32) f = (hi >> (sh - 32)) & 127u;
    else f = __funnelshift_r(lo, hi, sh) & 127u;
    d[NS - 1 - k] = (int)f - 64;
  }
  d[0] = (int)(Y >> (7 * (NS - 1)));
  if (bits >> 63) {
#pragma unroll
    for (int k = 0; k < NS; ++k) d[k] = -d[k];
  }
}

// BF16 bit pattern of a small integer (|v| <= 256, exact): 1.5*2^23 + v keeps the float
// in [2^23, 2^24) where its spacing is 1, so adding v to the bit pattern and
// subtracting 1.5*2^23 gives (float)v exactly; the top 16 bits are the BF16 value
__device__ __forceinline__ unsigned int bf16_of_int(int v) {
  return __float_as_uint(__int_as_float(0x4B400000 + v) - 12582912.0f) >> 16;
}

static_assert(HSPLIT == 4, "the halves split the groups as [0, 4) and [4, NG)");

// int64 v (|v| < 2^62) times 2^p as an IEEE double: the conversion to nearest, then p added
// to the exponent field with one integer addition (0 when v = 0 or the result would
// fall below the normal range, far below the tile's FP64-class accuracy; infinity above
// the range; NaN where p holds a kNonFiniteScale)
__device__ __forceinline__ double ldexp_int(long long v, int p) {
  const double x = __ll2double_rn(v);
  const int hi = __double2hiint(x);
  const int e = ((hi >> 20) & 0x7FF) + p;
  if (p > kNonFiniteScale / 2) return __hiloint2double(0x7FF80000, 0);
  if (v == 0 || e <= 0) return 0.0;
  if (e >= 0x7FF) return __hiloint2double((hi & (int)0x80000000) | 0x7FF00000, 0);
  return __hiloint2double(hi + (int)((unsigned)p << 20), __double2loint(x));
}

// The double nearest to (h 2^SH + l) 2^p for the two exact halves of an element's group
// sums (|h|, |l| < 2^46, SH = 7 (NG - HSPLIT)): both are shifted down by s so that the
// sum fits in 62 bits (s <= 13; the bits of l dropped by the shift lie more than 8 bits
// below the sum's last significant bit), then one conversion.  One FP64-pipe operation
// per value instead of two conversions and an addition (GB300's FP64 pipe is narrow).
__device__ __forceinline__ double rebuild(long long h, long long l, int p) {
  constexpr int SH = 7 * (NG - HSPLIT);
  const unsigned long long ah = h < 0 ? 0ull - (unsigned long long)h : (unsigned long long)h;
  const int s = max(0, (64 - __clzll((long long)ah)) + SH - 61);
  const long long v = h * (1ll << (SH - s)) + (l >> s);
  return ldexp_int(v, p + s);
}

// ---------------------------------------------------------------------------
// scale pre-pass: ea[u][m] for rows of op(A), eb[u][j] for columns of op(B)
// ---------------------------------------------------------------------------
__global__ void oz_scale_kernel(GemmArgs g, int* ea, int* eb, int first) {
  const int u = blockIdx.y;
  if (g.active && !g.active[u]) return;
  const int n = g.n;
  const bool forA = blockIdx.x + first == 0;
  const zc* M = forA ? g.A.at(u) : g.B.at(u);
  const int op = forA ? g.opA : g.opB;
  int* out = (forA ? ea : eb) + (size_t)u * n;
  // "row-type" vectors are contiguous rows of the stored matrix:
  //   rows of op(A) with op N, columns of op(B) with op H
  const bool contiguous = forA ? (op == OP_N) : (op == OP_H);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (contiguous) {
    for (int r = warp; r < n; r += blockDim.x >> 5) {
      unsigned int v = 0;
      for (int k = lane; k < n; k += 32) {
        const zc x = M[(size_t)r * n + k];
        v = max(v, max(abs_hi(x.x), abs_hi(x.y)));
      }
      for (int off = 16; off > 0; off >>= 1) v = max(v, __shfl_down_sync(0xffffffffu, v, off));
      if (lane == 0) out[r] = scale_exp_hi(v);
    }
  } else {
    for (int c = threadIdx.x; c < n; c += blockDim.x) {
      unsigned int v = 0;
      for (int k = 0; k < n; ++k) {
        const zc x = M[(size_t)k * n + c];
        v = max(v, max(abs_hi(x.x), abs_hi(x.y)));
      }
      out[c] = scale_exp_hi(v);
    }
  }
}


// CL CTAs of a cluster are the CL column tiles of one 128-row tile (grid x is padded to a
// multiple of CL): each digitizes TM/CL of the A rows into every member's shared memory
//
// Warp roles: warps 0..7 produce digits (and run the epilogue), warp 8 issues the MMAs,
// warp 9 releases stages.  Handshakes are mbarriers only: full[s] collects one arrival
// per producer warp of every member (their stores into this member's stage s are
// done); mdone[s] the commit of this member's MMAs reading stage s; empty[s] one
// arrival per member, sent by that member's release warp once its mdone[s] phase has
// completed (its MMAs read A rows that this member wrote, so a producer may overwrite
// stage s only when every member's MMAs are done with it).
template <int CL>
__global__ void __launch_bounds__(NT + 64, 1) zgemm_oz_kernel(GemmArgs g, const int* ea, const int* eb, int* err,
                                                             int unit_alpha_beta) {
  const int u = blockIdx.z;
  if (g.active && !g.active[u]) return;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  uint64_t* bars = reinterpret_cast<uint64_t*>(base + 2 * STAGE);   // full[2], empty[2], done, mdone[2]
  uint64_t* full = bars;
  uint64_t* empty = bars + 2;
  uint64_t* done = bars + 4;
  uint64_t* mdone = bars + 5;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(base + 2 * STAGE + 56);
  __shared__ int s_fail;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n = g.n;
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TNC;
  const zc* A = g.A.at(u);
  const zc* B = g.B.at(u);
  const int* eA = ea + (size_t)u * n;
  const int* eB = eb + (size_t)u * n;

  if (tid == 0) {
    mbar_init(&full[0], 8 * CL);
    mbar_init(&full[1], 8 * CL);
    mbar_init(&empty[0], CL);
    mbar_init(&empty[1], CL);
    mbar_init(done, 1);
    mbar_init(&mdone[0], 1);
    mbar_init(&mdone[1], 1);
    s_fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;

  const uint32_t rank = cluster_ctarank();
  const uint32_t lbase = smem_u32(base);
  uint32_t rbase[CL];
#pragma unroll
  for (int r = 0; r < CL; ++r) rbase[r] = mapa_shared(lbase, (uint32_t)r);
  cluster_sync();   // every member is resident (barriers initialized) before remote stores

  const int nchunks = (n + KC - 1) / KC;
  // work items: threads 0..127 -- A row am (this member's share), AK consecutive
  // complex k from ak; threads 128..255 -- B column bn, 4 consecutive complex k from bk
  constexpr int AK = 16 / (128 / (TM / CL));   // 4 for CL = 4, 8 for CL = 2
  const bool is_a = tid < 128;
  const int it = tid & 127;
  const int am = (int)rank * (TM / CL) + it / (KC / AK), ak = (it % (KC / AK)) * AK;
  const int bn = it >> 2, bk = (it & 3) * 4;
  const int gm = m0 + am, gn = n0 + bn;
  const int escale = is_a ? ((gm < n) ? eA[gm] : 0) : ((gn < n) ? eB[gn] : 0);
  constexpr int NV = (AK > 4) ? AK : 4;   // complex entries held per thread
  zc rv[NV];
  auto load = [&](int c) {
    const int k0 = c * KC;
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      rv[j] = zmake(0.0, 0.0);
      if (is_a) {
        const int gk = k0 + ak + j;
        if (j < AK && gm < n && gk < n)
          rv[j] = (g.opA == OP_N) ? A[(size_t)gm * n + gk] : zconj(A[(size_t)gk * n + gm]);
      } else {
        const int gk = k0 + bk + j;
        if (j < 4 && gn < n && gk < n)
          rv[j] = (g.opB == OP_N) ? B[(size_t)gk * n + gn] : zconj(B[(size_t)gn * n + gk]);
      }
    }
  };
  if (warp == 8) {
    // ---------------- MMA warp: one elected lane issues, the others idle
    if (lane == 0) {
      for (int c = 0; c < nchunks; ++c) {
        const int s = c & 1;
        if (!mbar_wait_cluster(&full[s], (uint32_t)((c >> 1) & 1))) s_fail = 1;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t st_off = (uint32_t)(s * STAGE);
        // descriptors of slice 0 at k-step 0; the others differ by compile-time address
        // offsets, added to the start-address field (16-byte units, no carry out of it)
        const uint64_t da = sdesc64(lbase + st_off), db = sdesc64(lbase + st_off + NS * A_SLICE);
        const uint32_t first_chunk = (c == 0) ? 1u : 0u;
#pragma unroll
        for (int gsum = 0; gsum < NS; ++gsum) {        // scale group s + t
#pragma unroll
          for (int ps = 0; ps <= gsum; ++ps) {
            const int pt = gsum - ps;
#pragma unroll
            for (int ks = 0; ks < 2; ++ks) {           // K = 16 bf16 (32 bytes) per instruction
              const uint32_t acc = (ps == 0 && ks == 0) ? (first_chunk ^ 1u) : 1u;
              mma_bf16(tmem + (uint32_t)(gsum * NR),
                       da + (uint64_t)((ps * A_SLICE + ks * 32) >> 4),
                       db + (uint64_t)((pt * B_SLICE + ks * 32) >> 4), acc);
            }
          }
        }
        mma_commit(&mdone[s]);
      }
      mma_commit(done);
    }
  } else if (warp == 9) {
    // ---------------- release warp: once this member's MMAs of chunk c are done, one
    // arrival on empty[c & 1] of every member (only chunks whose stage is refilled)
    if (lane == 0) {
      for (int c = 0; c + 2 < nchunks; ++c) {
        const int s = c & 1;
        if (!mbar_wait(&mdone[s], (uint32_t)((c >> 1) & 1))) s_fail = 1;
#pragma unroll
        for (int r = 0; r < CL; ++r) mbar_arrive_remote(mapa_shared(smem_u32(&empty[s]), (uint32_t)r));
      }
    }
  } else {
  // ---------------- producer warps
  if (nchunks > 0) load(0);
  for (int c = 0; c < nchunks; ++c) {
    const int s = c & 1;
    if (c >= 2) {
      // every member's MMAs of chunk c-2 must be done with stage s (a timed-out wait is
      // recorded and the loop goes on)
      if (!mbar_wait_cluster(&empty[s], (uint32_t)(((c - 2) >> 1) & 1))) s_fail = 1;
    }
    const uint32_t st_off = (uint32_t)(s * STAGE);
    unsigned char* Bsl = base + st_off + NS * A_SLICE;
    zc cv[NV];
#pragma unroll
    for (int j = 0; j < NV; ++j) cv[j] = rv[j];
    if (c + 1 < nchunks) load(c + 1);
    unsigned int pr[NS][NV / 2], pi[NS][NV / 2];
#pragma unroll
    for (int j = 0; j < NV; ++j) {
      int dr[NS], di[NS];
      digits(cv[j].x, escale, dr);
      digits(cv[j].y, escale, di);
#pragma unroll
      for (int q = 0; q < NS; ++q) {
        if (j & 1) {
          pr[q][j >> 1] |= bf16_of_int(dr[q]) << 16;
          pi[q][j >> 1] |= bf16_of_int(di[q]) << 16;
        } else {
          pr[q][j >> 1] = bf16_of_int(dr[q]);
          pi[q][j >> 1] = bf16_of_int(di[q]);
        }
      }
    }
    if (is_a) {
      // A': real part -> columns ak.., imaginary part -> KC+ak..; into every member
      const uint32_t o_r = st_off + sw64(am, ak), o_i = st_off + sw64(am, KC + ak);
#pragma unroll
      for (int q = 0; q < NS; ++q) {
#pragma unroll
        for (int r = 0; r < CL; ++r) {
          if (AK == 8) {
            st_cluster_v4(rbase[r] + o_r + q * A_SLICE, pr[q][0], pr[q][1], pr[q][2], pr[q][3]);
            st_cluster_v4(rbase[r] + o_i + q * A_SLICE, pi[q][0], pi[q][1], pi[q][2], pi[q][3]);
          } else {
            st_cluster_v2(rbase[r] + o_r + q * A_SLICE, pr[q][0], pr[q][1]);
            st_cluster_v2(rbase[r] + o_i + q * A_SLICE, pi[q][0], pi[q][1]);
          }
        }
      }
    } else {
      // B'^T: row bn: [Re | -Im] of column n0+bn;  row TNC+bn: [Im | Re]; local only
      const uint32_t o1 = sw64(bn, bk), o2 = sw64(bn, KC + bk), o3 = sw64(TNC + bn, bk), o4 = sw64(TNC + bn, KC + bk);
#pragma unroll
      for (int q = 0; q < NS; ++q) {
        unsigned char* P = Bsl + q * B_SLICE;
        *reinterpret_cast<uint2*>(P + o1) = make_uint2(pr[q][0], pr[q][1]);
        *reinterpret_cast<uint2*>(P + o2) = make_uint2(pi[q][0] ^ 0x80008000u, pi[q][1] ^ 0x80008000u);
        *reinterpret_cast<uint2*>(P + o3) = make_uint2(pi[q][0], pi[q][1]);
        *reinterpret_cast<uint2*>(P + o4) = make_uint2(pr[q][0], pr[q][1]);
      }
    }
    // generic-proxy stores (local and remote) become visible to the tensor cores; one
    // arrival per warp on every member's full[s]
    asm volatile("fence.proxy.async.shared::cluster;" ::: "memory");
    __syncwarp();
    if (lane == 0) {
#pragma unroll
      for (int r = 0; r < CL; ++r) mbar_arrive_remote(mapa_shared(smem_u32(&full[s]), (uint32_t)r));
    }
  }
  // all MMAs of this member done (the MMA warp's last commit)
  if (nchunks > 0 && !mbar_wait(done, 0u)) s_fail = 1;
  }
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (s_fail) {
    if (tid == 0) raise_error(err, NEGF_ERR_TIMEOUT);
  } else if (warp < 8) {
    // ---- epilogue: warp w reads TMEM lanes 32*(w%4)..; complex columns 16*(w/4) .. +15, 8 at a time
    const int q = warp & 3, h = warp >> 2;
    const int row = m0 + 32 * q + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(32 * q) << 16);
    zc* D = g.D.at(u);
    const zc* Cm = g.C.p ? g.C.at(u) : nullptr;
    const int er = (row < n) ? eA[row] : 0;
#pragma unroll 1
    for (int cc = 0; cc < TNC / 16; ++cc) {
      const int j0 = (TNC / 2) * h + 8 * cc;   // complex column within the tile
      // group g (d = g + 2) weighs 2^(7 (NG-1-g)) relative to the last group; the two
      // halves [0, HSPLIT) and [HSPLIT, NG) are each exact in int64 below 2^53
      long long hre[8], him[8], lre[8], lim[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) { hre[j] = 0; him[j] = 0; lre[j] = 0; lim[j] = 0; }
#pragma unroll
      for (int d = 0; d < NG; ++d) {
        uint32_t vr[8], vi[8];
        TC_LD8(lane_base + (uint32_t)(d * NR + j0), vr);
        TC_LD8(lane_base + (uint32_t)(d * NR + TNC + j0), vi);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
        const int sh = (d < HSPLIT) ? 7 * (HSPLIT - 1 - d) : 7 * (NG - 1 - d);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const long long gr = ((long long)__float2int_rn(__uint_as_float(vr[j]))) << sh;
          const long long gi = ((long long)__float2int_rn(__uint_as_float(vi[j]))) << sh;
          if (d < HSPLIT) { hre[j] += gr; him[j] += gi; }
          else { lre[j] += gr; lim[j] += gi; }
        }
      }
      if (row < n) {
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int gcol = n0 + j0 + j;
          if (gcol < n) {
            const int p = er + eB[gcol] - 7 * (NS + 1);     // scale of the last group
            zc acc = zmake(rebuild(hre[j], lre[j], p), rebuild(him[j], lim[j], p));
            zc v;
            if (unit_alpha_beta) {
              // alpha = +-1, beta in {0, +-1}: signs only, one FP64 add
              v = (g.alpha.x < 0) ? zmake(-acc.x, -acc.y) : acc;
              if (Cm && g.beta.x != 0.0) {
                const zc cv = Cm[(size_t)row * n + gcol];
                v = (g.beta.x > 0) ? zadd(v, cv) : zsub(v, cv);
              }
            } else {
              v = zmul(g.alpha, acc);
              if (Cm) v = zadd(v, zmul(g.beta, Cm[(size_t)row * n + gcol]));
            }
            if (g.plus_identity && row == gcol) v.x += 1.0;
            D[(size_t)row * n + gcol] = v;
          }
        }
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512) : "memory");
  }
  cluster_sync();   // no member leaves while another may still address its shared memory
}

}  // namespace

// exact group sums need NS * 64 * 64 * 2n <= 2^24 (n <= 256 for NS <= 8)
bool oz_inkernel_supported(int n) { return n >= 16 && n <= 256; }

size_t oz_scratch_bytes(int n, int units) { return sizeof(int) * 2 * (size_t)n * units; }

cudaError_t zgemm_oz(const GemmArgs& g, void* scratch, int* err, cudaStream_t s) {
  if (g.units <= 0 || g.n <= 0) return cudaSuccess;
  if (!scratch) return cudaErrorInvalidValue;
  // cluster size: a tuning parameter (NEGF_OZ_CLUSTER = 2 or 4, default kCluster)
  const char* env = getenv("NEGF_OZ_CLUSTER");
  const int CL = (env && atoi(env) == 2) ? 2 : kCluster;
  cudaError_t e = once_per_device(INIT_OZ, [](int) {
    cudaError_t r = cudaFuncSetAttribute(zgemm_oz_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    if (r == cudaSuccess)
      r = cudaFuncSetAttribute(zgemm_oz_kernel<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM_BYTES);
    return r;
  });
  if (e != cudaSuccess) return e;
  int* ea = (int*)scratch;
  int* eb = ea + (size_t)g.n * g.units;
  oz_scale_kernel<<<dim3(2, g.units), 256, 0, s>>>(g, ea, eb, 0);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int unit_ab = ((g.alpha.y == 0.0 && (g.alpha.x == 1.0 || g.alpha.x == -1.0)) &&
                       (!g.C.p || (g.beta.y == 0.0 && (g.beta.x == 0.0 || g.beta.x == 1.0 || g.beta.x == -1.0))))
                          ? 1 : 0;
  const int tiles_n = (g.n + TNC - 1) / TNC;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((tiles_n + CL - 1) / CL * CL, (g.n + TM - 1) / TM, g.units);
  cfg.blockDim = dim3(NT + 64, 1, 1);
  cfg.dynamicSmemBytes = SMEM_BYTES;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CL;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  if (CL == 2) e = cudaLaunchKernelEx(&cfg, zgemm_oz_kernel<2>, g, (const int*)ea, (const int*)eb, err, unit_ab);
  else e = cudaLaunchKernelEx(&cfg, zgemm_oz_kernel<4>, g, (const int*)ea, (const int*)eb, err, unit_ab);
  if (e != cudaSuccess) return e;
  return cudaGetLastError();
}

}  // namespace negf

namespace negf {
namespace {
// The failure-detection self test: one thread waits, with the product kernels' bounded
// wait, on an mbarrier that nothing arrives on, so that the wait runs out after
// `limit_ns`; it then raises NEGF_ERR_TIMEOUT on the context's error word.  Nothing
// else (no bulk copy, no MMA, no other CTA) is in flight.
__global__ void wait_selftest_kernel(int* err, unsigned long long limit_ns) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) mbar_init(&bar, 1);
  __syncthreads();
  if (threadIdx.x == 0 && !mbar_wait_ns(&bar, 0u, limit_ns)) raise_error(err, NEGF_ERR_TIMEOUT);
}
}  // namespace

cudaError_t wait_selftest(int* err, unsigned long long limit_ns, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(err, limit_ns);
  return cudaGetLastError();
}
}  // namespace negf
