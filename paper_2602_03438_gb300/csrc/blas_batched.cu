// Batched complex block kernels on CUDA cores: FP64 GEMM and Gauss-Jordan
// inversion (FP64 or FP32 arithmetic).  These are the building blocks of the
// RGF recursions (every step is a product or an inverse of b x b blocks,
// batched over independent energy points, Sec. II of the paper).
#include <atomic>
#include <mutex>

#include "negf_internal.cuh"

namespace negf {

namespace {
std::mutex g_init_mutex;
std::atomic<bool> g_init_done[kMaxDevices][INIT_NSLOT];
}  // namespace

cudaError_t once_per_device(int slot, const std::function<cudaError_t(int device)>& init) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices || slot < 0 || slot >= INIT_NSLOT) return cudaErrorInvalidValue;
  if (g_init_done[dev][slot].load(std::memory_order_acquire)) return cudaSuccess;
  std::lock_guard<std::mutex> lock(g_init_mutex);
  if (g_init_done[dev][slot].load(std::memory_order_relaxed)) return cudaSuccess;
  e = init(dev);
  if (e == cudaSuccess) g_init_done[dev][slot].store(true, std::memory_order_release);
  return e;
}

// ---------------------------------------------------------------------------
// FP64 complex GEMM: D = alpha op(A) op(B) + beta C, one thread per element of D (32
// consecutive elements of the row-major block per warp), operands straight from L1/L2.
// GB300's FP64 pipe takes 64 clocks per instruction and warp in each of an SM's four
// partitions, so the kernel is bound by 4 n FP64 FMAs per element and nothing else: the
// one load pair per 256 clocks of the pipe needs no staging, while square tiles spent
// the pipe on padding.  With C: 96 units of n = 40 206 -> 55 us, 20 of 100 473 -> 149 us, 512 of
// 8 71 -> 14 us, 128 of 128 2117 -> 1776 us (1.21 TFLOP/s), 8 of 256 1066 -> 882, 2 of 512 2117 ->
// 1751, one of 1000 8158 -> 6517 us.  Conjugated operands, which a warp reads with a stride of n, take
// the same time to 0.2% at every size from 8 to 1000 (the pipe hides them).
// ---------------------------------------------------------------------------
constexpr int kF64Threads = 128;
__global__ void __launch_bounds__(kF64Threads) zgemm_f64_kernel(GemmArgs g) {
  pdl_begin();
  const int u = blockIdx.y;
  if (g.active && !g.active[u]) return;
  const int n = g.n;
  const int e = blockIdx.x * kF64Threads + threadIdx.x;
  if (e >= n * n) return;
  const int r = e / n, c = e - r * n;
  const bool hA = g.opA != OP_N, hB = g.opB != OP_N;
  const zc* __restrict__ pa = g.A.at(u) + (hA ? r : (size_t)r * n);
  const zc* __restrict__ pb = g.B.at(u) + (hB ? (size_t)c * n : c);
  const int sa = hA ? n : 1, sb = hB ? 1 : n;
  // conjugation by the sign bit (a negation chosen at run time is an FP64 instruction)
  const int ma = hA ? (int)0x80000000 : 0, mb = hB ? (int)0x80000000 : 0;
  auto flip = [](double x, int m) { return __hiloint2double(__double2hiint(x) ^ m, __double2loint(x)); };
  zc acc = zmake(0.0, 0.0);
  int k = 0;
  for (; k + 4 <= n; k += 4) {
    zc a[4], b[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      a[q] = pa[(size_t)(k + q) * sa];
      b[q] = pb[(size_t)(k + q) * sb];
    }
#pragma unroll
    for (int q = 0; q < 4; ++q)
      zfma(acc, zmake(a[q].x, flip(a[q].y, ma)), zmake(b[q].x, flip(b[q].y, mb)));
  }
  for (; k < n; ++k) {
    const zc a = pa[(size_t)k * sa], b = pb[(size_t)k * sb];
    zfma(acc, zmake(a.x, flip(a.y, ma)), zmake(b.x, flip(b.y, mb)));
  }
  zc v = zmul(g.alpha, acc);
  if (g.C.p) v = zadd(v, zmul(g.beta, g.C.at(u)[e]));
  g.D.at(u)[e] = v;
}

cudaError_t zgemm_f64(const GemmArgs& g, cudaStream_t s) {
  if (g.units <= 0 || g.n <= 0) return cudaSuccess;
  const dim3 grid((unsigned)(((long long)g.n * g.n + kF64Threads - 1) / kF64Threads), g.units);
  launch_pdl(zgemm_f64_kernel, grid, kF64Threads, 0, s, g);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Gauss-Jordan inversion with partial pivoting, one CTA per unit.
//   for k: p = first argmax_{r>=k} |W[r][k]|; swap rows p,k; d = W[k][k];
//          row k <- row k / d with W[k][k] := 1/d;
//          for r != k: f = W[r][k]; row r <- row r - f * row k with W[r][k] := -f/d
//   finally undo the row swaps as column swaps in reverse order.
// ---------------------------------------------------------------------------
template <typename R> struct CT;
template <> struct CT<double> { typedef double2 T; };
template <> struct CT<float> { typedef float2 T; };

template <typename R>
__device__ __forceinline__ typename CT<R>::T cmk(R a, R b) {
  typename CT<R>::T v; v.x = a; v.y = b; return v;
}

constexpr int kInvThreads = 1024;

// Work split: thread t owns column c = t mod n and rows r0, r0 + rs, ... with
// r0 = t div n, rs = kInvThreads div n (threads beyond rs * n only help with the
// copies); the pivot row value of its column stays in a register during the update.
// One warp finds the pivot; the row interchange is folded into the update (the old
// row k is staged in shared memory); three barriers per step.
template <typename R, bool SMEM>
__global__ void __launch_bounds__(kInvThreads) zinv_kernel(BMat X, BMat M, int n, const int* active,
                                                           typename CT<R>::T* scratch, int32_t* status) {
  pdl_begin();
  typedef typename CT<R>::T C;
  const int u = blockIdx.x;
  if (active && !active[u]) return;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  C* W;
  unsigned char* tail;
  if (SMEM) {
    W = reinterpret_cast<C*>(smem_raw);
    tail = smem_raw + sizeof(C) * (size_t)n * (n + 1);
  } else {
    W = scratch + (size_t)u * n * (n + 1);
    tail = smem_raw;
  }
  C* prow = reinterpret_cast<C*>(tail);
  C* fcol = prow + n;
  C* krow = fcol + n;
  int* piv = reinterpret_cast<int*>(krow + n);
  __shared__ int s_p;
  __shared__ int s_sing;
  __shared__ C s_dinv;

  const int tid = threadIdx.x, lane = tid & 31;
  const zc* Min = M.at(u);
  const int nn = n * n;
  const int ld = n + 1;   // padded row stride: column reads hit distinct banks
  for (int i = tid; i < nn; i += kInvThreads) {
    const int r = i / n, c = i - r * n;
    const zc v = Min[i];
    W[(size_t)r * ld + c] = cmk<R>((R)v.x, (R)v.y);
  }
  if (tid == 0) s_sing = 0;
  const int rs = kInvThreads / n;           // >= 1 for n <= kInvThreads
  const int mc = tid % n, r0 = tid / n;     // this thread's column and first row
  const bool upd = r0 < rs;
  __syncthreads();

  for (int k = 0; k < n; ++k) {
    // -- pivot (warp 0): first row r >= k with the largest |W[r][k]|^2
    if (tid < 32) {
      R best = (R)-1;
      int bi = n;
      for (int r = k + lane; r < n; r += 32) {
        const C v = W[(size_t)r * ld + k];
        const R a = v.x * v.x + v.y * v.y;
        if (a > best) { best = a; bi = r; }
      }
#pragma unroll
      for (int off = 16; off > 0; off >>= 1) {
        const R ob = __shfl_down_sync(0xffffffffu, best, off);
        const int oi = __shfl_down_sync(0xffffffffu, bi, off);
        if (ob > best || (ob == best && oi < bi)) { best = ob; bi = oi; }
      }
      if (lane == 0) {
        if (!(best > (R)0)) { s_sing = 1; bi = k; }
        s_p = bi;
        piv[k] = bi;
        const C d = W[(size_t)bi * ld + k];
        const R den = d.x * d.x + d.y * d.y;
        s_dinv = (den > (R)0) ? cmk<R>(d.x / den, -d.y / den) : cmk<R>((R)0, (R)0);
      }
    }
    __syncthreads();
    const int p = s_p;
    // -- scaled pivot row (from row p), elimination factors of the swapped rows, and a
    //    copy of the old row k (which becomes row p)
    if (tid < n) {
      const C dinv = s_dinv;
      const C v = (tid == k) ? cmk<R>((R)1, (R)0) : W[(size_t)p * ld + tid];
      prow[tid] = cmk<R>(v.x * dinv.x - v.y * dinv.y, v.x * dinv.y + v.y * dinv.x);
      fcol[tid] = (tid == k) ? cmk<R>((R)0, (R)0) : W[(size_t)(tid == p ? k : tid) * ld + k];
      krow[tid] = W[(size_t)k * ld + tid];
    }
    __syncthreads();
    // -- rank-1 update: row k <- pivot row; row r <- (swapped) row r - f_r * pivot row,
    //    the pivot column entering as 0 (so that it becomes -f_r / d)
    if (upd) {
      const C pc = prow[mc];
      const C zero = cmk<R>((R)0, (R)0);
      const C kr = krow[mc];
      int r = r0;
      // four rows per iteration: their loads are independent and issued together (FP32
      // and n >= 96, where it measured faster; the FP64 matrix of b = 128 lives in
      // global scratch, and small blocks have few rows per thread)
      if (sizeof(R) == 4 && n >= 96)
      for (; r + 3 * rs < n; r += 4 * rs) {
        C w[4], f[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int rq = r + q * rs;
          w[q] = (mc == k) ? zero : ((rq == p) ? kr : W[(size_t)rq * ld + mc]);
          f[q] = fcol[rq];
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          const int rq = r + q * rs;
          C x = w[q];
          x.x = x.x - (f[q].x * pc.x - f[q].y * pc.y);
          x.y = x.y - (f[q].x * pc.y + f[q].y * pc.x);
          W[(size_t)rq * ld + mc] = (rq == k) ? pc : x;
        }
      }
      for (; r < n; r += rs) {
        const size_t i = (size_t)r * ld + mc;
        if (r == k) {
          W[i] = pc;
        } else {
          C w = (mc == k) ? zero : ((r == p) ? kr : W[i]);
          const C f = fcol[r];
          // (the product first: one rounding of the entry's own size; as two FMAs onto w, FP64 took a
          // third less time and had a third more error)
          w.x = w.x - (f.x * pc.x - f.y * pc.y);
          w.y = w.y - (f.x * pc.y + f.y * pc.x);
          W[i] = w;
        }
      }
    }
    __syncthreads();
  }
  // -- undo the row interchanges: swap columns k and piv[k], last pivot first
  for (int k = n - 1; k >= 0; --k) {
    const int p = piv[k];
    if (p != k) {
      for (int r = tid; r < n; r += kInvThreads) {
        C t = W[(size_t)r * ld + k];
        W[(size_t)r * ld + k] = W[(size_t)r * ld + p];
        W[(size_t)r * ld + p] = t;
      }
    }
    __syncthreads();
  }
  zc* Xo = X.at(u);
  for (int i = tid; i < nn; i += kInvThreads) {
    const int r = i / n, c = i - r * n;
    const C v = W[(size_t)r * ld + c];
    Xo[i] = zmake((double)v.x, (double)v.y);
  }
  if (tid == 0 && s_sing && status) status[u] = NEGF_ERR_SINGULAR;
}

static size_t inv_tail_bytes(int n, size_t csz) { return 3 * csz * n + sizeof(int) * n + 16; }
static const size_t kInvSmemMax = 200 * 1024;

size_t zinv_scratch_bytes(int n, int units, int single) {
  const size_t csz = single ? sizeof(float2) : sizeof(double2);
  if (csz * (size_t)n * (n + 1) + inv_tail_bytes(n, csz) <= kInvSmemMax) return 0;
  return csz * (size_t)n * (n + 1) * units;
}

template <typename R>
static cudaError_t launch_inv(BMat X, BMat M, int n, int units, const int* active, void* scratch,
                              int32_t* status, cudaStream_t s) {
  typedef typename CT<R>::T C;
  const size_t full = sizeof(C) * (size_t)n * (n + 1) + inv_tail_bytes(n, sizeof(C));
  if (full <= kInvSmemMax) {
    cudaError_t e = cudaFuncSetAttribute(zinv_kernel<R, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)full);
    if (e != cudaSuccess) return e;
    launch_pdl(zinv_kernel<R, true>, units, kInvThreads, full, s, X, M, n, active, nullptr, status);
  } else {
    if (!scratch) return cudaErrorInvalidValue;
    const size_t t = inv_tail_bytes(n, sizeof(C));
    launch_pdl(zinv_kernel<R, false>, units, kInvThreads, t, s, X, M, n, active, (C*)scratch, status);
  }
  return cudaGetLastError();
}

// FP64 inverses run as column tiles over several CTAs per block (inv_tiles.cu) where there is
// scratch for it and one CTA per block (a flat time up to kSms units, then the next round) would
// leave SMs idle or keep the matrix in global memory.  Measured (us, tiles : one CTA): n = 16, 152
// blocks 63 : 50, 160 63 : 92, 800 158 : 261; n = 20, 304 127 : 125; n = 24, 64 91 : 85, 160 101 : 159; n =
// 28, 8 104 : 108, 90 111 : 107, 304 203 : 209; n = 32, 64 117 : 133, 96 128 : 132, 120 131 : 133, 152 143 :
// 133, 160 144 : 256; n = 36, 96 153 : 169, 112 171 : 169, 152 199 : 170; n = 40, 1 137 : 206, 136 181 : 206,
// 152 208 : 207, 400 364 : 603; n = 44, 152 255 : 252; n = 48, 152 263 : 303; n = 64, 8 213 : 586, 152 412 :
// 588, 600 1200 : 2325; n = 72, 152 814 : 805, 400 1984 : 2391; n = 96, 60 675 : 1690, 300 2620 : 3363; n =
// 111, 152 1826 : 2597; n = 128, 16 558 : 3818, 400 6115 : 11459.
static bool f64_tiles(int n, int units) {
  if (n >= 40) return true;
  return (n >= 32 && units <= 96) || (n >= 16 && units > kSms);
}

// FP32 blocks up to 128 are inverted in registers, one CTA per block and SM, in rounds of 120 us
// at n = 128; tiles take about 100 us + 0.6 per block and win where the last round of the
// registers is far from full.  Measured (us, tiles : registers, with the refinement) at n = 97: 152
// blocks 445 : 385, 153 484 : 509, 230 644 : 637, 304 759 : 735, 305 796 : 854, 456 1083 : 1070, 460 1117 :
// 1186, 1024 2313 : 2330; n = 112: 152 469 : 414, 160 526 : 563, 260 718 : 723, 304 800 : 792, 400 1031 :
// 1077, 1024 2447 : 2516; n = 128: 153 565 : 619, 230 745 : 763, 304 873 : 858, 305 908 : 1009, 456 1245 :
// 1243, 512 1396 : 1475, 1024 2679 : 2700.  The line, drawn for n = 128, is within 1% of the better
// side for 97 to 127 too; n = 96, 512 alone 237 : 246.  A mask may leave few of the units.
bool f32_tiles(int n, int units, const int* active) {
  if (n <= 96 || n > 128) return n > 128;
  return !active && units > kSms && 500 + 3ll * units < 600ll * ((units + kSms - 1) / kSms);
}

cudaError_t zinv(BMat X, BMat M, int n, int units, const int* active, int single, void* scratch,
                 int32_t* status, cudaStream_t s, void* lent, size_t lent_bytes, bool few) {
  if (units <= 0 || n <= 0) return cudaSuccess;
  if (n <= 512 && (single ? f32_tiles(n, units, active) : f64_tiles(n, units))) {
    const size_t need = zinv_tiles_bytes(n, units, single);
    void* t = lent_bytes >= need ? lent : (zinv_scratch_bytes(n, units, single) >= need ? scratch : nullptr);
    if (t) return zinv_tiles(X, M, n, units, active, single, t, status, s, few);
  }
  if (single && n <= 128) return zinv_reg(X, M, n, units, active, status, s);
  if (single) return launch_inv<float>(X, M, n, units, active, scratch, status, s);
  return launch_inv<double>(X, M, n, units, active, scratch, status, s);
}

}  // namespace negf
