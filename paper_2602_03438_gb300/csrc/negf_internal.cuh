// Internal types shared by the translation units of libnegf (not part of the C ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <functional>
#include <string>
#include <vector>

#include "../../include/negf.h"

namespace negf {

// ---------------------------------------------------------------------------
// one-time set-up per GPU: kernel function attributes (dynamic shared memory size,
// occupancy queries) are properties of a device, so each device gets its own set-up,
// and several host threads may arrive at once.  `init(device)` runs with that device
// current, under a process-wide lock, at most once per (device, slot); a failed init
// is not recorded, so the next call retries it.
// ---------------------------------------------------------------------------
enum InitSlot { INIT_OZ = 0, INIT_TC, INIT_MLP, INIT_SMALL, INIT_OBC_SMALL, INIT_OZB, INIT_OZB_LO, INIT_OZB16,
                INIT_OZB16_LO, INIT_INV32, INIT_INV64, INIT_INV96, INIT_INV128,
                INIT_INVC_F256, INIT_INVC_D64, INIT_INVC_D128, INIT_NSLOT };
constexpr int kMaxDevices = 64;
cudaError_t once_per_device(int slot, const std::function<cudaError_t(int device)>& init);

constexpr int kSms = 152;   // multiprocessors of a GB300, for the rules that choose a kernel by rounds of them

// Launches that may start while the kernel before them on the stream drains: `k` calls
// pdl_begin() before it touches global memory (every thread, before any return), which waits
// until that kernel has finished.  What is saved is the launch latency and the set-up behind a
// kernel's last CTAs.  Product of n = 128 (two launches), us: 1024 blocks 516 -> 508, 152 99 ->
// 93, 16 27 -> 23.  No explicit trigger: letting the next kernel's CTAs in before the CTAs of
// this one exit cost 5% (1024 blocks 541, 64 x 1000 213 -> 235).
__device__ __forceinline__ void pdl_begin() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
}
template <class... P, class... A>
cudaError_t launch_pdl(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at = {};
  at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at.val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, k, P(args)...);
}

typedef double2 zc;   // complex128, interleaved (re, im)
typedef float2 cc;    // complex64

// ---------------------------------------------------------------------------
// complex helpers
// ---------------------------------------------------------------------------
__host__ __device__ __forceinline__ zc zmake(double r, double i) { return make_double2(r, i); }
__host__ __device__ __forceinline__ zc zadd(zc a, zc b) { return make_double2(a.x + b.x, a.y + b.y); }
__host__ __device__ __forceinline__ zc zsub(zc a, zc b) { return make_double2(a.x - b.x, a.y - b.y); }
__host__ __device__ __forceinline__ zc zmul(zc a, zc b) {
  return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x);
}
__host__ __device__ __forceinline__ zc zconj(zc a) { return make_double2(a.x, -a.y); }
__host__ __device__ __forceinline__ zc zscale(zc a, double s) { return make_double2(a.x * s, a.y * s); }
// |a|^2 (two FP64 operations, where hypot takes many on GB300's narrow FP64 pipe)
__host__ __device__ __forceinline__ double zabs2(zc a) { return fma(a.x, a.x, a.y * a.y); }
// a += b * c
__host__ __device__ __forceinline__ void zfma(zc& a, zc b, zc c) {
  a.x = fma(b.x, c.x, fma(-b.y, c.y, a.x));
  a.y = fma(b.x, c.y, fma(b.y, c.x, a.y));
}

// ---------------------------------------------------------------------------
// batched square-matrix operands: unit u's n x n row-major matrix at p + u*us, or, with
// inner > 1, at p + (u / inner) us + (u % inner) us2 (units that are (energy, partition)
// pairs of the partitioned sweeps)
// ---------------------------------------------------------------------------
struct BMat {
  zc* p;
  long long us;        // unit stride in elements; 0 => one matrix shared by all units
  int inner = 0;       // > 1: units form an (outer, inner) grid
  long long us2 = 0;   // stride of the inner index
  const long long* off = nullptr;   // device [units]: unit u at p + off[u] (the work list of an uneven batch)
  __host__ __device__ zc* at(int u) const {
    if (off) return p + off[u];
    return inner > 1 ? p + (long long)(u / inner) * us + (long long)(u % inner) * us2 : p + (long long)u * us;
  }
  // the plain layout (unit u at p + u us): kernels that are sensitive to the size of
  // their arguments get a specialization for it
  __host__ __device__ bool plain() const { return !off && inner <= 1; }
};

enum Op { OP_N = 0, OP_H = 2 };   // as stored / conjugate transpose

// one batched GEMM: D[u] = alpha op(A[u]) op(B[u]) + beta C[u]   (all n x n)
struct GemmArgs {
  BMat D, A, B, C;     // C.p may be NULL (beta ignored)
  int opA, opB;
  zc alpha, beta;
  int n;               // matrix size
  int units;           // batch
  const int* active;   // per unit, nullable: 0 => unit skipped
  int plus_identity = 0;   // sliced kernels: D += I after the rest (the residual I - M X in one product)
  // byte-digit product: op(A)'s scales and digit images are still in the scratch from the
  // previous product on the same op(A) (same layout, units, mask and variant), so that only
  // op(B)'s column scales are made before the product
  int reuse_a = 0;
};

// ---------------------------------------------------------------------------
// library context
// ---------------------------------------------------------------------------
// kernel classes of the timing facility (negf_profile_*)
enum KClass { K_GEMM_TC = 0, K_GEMM_F64 = 1, K_INV_F32 = 2, K_INV_F64 = 3, K_OTHER = 4, K_GEMM_OZ = 5, K_GEMM_OZ_LO = 6,
              K_NCLASS = 7 };

struct ProfRec {
  int cls;
  cudaEvent_t ev0, ev1;
  double flops, bytes;
};

struct Ctx {
  int device = 0;
  int num_sms = 0;
  void* ws = nullptr;           // device workspace
  size_t ws_bytes = 0;
  int* d_err = nullptr;         // device error word (worst negative code, as min)
  int* h_pinned = nullptr;      // small pinned host buffer for flags
  std::string last_error;
  long long launches = 0;       // kernels launched by this context
  bool prof = false;            // bracket GEMM / inverse launches with events
  std::vector<ProfRec> recs;
  std::vector<cudaEvent_t> pool;
  int oz_variant[513] = {0};    // tile variant of the sliced product per block size (autotuner)
  long long k_launches[K_NCLASS] = {};
  double k_ms[K_NCLASS] = {};
  double k_flops[K_NCLASS] = {};
  double k_bytes[K_NCLASS] = {};
  cudaEvent_t take_event() {
    if (!pool.empty()) { cudaEvent_t e = pool.back(); pool.pop_back(); return e; }
    cudaEvent_t e = nullptr;
    cudaEventCreate(&e);
    return e;
  }
};

// error word codes are stored as positive magnitudes with atomicMax
__device__ __forceinline__ void raise_error(int* err, int code) {
  if (err) atomicMax(err, -code);
}

// ---------------------------------------------------------------------------
// kernel launchers (return cudaGetLastError())
// ---------------------------------------------------------------------------
// FP64 complex GEMM on CUDA cores
cudaError_t zgemm_f64(const GemmArgs& g, cudaStream_t s);
// 3-term TF32-split complex GEMM on tcgen05 tensor cores (FP32 accumulate in TMEM)
cudaError_t zgemm_tc(const GemmArgs& g, int* err, cudaStream_t s);
// the byte-digit product with 5 digits per value (error ~2^-39 of the row x column norms),
// for products whose result is a small correction; scratch as for zgemm_ozt_variant
cudaError_t zgemm_ozt_lo(const GemmArgs& g, void* scratch, int* err, cudaStream_t s);
// one bounded device wait that runs out after limit_ns and raises NEGF_ERR_TIMEOUT on err
cudaError_t wait_selftest(int* err, unsigned long long limit_ns, cudaStream_t s);
bool tc_supported(int n);
// The scale exponent of a row or column with a NaN or an infinity in it (the others are below 1100):
// the sliced products' results of that row or column are NaN
constexpr int kNonFiniteScale = 1 << 20;
// FP64-class complex GEMM on the tensor cores by exact accumulation of digit slices, all
// digits made in the kernel (BF16, 16 <= n <= 256); `scratch` holds oz_scratch_bytes(n,
// units) bytes of per-row/column scales
cudaError_t zgemm_oz(const GemmArgs& g, void* scratch, int* err, cudaStream_t s);
bool oz_inkernel_supported(int n);
size_t oz_scratch_bytes(int n, int units);
// the same accuracy from byte digits (FP16, gemm_ozb.cu, 16 <= n <= 512), op(A)'s digits made
// once into `scratch` (ozt_scratch_bytes(n, units) bytes) and streamed to the tensor cores
bool oz_supported(int n);
size_t ozt_scratch_bytes(int n, int units);
// tile variants (the autotuner's choices): the default rule, tiles of 16 complex columns
// (n <= 128), tiles of 32 (n <= 128), tiles of 32 (any n).  The last two are one kernel: both
// numbers stand in saved tunings.
enum OzVariant { OZ_DEFAULT = 0, OZ_HALF = 1, OZ_PERSISTENT = 2, OZ_FULL = 3, OZ_NVARIANT = 4 };
bool oz_variant_supported(int n, int variant);
cudaError_t zgemm_ozt_variant(const GemmArgs& g, void* scratch, int* err, cudaStream_t s, int variant);

// X[u] = M[u]^{-1} by Gauss-Jordan with partial pivoting (first max |.| in row
// order).  FP64, or FP32 (`single` != 0) with the result written back in FP64.
// Work storage: in shared memory when it fits, otherwise `scratch` (units * n*n
// complex of the working precision).  status[u] (nullable, indexed status_base+u)
// gets NEGF_ERR_SINGULAR on an exactly zero pivot.
// `lent` (lent_bytes, nullable): 16-byte aligned scratch the caller does not need meanwhile.
// few: the mask is expected to be empty or nearly so.  With more units set the result is the same and
// the time above the launches' (n = 128, FP64: none of 384 set 6 us against 110, 4 414 : 429, 16
// 680 : 538, 400 8.9 : 5.7 ms).
cudaError_t zinv(BMat X, BMat M, int n, int units, const int* active, int single, void* scratch,
                 int32_t* status, cudaStream_t s, void* lent = nullptr, size_t lent_bytes = 0, bool few = false);
size_t zinv_scratch_bytes(int n, int units, int single);
bool f32_tiles(int n, int units, const int* active);   // the FP32 inverse runs better with scratch for tiles
// the inverse as column tiles, several CTAs per block (inv_tiles.cu; n <= 512); `scratch`
// holds zinv_tiles_bytes(n, units, single) bytes, 16-byte aligned
cudaError_t zinv_tiles(BMat X, BMat M, int n, int units, const int* active, int single, void* scratch, int32_t* status,
                       cudaStream_t s, bool few = false);
size_t zinv_tiles_bytes(int n, int units, int single);
// FP32, n <= 128: one CTA per block, the matrix in registers, no scratch
cudaError_t zinv_reg(BMat X, BMat M, int n, int units, const int* active, int32_t* status, cudaStream_t s);

// block i of unit u at p + u us + i is (a device's diagonal or off-diagonal output
// blocks, or a workspace slot array [i][u])
struct SBlk {
  zc* p;
  long long us, is;
  __host__ __device__ zc* at(int u, int i) const { return p + (long long)u * us + (long long)i * is; }
};
// ---------------------------------------------------------------------------
// one device of the (possibly uneven) batch, as the kernels see it
// ---------------------------------------------------------------------------
struct DevView {
  const zc* Hd;   // block 0 of this device
  const zc* Hu;
  const zc* Sd;   // NULL => identity
  const zc* Su;   // NULL => zero
  const double* E;
  double eta;
  int nb, b;
};

struct ScatView {
  const zc* sigR;        // NULL or this device's block 0 (energy 0)
  const zc* sigL;
  const double* scale;   // NULL or [ne][nb] of this device
  long long e_stride;    // elements between energies (0 = shared)
};

// one device of an uneven batch as the batched sweeps over (device, energy) units see it
struct UnitDev {
  DevView dv;
  ScatView sc;
  const zc *sigma_L, *sigma_R;   // this device's lead blocks (energy 0)
  const double *fL, *fR;         // this device's occupations (energy 0), nullable
};

// the open boundary of blocks of b <= kObcSmallB in one launch, one CTA per lead unit (u < U:
// the left lead of energy unit u, else the right lead of unit u - U), FP64: decimation to
// convergence, Newton polishing, Sigma.  Energy unit k is energy e0 + k of `dv`, or energy
// unit_e[k] of device udev[unit_dev[k]] when udev is given.  done, iters, nsteps, res
// ([2U]) as the batched path leaves them; gs_L, gs_R nullable.
constexpr int kObcSmallB = 16;
// A lead unit whose decimation blows up or whose Newton polishing diverges starts again: decimation at restart_widen times
// the broadening, then up to kRestartSteps Newton steps at its own.  Where eps is nearly singular
// on the way (condition 1e7 to 2e9 at eta = 1e-6), rounding leaves the surface function with a
// residual of 1e-4 to 1e-2, outside Newton's basin: the result was then wrong by 1e-5 to 1e-3,
// and which units it hit changed with every change of rounding (b = 128: 1 to 2 of 100 calls of
// 192 energies).  A larger broadening lowers the condition, and up to several times the
// lead's own (b = 128; wider for small blocks) its surface function lies inside the basin.  18
// such units of b = 8 to 128, one restart at 2, 3, 4, 5, 6 times the broadening: 52, 68, 62, 62,
// 60 of 72 trials solved; one of b = 16 wants 8 and more.
// A step counts as divergence where it multiplies the residual by kDiverged and more or makes
// it non-finite: a unit that ends at its rounding floor (|g| near 1 / eta) does not.
constexpr int kRestarts = 5, kRestartSteps = 6;
constexpr double kDiverged = 100.0;
__host__ __device__ constexpr double restart_widen(int k) { return k == 0 ? 3.0 : k == 1 ? 5.0 : k == 2 ? 2.0 : k == 3 ? 8.0 : 16.0; }
// Where more units are open than this, the cause is not a chance one (a broadening below what the
// decimation can resolve): one restart is tried, not all
__host__ __device__ constexpr int restart_many(int units) { return units / 16 > 4 ? units / 16 : 4; }
struct ObcSmall {
  DevView dv;
  int e0, U, b, max_iter;
  const UnitDev* udev;
  const int *unit_dev, *unit_e;
  double tol, target, accept;
  BMat sigma_L, sigma_R, gs_L, gs_R;
  int *done, *iters, *nsteps, *open;   // open: scratch of 2U
  double* res;
};
cudaError_t obc_small(const ObcSmall& a, cudaStream_t s);

// the whole forward and backward sweep of U energies of one device with blocks of b <= 16
// in one launch (one CTA per energy, FP64).  Ad [nb], Au/Al [nb-1], Sl/Sg [nb] hold the
// assembled blocks with unit stride b*b and block stride U*b*b; Y: the workspace of the
// products A_{i+1,i} g_i; gR, gL, gG: the diagonal blocks (left-connected on the forward
// sweep, overwritten with G, G^<, G^> on the backward sweep); Ru, Rl, Ll, Gl: the
// off-diagonal outputs G_{i,i+1}, G_{i+1,i}, G^<_{i+1,i}, G^>_{i+1,i} (p nullable);
// nk Keldysh kinds (0: retarded only, 1: G^<, 2: G^< and G^>).  status[u] (nullable) gets
// NEGF_ERR_SINGULAR on a zero pivot.
struct SmallSweep {
  int nb, b, U, nk;
  const zc *Ad, *Au, *Al, *Sl, *Sg;
  SBlk Y, gR, gL, gG, Ru, Rl, Ll, Gl;
  int32_t* status;
};
bool rgf_small_supported(int b, int mixed);
bool rgf_small_optional(int b, int mixed);   // runs step by step where the workspace is too small for the one launch
cudaError_t rgf_small_sweep(const SmallSweep& a, cudaStream_t s);

// Eq. (3) on a uniform grid: Y[e][i] = sum_{m=-M..M} w_m X[e-m][i] for i < nelem (element i
// of energy e at X + e ld + i), by a zero-padded FFT of size N = 2^conv_log2_size(ne, M)
// >= ne + M (N <= 8192).  w_dev: device [2M+1]; Wh: device scratch of
// conv_spectrum_bytes(ne, M) bytes for the kernel's spectrum.
int conv_log2_size(int ne, int M);
size_t conv_spectrum_bytes(int ne, int M);
cudaError_t energy_convolution(const zc* X, zc* Y, long long ld, int nelem, int ne, int M, const double* w_dev,
                               zc* Wh, cudaStream_t s);
// mixing step of the self-consistent loop over n elements: stats[0..2] (device) receive
// max|SLn - SL|, max|SGn - SG|, max(|SLn|, |SGn|); then SL, SG move by `mix` towards SLn,
// SGn and SR = (SG - SL) / 2
cudaError_t scba_mix(zc* SL, zc* SG, zc* SR, const zc* SLn, const zc* SGn, long long n, double mix, double* stats,
                     cudaStream_t s);

// sets the thread-local message returned by negf_last_error(NULL)
void negf_set_error_message(const char* msg);

}  // namespace negf
