// Batched Gauss-Jordan inverse with partial pivoting in FP32 (the first stage of the refined
// inverse, row a7 of the hot path) and in FP64: spread over several CTAs per block, and below
// for FP32 blocks up to 128 by one CTA with the matrix in registers.
//
// The n x n matrix lives in global scratch (L2 resident) as column tiles of TW columns (16 in
// FP32, 8 in FP64).  Launch k applies panel k to every other tile and factors panel k + 1:
// one CTA per (tile, unit) with one thread per matrix row, the row's TW entries in
// registers.  A masked launch covers up to kMaskedUnits units at a time, each CTA walking
// the units of its column, so that a mask with few units set costs few CTAs.
//   * In-place Gauss-Jordan leaves in the panel's own columns the matrix C that takes any
//     other column y to its new value: with y_K the panel's pivot rows, row r becomes
//     y_r + C_r y_K, and a pivot row C_r y_K.  So a tile's update is a rank-TW product
//     with C read row by row (coalesced) and y_K broadcast from shared memory.
//   * The CTA whose tile is the next panel runs that panel's pivot steps on its registers
//     right after its update, while the other CTAs update the rest.
//   * Rows never move: each row keeps the position it would hold after the interchanges
//     (the pivot is the first largest |.|^2 in position order), and the last kernel
//     gathers X[i][c] = W[row at position i][position of row c].
// What bounds it: the n sequential pivot steps, each about 250 instructions (FP64: some 50 of
// the FP64 pipe at 64 clocks) of every warp of one CTA and one barrier, plus a launch per
// panel; the updates (W and C from L2) run beside them.  Measured (GB300) against one CTA
// per block: FP32 n = 512, 16 blocks 27.9 -> 0.88 ms; n = 256, 8 blocks 4.01 -> 0.27 ms; FP64
// n = 128, one block 3.81 -> 0.43 ms, 400 blocks 11.5 -> 6.1 ms; n = 512, 2 blocks 223 -> 5.4 ms.
// TW: a row's entries fit in 32 registers, and the update reads C once for TW columns.
#include <algorithm>
#include <type_traits>

#include "negf_internal.cuh"

namespace negf {

namespace {

constexpr int kMaxN = 512;
constexpr int kMaskedUnits = 96;

template <typename R> struct Tr;
template <> struct Tr<float> { typedef float2 C; static constexpr int TW = 16; };
template <> struct Tr<double> { typedef double2 C; static constexpr int TW = 8; };

// A unit's matrix in 16-byte vectors of V entries of one row (two FP32 columns side by side,
// one FP64), rows consecutive, so that a warp's rows of one vector are one segment; an odd
// last FP32 column alone.
template <typename C>
__device__ __forceinline__ size_t elem(int n, int r, int j) {
  if (sizeof(C) == 16) return (size_t)j * n + r;
  const size_t base = (size_t)(j >> 1) * 2 * n;
  return ((j | 1) < n) ? base + 2 * (size_t)r + (j & 1) : base + r;
}

// entries of one unit's matrix, even so that the vectors stay 16-byte aligned
__host__ __device__ __forceinline__ size_t tile_stride(int n) { return ((size_t)n * n + 1) & ~(size_t)1; }

template <typename C>
__device__ __forceinline__ C czero() {
  C z;
  z.x = z.y = 0;
  return z;
}
__device__ __forceinline__ void cfma(float2& a, float2 b, float2 c) {   // a += b c
  a.x = fmaf(b.x, c.x, fmaf(-b.y, c.y, a.x));
  a.y = fmaf(b.x, c.y, fmaf(b.y, c.x, a.y));
}
__device__ __forceinline__ void cfma(double2& a, double2 b, double2 c) { zfma(a, b, c); }

// the vector of a row that starts at column j (a multiple of V), zeros past n
template <typename C>
__device__ __forceinline__ void load_vec(const C* W, int n, int r, int j, C* v) {
  constexpr int V = 16 / sizeof(C);
#pragma unroll
  for (int x = 0; x < V; ++x) v[x] = czero<C>();
  if (j + V <= n) *reinterpret_cast<uint4*>(v) = *reinterpret_cast<const uint4*>(W + elem<C>(n, r, j));
  else if (j < n) v[0] = W[elem<C>(n, r, j)];
}
template <typename C>
__device__ __forceinline__ void store_vec(C* W, int n, int r, int j, const C* v) {
  constexpr int V = 16 / sizeof(C);
  if (j + V <= n) *reinterpret_cast<uint4*>(W + elem<C>(n, r, j)) = *reinterpret_cast<const uint4*>(v);
  else if (j < n) W[elem<C>(n, r, j)] = v[0];
}

// Ordering key of a pivot candidate's |.|^2 (hi, lo): the bits of a non-negative float or
// double, with 1 for zero and NaN, 0 for rows that are not candidates
__device__ __forceinline__ void pivot_key(bool cand, float v, unsigned int& hi, unsigned int& lo) {
  hi = cand ? (v > 0.f ? __float_as_uint(v) + 1u : 1u) : 0u;
  lo = 0u;
}
__device__ __forceinline__ void pivot_key(bool cand, double v, unsigned int& hi, unsigned int& lo) {
  const long long b = __double_as_longlong(v);
  const bool pos = b > 0 && b <= 0x7FF0000000000000ll;
  hi = cand ? (pos ? (unsigned int)(b >> 32) + 1u : 1u) : 0u;
  lo = (cand && pos) ? (unsigned int)b : 0u;
}
// the warp's largest (hi, lo), and whether this lane holds it
template <typename R>
__device__ __forceinline__ bool warp_max(unsigned int& hi, unsigned int& lo) {
  const unsigned int h = __reduce_max_sync(0xffffffffu, hi);
  bool is = hi == h;
  hi = h;
  if (sizeof(R) == 8) {
    const unsigned int l = __reduce_max_sync(0xffffffffu, is ? lo : 0u);
    is = is && lo == l;
    lo = l;
  }
  return is;
}

// 1 / d (0 for 0)
__device__ __forceinline__ float2 cinv(float2 d) {
  const float den = d.x * d.x + d.y * d.y;
  if (!(den > 1e-36f && den < 1e36f))   // 1 / den may be out of range
    return (den > 0.f) ? make_float2(d.x / den, -d.y / den) : make_float2(0.f, 0.f);
  const float r = __frcp_rn(den);
  return make_float2(d.x * r, -d.y * r);
}
__device__ __forceinline__ double2 cinv(double2 d) {
  const double den = zabs2(d);
  if (!(den > 0.0)) return make_double2(0.0, 0.0);
  if (den < 1e-290) return make_double2(d.x / den, -d.y / den);   // 1 / den may overflow
  const double r = 1.0 / den;                                     // one division on the FP64 pipe
  return make_double2(d.x * r, -d.y * r);
}

// double <-> float with integers: the conversion instructions take a warp 64 clocks of the
// FP64 pipe each.  Round to nearest even; what is not a normal number in both formats
// (or rounds up past one) goes through the cast.
__device__ __forceinline__ float to_f32(double v) {
  const unsigned int hi = (unsigned int)__double2hiint(v), lo = (unsigned int)__double2loint(v);
  const unsigned int e = (hi >> 20) & 0x7ffu;
  if (((hi & 0x7fffffffu) | lo) == 0u) return __uint_as_float(hi);
  if (e - 897u >= 253u) return (float)v;
  const unsigned int m = __funnelshift_l(lo, (hi & 0x7fffffffu) - (896u << 20), 3);
  const unsigned int rest = lo << 3;   // the 29 bits cut off, at the top
  const unsigned int up = (rest > 0x80000000u || (rest == 0x80000000u && (m & 1u))) ? 1u : 0u;
  return __uint_as_float((m + up) | (hi & 0x80000000u));
}
__device__ __forceinline__ double to_f64(float v) {
  const unsigned int b = __float_as_uint(v), a = b & 0x7fffffffu;
  if (a == 0u) return __hiloint2double((int)b, 0);
  if (a - 0x800000u >= 0x7f000000u) return (double)v;
  return __hiloint2double((int)(((a >> 3) + (896u << 20)) | (b & 0x80000000u)), (int)(a << 29));
}

__device__ __forceinline__ void narrow(float2& a, zc v) { a = make_float2(to_f32(v.x), to_f32(v.y)); }
__device__ __forceinline__ void narrow(double2& a, zc v) { a.x = v.x; a.y = v.y; }
__device__ __forceinline__ zc widen(float2 v) { return zmake(to_f64(v.x), to_f64(v.y)); }
__device__ __forceinline__ zc widen(double2 v) { return zmake(v.x, v.y); }

template <typename C>
struct TileInv {
  BMat M, X;
  int n, units;
  const int* active;
  C* W;              // [unit][tile_stride(n)]
  uint16_t* pos;     // [2][unit][n]: positions of the rows, alternating between the panels
  int32_t* status;
};

// panel = -1: take the tiles from M and factor panel 0; else apply that panel and factor
// the next one
template <typename R, int NT>
__device__ __forceinline__ void tile_step(const TileInv<typename Tr<R>::C>& g, int panel, int t, int u) {
  typedef typename Tr<R>::C C;
  constexpr int TW = Tr<R>::TW, V = 16 / sizeof(C);
  const int n = g.n, r = threadIdx.x, lane = r & 31, warp = r >> 5;
  const bool has = r < n;
  C* W = g.W + (size_t)u * tile_stride(n);
  const size_t prow_n = (size_t)g.units * n;
  const uint16_t* pos_in = g.pos + (size_t)(panel & 1) * prow_n + (size_t)u * n;
  __shared__ __align__(16) C yk[TW][TW];
  __shared__ __align__(16) C prow[2][NT / 32][TW + V];   // the warps' candidates: row and 1 / pivot
  __shared__ uint2 s_key[2][NT / 32];
  __shared__ int s_pos[2][NT / 32];

  alignas(16) C a[TW];
  int mypos = r;
  if (panel < 0) {
    const zc* Min = g.M.at(u);
#pragma unroll
    for (int c = 0; c < TW; ++c) {
      const int j = t * TW + c;
      a[c] = czero<C>();
      if (has && j < n) narrow(a[c], Min[(size_t)r * n + j]);
    }
  } else {
    int pj = -1;   // this row's pivot step within the panel
    if (has) {
      mypos = pos_in[r];
      pj = mypos - panel * TW;
    }
#pragma unroll
    for (int c = 0; c < TW; c += V) {
#pragma unroll
      for (int x = 0; x < V; ++x) a[c + x] = czero<C>();
      if (has) load_vec<C>(W, n, r, t * TW + c, a + c);
    }
    if (pj >= 0 && pj < TW) {
#pragma unroll
      for (int c = 0; c < TW; ++c) {
        yk[pj][c] = a[c];
        a[c] = czero<C>();
      }
    }
    if ((panel + 1) * TW > n) {   // a ragged last panel: no pivot rows past n
      for (int i = n - panel * TW + r / TW; i < TW; i += NT / TW) yk[i][r % TW] = czero<C>();
    }
    __syncthreads();
    // FP64: the panel's share summed apart and added once, so that an entry takes one rounding of its
    // own size per panel and not 16.  Error over the condition number, rms of 40 blocks, against one
    // CTA per block with the product formed first: n = 40 5.7e-17 : 6.4e-17, 64 7.3e-17 : 9.0e-17, 100
    // 7.9e-17 : 1.24e-16, 128 9.1e-17 : 1.21e-16.  Time 3% to 7% (n = 128, 400 blocks 5.73 -> 6.11 ms).
    constexpr bool APART = sizeof(R) == 8;
    C sum[APART ? TW : 1];
    if (APART) {
#pragma unroll
      for (int c = 0; c < (APART ? TW : 1); ++c) sum[c] = czero<C>();
    }
#pragma unroll 2
    for (int k = 0; k < TW; k += V) {
      alignas(16) C f[V];
#pragma unroll
      for (int x = 0; x < V; ++x) f[x] = czero<C>();
      if (has) load_vec<C>(W, n, r, panel * TW + k, f);
#pragma unroll
      for (int x = 0; x < V; ++x)
#pragma unroll
        for (int c = 0; c < TW; c += V) {
          alignas(16) C y[V];
          *reinterpret_cast<uint4*>(y) = *reinterpret_cast<const uint4*>(&yk[k + x][c]);
#pragma unroll
          for (int z = 0; z < V; ++z) cfma(APART ? sum[APART ? c + z : 0] : a[c + z], f[x], y[z]);
        }
    }
    if (APART) {
#pragma unroll
      for (int c = 0; c < (APART ? TW : 1); ++c) {
        a[c].x += sum[c].x;
        a[c].y += sum[c].y;
      }
    }
  }

  if (t == panel + 1) {
    // ---- the pivot steps of this panel
    const int k0 = t * TW, w = min(TW, n - k0);
    bool sing = false;
    // a rolled loop: the entries rotate by one column per step, so that a[0] is always the
    // pivot column, and are back in place after TW steps
#pragma unroll 1
    for (int j = 0; j < TW; ++j) {
      if (j >= w) {   // a ragged last panel: only the rotation
        const C z = a[0];
#pragma unroll
        for (int c = 1; c < TW; ++c) a[c - 1] = a[c];
        a[TW - 1] = z;
        continue;
      }
      const int k = k0 + j, bf = j & 1;
      // the largest |.|^2 among the rows at positions >= k, first in position order
      const R v = a[0].x * a[0].x + a[0].y * a[0].y;
      const bool cand = has && mypos >= k;
      unsigned int hi, lo;
      pivot_key(cand, v, hi, lo);
      const bool top = warp_max<R>(hi, lo);
      C own;   // FP64: every row's 1 / entry beside the search (472 against 488 us at n = 128); only the pivot's is used
      if constexpr (sizeof(R) == 8) own = cinv(a[0]);
      int p = __reduce_min_sync(0xffffffffu, (cand && top) ? mypos : kMaxN);
      // every warp publishes its own candidate with its row; one barrier, then all
      // threads pick the winner (the buffers alternate: a warp may be one step ahead)
      if (cand && mypos == p) {
        s_key[bf][warp] = make_uint2(hi, lo);
        s_pos[bf][warp] = p;
#pragma unroll
        for (int c = 0; c < TW; ++c) prow[bf][warp][c] = a[c];
        if constexpr (sizeof(R) == 8) prow[bf][warp][TW] = own;
      } else if (lane == 0 && hi == 0u) {
        s_key[bf][warp] = make_uint2(0u, 0u);
        s_pos[bf][warp] = kMaxN;
      }
      __syncthreads();
      const uint2 wk = (lane < NT / 32) ? s_key[bf][lane] : make_uint2(0u, 0u);
      const int wp = (lane < NT / 32) ? s_pos[bf][lane] : kMaxN;
      hi = wk.x;
      lo = wk.y;
      const bool wtop = warp_max<R>(hi, lo);
      p = __reduce_min_sync(0xffffffffu, wtop ? wp : kMaxN);
      const int ww = __ffs(__ballot_sync(0xffffffffu, wtop && wp == p)) - 1;
      const C* pr = prow[bf][ww];
      C di;
      if constexpr (sizeof(R) == 8) di = pr[TW];
      else di = cinv(pr[0]);   // 0: a zero column, where the first row left stands in for the pivot
      if (hi <= 1u) sing = true;
      const bool win = has && mypos == p;
      // row r -= f (pivot row / d), with -f / d in place of the pivot column; the pivot
      // row becomes itself / d
      const C f = a[0];
      C h;
      h.x = f.y * di.y - f.x * di.x;
      h.y = -(f.x * di.y + f.y * di.x);
      if (win) {
#pragma unroll
        for (int c = 1; c < TW; ++c) a[c] = czero<C>();
        h = di;
      }
#pragma unroll
      for (int c = 0; c < TW; c += V) {
        alignas(16) C y[V];
        *reinterpret_cast<uint4*>(y) = *reinterpret_cast<const uint4*>(pr + c);
#pragma unroll
        for (int z = 0; z < V; ++z) {
          if (c + z > 0) {
            cfma(a[c + z], h, y[z]);
            a[c + z - 1] = a[c + z];
          }
        }
      }
      a[TW - 1] = h;
      if (mypos == k) mypos = p;   // the row at position k takes the pivot row's place
      if (win) mypos = k;
    }
    if (has) g.pos[(size_t)((panel + 1) & 1) * prow_n + (size_t)u * n + r] = (uint16_t)mypos;
    if (sing && r == 0 && g.status) g.status[u] = NEGF_ERR_SINGULAR;
  }
  if (has) {
#pragma unroll
    for (int c = 0; c < TW; c += V) store_vec<C>(W, n, r, t * TW + c, a + c);
  }
}

// the next unit with its flag set, from u on in steps of `stride` (g.units: none left).  Flags are
// read a warp at a time.
template <typename C>
__device__ __forceinline__ int next_unit(const TileInv<C>& g, int u, int stride) {
  if (!g.active) return min(u, g.units);
  for (; u < g.units; u += 32 * stride) {
    const long long x = u + (long long)(threadIdx.x & 31) * stride;
    const unsigned int m = __ballot_sync(0xffffffffu, x < g.units && g.active[x]);
    if (m) return u + (__ffs(m) - 1) * stride;
  }
  return g.units;
}

// The CTAs that factor the next panel come first (blockIdx.y = 0): where the launch takes more
// than one round of the SMs, no pivot chain starts in the last.  FP32 n = 512, 16 blocks 1298 ->
// 880 us; n = 200, 40 blocks 339 -> 276; FP64 n = 128, 64 blocks 1330 -> 1025.
template <typename R, int NT>
__global__ void __launch_bounds__(NT, (sizeof(R) == 4 ? 1024 : 512) / NT)
    inv_tile_kernel(TileInv<typename Tr<R>::C> g, int panel) {
  pdl_begin();
  const int t = (panel + 1 + (int)blockIdx.y) % (int)gridDim.y, stride = gridDim.x;
  if (t == panel) return;
  for (int u = next_unit(g, blockIdx.x, stride); u < g.units; u = next_unit(g, u + stride, stride)) {
    tile_step<R, NT>(g, panel, t, u);
    __syncthreads();   // the next unit of this CTA reuses the shared buffers
  }
}

// X[i][c] = W[row at position i][position of row c], in FP64, for rows i0 .. i0 + rows - 1 (<= 16)
constexpr int kOutRows = 16;
template <typename C>
__device__ __forceinline__ void gather_rows(const TileInv<C>& g, int last_panel, int u, int i0, int rows) {
  const int n = g.n;
  __shared__ int s_pos[kMaxN];
  __shared__ int s_row[kOutRows];
  const uint16_t* pos = g.pos + (size_t)(last_panel & 1) * g.units * n + (size_t)u * n;
  for (int r = threadIdx.x; r < n; r += blockDim.x) {
    const int p = pos[r];
    s_pos[r] = p;
    if (p >= i0 && p < i0 + rows) s_row[p - i0] = r;
  }
  __syncthreads();
  const C* W = g.W + (size_t)u * tile_stride(n);
  zc* X = g.X.at(u);
  for (int i = threadIdx.x >> 5; i < rows; i += (int)blockDim.x >> 5) {
    const int r = s_row[i];
#pragma unroll 4
    for (int c = threadIdx.x & 31; c < n; c += 32) X[(size_t)(i0 + i) * n + c] = widen(W[elem<C>(n, r, s_pos[c])]);
  }
  __syncthreads();
}

template <typename C>
__global__ void __launch_bounds__(256) inv_gather_kernel(TileInv<C> g, int last_panel) {
  pdl_begin();
  const int i0 = blockIdx.x * kOutRows, stride = gridDim.y;
  for (int u = next_unit(g, blockIdx.y, stride); u < g.units; u = next_unit(g, u + stride, stride))
    gather_rows(g, last_panel, u, i0, min(kOutRows, g.n - i0));
}

// Up to 16 tiles and few units: one cluster per unit with a CTA per tile, cluster barriers in
// place of the launches (the tiles still pass through L2).  No gaps between the panels, and
// a mask without units costs one launch; but a waiting cluster holds its SMs, so more units
// run better as launches.  Measured (GB300, us, launches : cluster): FP64 n = 128, no unit of
// 384 set 110 : 6, 4 units 429 : 414, 16 538 : 680, 400 5745 : 8883; n = 64, 8 214 : 203.  FP32 n =
// 140, 4 148 : 137, 8 148 : 165; n = 200, 4 209 : 198, 8 210 : 231; n = 256, 4 267 : 252, 16 291 : 322.
constexpr int kMaxCluster = 16;   // more than 8 CTAs: opted in, every GPC has room for them
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release;\n\tbarrier.cluster.wait.acquire;" ::: "memory");
}
template <typename R, int NT>
__global__ void __launch_bounds__(NT, (sizeof(R) == 4 ? 1024 : 512) / NT)
    inv_cluster_kernel(TileInv<typename Tr<R>::C> g, int tiles) {
  pdl_begin();
  const int t = blockIdx.x, per = (g.n + gridDim.x - 1) / gridDim.x, i0 = t * per, stride = gridDim.y;
  // (the CTAs of a cluster share blockIdx.y and so take the same units)
  for (int u = next_unit(g, blockIdx.y, stride); u < g.units; u = next_unit(g, u + stride, stride)) {
    for (int panel = -1; panel < tiles; ++panel) {
      if (t < tiles && t != panel) tile_step<R, NT>(g, panel, t, u);
      cluster_barrier();
    }
    gather_rows(g, tiles - 1, u, i0, max(0, min(per, g.n - i0)));
  }
}

template <typename R, int NT>
cudaError_t launch_tiles(const TileInv<typename Tr<R>::C>& g, int tiles, int rows, cudaStream_t s) {
  for (int panel = -1; panel < tiles; ++panel) {
    cudaError_t e = launch_pdl(inv_tile_kernel<R, NT>, dim3(rows, tiles), NT, 0, s, g, panel);
    if (e != cudaSuccess) return e;
  }
  return launch_pdl(inv_gather_kernel<typename Tr<R>::C>, dim3((g.n + kOutRows - 1) / kOutRows, rows), 256, 0, s, g, tiles - 1);
}

template <typename R, int NT>
cudaError_t launch_cluster(const TileInv<typename Tr<R>::C>& g, int tiles, int rows, int slot, cudaStream_t s) {
  const int cs = tiles <= 8 ? 8 : kMaxCluster;
  cudaError_t e = once_per_device(slot, [](int) {
    return cudaFuncSetAttribute(inv_cluster_kernel<R, NT>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(cs, rows);
  cfg.blockDim = dim3(NT);
  cfg.stream = s;
  cudaLaunchAttribute at[2] = {};
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, inv_cluster_kernel<R, NT>, g, tiles);
}

template <typename R, int NT>
cudaError_t launch_inv(const TileInv<typename Tr<R>::C>& g, int tiles, int rows, bool cluster, int slot, cudaStream_t s) {
  if constexpr (NT <= kMaxCluster * Tr<R>::TW)
    if (cluster) return launch_cluster<R, NT>(g, tiles, rows, slot, s);
  return launch_tiles<R, NT>(g, tiles, rows, s);
}

template <typename R>
cudaError_t run(BMat X, BMat M, int n, int units, const int* active, bool few, void* scratch, int32_t* status,
                cudaStream_t s) {
  typedef typename Tr<R>::C C;
  TileInv<C> g;
  g.M = M; g.X = X; g.n = n; g.units = units; g.active = active;
  g.W = (C*)scratch;
  g.pos = (uint16_t*)(g.W + tile_stride(n) * units);
  g.status = status;
  const int tiles = (n + Tr<R>::TW - 1) / Tr<R>::TW;
  const int rows = std::min(units, active ? kMaskedUnits : 65535);
  const bool cluster = active ? few : units * (tiles <= 8 ? 1 : 2) <= 8;
  if constexpr (sizeof(R) == 8) {
    if (n <= 64) return launch_inv<R, 64>(g, tiles, rows, cluster, INIT_INVC_D64, s);
    if (n <= 128) return launch_inv<R, 128>(g, tiles, rows, cluster, INIT_INVC_D128, s);
  } else if (n <= 128) {
    return launch_tiles<R, 128>(g, tiles, rows, s);
  }
  return n <= 256 ? launch_inv<R, 256>(g, tiles, rows, cluster, INIT_INVC_F256, s)
                  : launch_inv<R, 512>(g, tiles, rows, false, 0, s);
}

// ---------------------------------------------------------------------------
// n <= 128 in FP32: the same elimination by one CTA per block with the matrix in registers.
// Thread (r, q) holds 32 columns of row r: panels q and q + NQ of 16 columns each (NQ groups of
// NR threads, cyclic so that consecutive panels belong to different groups).  The owner of
// the next panel brings it up to date first, runs its 16 pivot steps (one barrier of its warps
// per step) and publishes it, while the other groups still apply the panel before to all their
// columns; the owner's own second panel catches up one round later.
// A published panel is its columns C and the rows' positions; each group takes the pivot rows
// y_K of its own columns through shared memory.  No launch per panel and no pass over the
// matrix: bound by the chain of n pivot steps, some 1000 clocks each (two barriers' worth of
// exchange, one reciprocal, 15 column updates); the next step's search starts among them.
// Measured (GB300, us, against column tiles): one block of 128 120 : 114, 64 blocks 123 : 137, 152
// 125 : 187, 200 241 : 213, 304 244 : 259, 512 476 : 406, 1024 830 : 818; 512 of 96 246 : 237; 600 of 64
// 77 : 115; 1000 of 32 36 : 62.  At 96 rows two CTAs per SM pay for a few spilled registers (344 with one).
// ---------------------------------------------------------------------------
constexpr int RC = 32;        // columns per thread
constexpr int RP = 16;        // columns per panel
constexpr int RCS = RP + 1;   // row stride of C (banks)

template <int NR>
constexpr size_t reg_smem() {   // the whole matrix on the way in and out; between them C of 3 panels, y_K of 2
  const size_t mat = sizeof(float2) * NR * (NR + 1), ck = sizeof(float2) * (3 * NR * RCS + 2 * RP * NR);
  return mat > ck ? mat : ck;
}

// a barrier of one group's NR threads
template <int NR>
__device__ __forceinline__ void group_barrier(int q) {
  if (NR == 32) __syncwarp();
  else if (q == 0) asm volatile("bar.sync 1, %0;" ::"n"(NR) : "memory");
  else if (q == 1) asm volatile("bar.sync 2, %0;" ::"n"(NR) : "memory");
  else if (NR > 64 && q == 2) asm volatile("bar.sync 3, %0;" ::"n"(NR) : "memory");
  else if (NR > 96) asm volatile("bar.sync 4, %0;" ::"n"(NR) : "memory");
}

// The pivot steps of the panel in b (w of its 16 columns are in range, k0: the first), by the NR
// threads of its group
template <int NR>
__device__ __forceinline__ void reg_pivots(float2 (&b)[RP], int k0, int w, bool has, int q, int wq, int lane, int& mypos,
                                           bool& sing, float2 (*prow)[NR / 32][RP + 2], unsigned int (*s_key)[4],
                                           int (*s_pos)[4]) {
  constexpr int NW = NR / 32;
  unsigned int hi, lo;
  bool cand = has && mypos >= k0;
  pivot_key(cand, b[0].x * b[0].x + b[0].y * b[0].y, hi, lo);
  bool top = warp_max<float>(hi, lo);
  float2 own = cinv(b[0]);   // every row's, beside the search: only the pivot's is used
#pragma unroll 1
  for (int j = 0; j < w; ++j) {   // entries rotate by one column per step, as above
    const int k = k0 + j, bf = j & 1;
    bool lead = cand && top;
    const unsigned int tops = __ballot_sync(0xffffffffu, lead);
    if (tops & (tops - 1u)) {   // (the same for the whole warp) several: the first in position order
      const int first = __reduce_min_sync(0xffffffffu, lead ? mypos : kMaxN);
      lead = lead && mypos == first;
    }
    if (lead) {
      s_key[bf][wq] = hi;
      s_pos[bf][wq] = mypos;
#pragma unroll
      for (int c = 0; c < RP; c += 2)
        *reinterpret_cast<float4*>(&prow[bf][wq][c]) = make_float4(b[c].x, b[c].y, b[c + 1].x, b[c + 1].y);
      prow[bf][wq][RP] = own;
    } else if (lane == 0 && hi == 0u) {
      s_key[bf][wq] = 0u;
      s_pos[bf][wq] = kMaxN;
    }
    group_barrier<NR>(q);
    int ww = 0, p;
    if (NW == 1) {
      p = s_pos[bf][0];
    } else {
      const uint4 kk = *reinterpret_cast<const uint4*>(s_key[bf]);
      const int4 pp = *reinterpret_cast<const int4*>(s_pos[bf]);
      const unsigned int ks[4] = {kk.x, kk.y, kk.z, kk.w};
      const int ps[4] = {pp.x, pp.y, pp.z, pp.w};
      hi = ks[0];
      p = ps[0];
#pragma unroll
      for (int x = 1; x < NW; ++x)
        if (ks[x] > hi || (ks[x] == hi && ps[x] < p)) {
          hi = ks[x];
          p = ps[x];
          ww = x;
        }
    }
    const float2* pr = prow[bf][ww];
    const float2 di = pr[RP];
    if (hi <= 1u) sing = true;
    const bool win = has && mypos == p;
    const float2 f = b[0];
    float2 h = make_float2(f.y * di.y - f.x * di.x, -(f.x * di.y + f.y * di.x));
    if (win) {
#pragma unroll
      for (int c = 1; c < RP; ++c) b[c] = make_float2(0.f, 0.f);
      h = di;
    }
    if (mypos == k) mypos = p;
    if (win) mypos = k;
    // the next pivot column first: its search runs while the others are updated
    cfma(b[1], h, pr[1]);
    cand = has && mypos > k;
    pivot_key(cand, b[1].x * b[1].x + b[1].y * b[1].y, hi, lo);
    top = warp_max<float>(hi, lo);
    b[0] = b[1];
#pragma unroll
    for (int c = 2; c < RP; c += 2) {
      const float4 y = *reinterpret_cast<const float4*>(pr + c);
      cfma(b[c], h, make_float2(y.x, y.y));
      b[c - 1] = b[c];
      cfma(b[c + 1], h, make_float2(y.z, y.w));
      b[c] = b[c + 1];
    }
    b[RP - 1] = h;
    own = cinv(b[0]);
  }
#pragma unroll 1
  for (int j = w; j < RP; ++j) {   // a short panel: the rest of the rotation
    const float2 z = b[0];
#pragma unroll
    for (int c = 1; c < RP; ++c) b[c - 1] = b[c];
    b[RP - 1] = z;
  }
}

// b += C y_K over the w columns of a panel
template <int NR>
__device__ __forceinline__ void reg_update(float2 (&b)[RP], const float2* fr, const float2* y0, int w) {
#pragma unroll 1
  for (int k = 0; k < w; ++k) {
    const float2 f = fr[k];
#pragma unroll
    for (int c = 0; c < RP; c += 2) {
      const float4 y = *reinterpret_cast<const float4*>(y0 + k * NR + c);
      cfma(b[c], f, make_float2(y.x, y.y));
      cfma(b[c + 1], f, make_float2(y.z, y.w));
    }
  }
}

// NR: rows rounded up to 32
template <int NR>
__global__ void __launch_bounds__(NR * (NR / RC), NR == 128 ? 1 : NR == 96 ? 2 : NR == 64 ? 4 : 8)
    inv_reg_kernel(BMat X, BMat M, int n, const int* active, int32_t* status) {
  pdl_begin();
  const int u = blockIdx.x;
  if (active && !active[u]) return;
  constexpr int NQ = NR / RC, NT = NR * NQ, NW = NR / 32;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float2* S = reinterpret_cast<float2*>(smem_raw);   // [NR][NR + 1]: the whole matrix, in and out
  float2* Cs = S;                                    // [3][NR][RCS]: panels' columns
  float2* yk = S + 3 * NR * RCS;                     // [2][RP][NR]: their pivot rows
  __shared__ __align__(16) float2 prow[2][NW][RP + 2];   // the warps' candidates: row and 1 / pivot
  __shared__ __align__(16) unsigned int s_key[2][4];
  __shared__ __align__(16) int s_pos[2][4];
  __shared__ int pos[2][NR], rowof[NR];
  const int tid = threadIdx.x, lane = tid & 31;
  const int r = tid % NR, q = tid / NR, wq = (tid % NR) >> 5;   // (a warp has one q)
  const bool has = r < n;
  const int drow = NT / n, dcol = NT - drow * n;   // NT entries further on

  {
    const zc* Min = M.at(u);
    const int nn = n * n;
    constexpr int B = 8;   // loads in flight per thread
    int rr = tid / n, c = tid - rr * n;
    for (int i = tid; i < nn; i += B * NT) {
      zc v[B];
#pragma unroll
      for (int x = 0; x < B; ++x)
        if (i + x * NT < nn) v[x] = Min[i + x * NT];
#pragma unroll
      for (int x = 0; x < B; ++x) {
        if (i + x * NT < nn) narrow(S[rr * (NR + 1) + c], v[x]);
        rr += drow;
        c += dcol;
        if (c >= n) { c -= n; ++rr; }
      }
    }
  }
  __syncthreads();
  float2 a[2][RP];   // panels q and q + NQ
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < RP; ++c) {
      const int j = (h * NQ + q) * RP + c;
      a[h][c] = (has && j < n) ? S[r * (NR + 1) + j] : make_float2(0.f, 0.f);
    }
  int mypos = r;
  bool sing = false;
  __syncthreads();

  const int np = (n + RP - 1) / RP;
  // The owner of the next panel updates it alone on the SM: the other groups' updates fill the
  // gaps of its pivot steps, which are the longer part.
  auto owner_first = [&](bool owner) {
    if (NQ == 1) return;
    if (owner) asm volatile("bar.arrive 5, %0;" ::"n"(NT) : "memory");
    else asm volatile("bar.sync 5, %0;" ::"n"(NT) : "memory");
  };
  // panel p's pivot steps, its columns and the positions to shared memory.  C has 3 buffers: the
  // owner of p reads panel p - 1 until it passes the barrier of p + 1.
  auto factor = [&](float2 (&b)[RP], int p) {
    reg_pivots<NR>(b, p * RP, min(RP, n - p * RP), has, q, wq, lane, mypos, sing, prow, s_key, s_pos);
    float2* cp = Cs + ((p % 3) * NR + r) * RCS;
#pragma unroll
    for (int c = 0; c < RP; ++c) cp[c] = b[c];
    pos[p & 1][r] = mypos;
  };
  auto apply = [&](float2 (&b)[RP], int h, int p) {   // panel p to this group's panel h
    reg_update<NR>(b, Cs + ((p % 3) * NR + r) * RCS, yk + (p & 1) * RP * NR + (h * NQ + q) * RP, min(RP, n - p * RP));
  };
  if (q == 0) factor(a[0], 0);
#pragma unroll
  for (int half = 0; half < 2; ++half) {
#pragma unroll 1
    for (int pq = 0; pq < NQ; ++pq) {
      const int p = half * NQ + pq;
      if (p >= np) break;
      __syncthreads();   // panel p is out
      const int nq = pq + 1 < NQ ? pq + 1 : 0;   // the group of panel p + 1
      const bool next = p + 1 < np;
      if (next && q != nq) owner_first(false);
      // the owner's other panel takes panel p - 1 now (a single group left nothing behind)
      if (NQ > 1 && q == pq && p > 0) apply(a[1 - half], 1 - half, p - 1);
      mypos = pos[p & 1][r];
      const int pj = mypos - p * RP;
      if (has && pj >= 0 && pj < RP) {   // a pivot row of this panel: y_K
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          if (q == pq && h == half) continue;
          float2* yp = yk + ((p & 1) * RP + pj) * NR + (h * NQ + q) * RP;
#pragma unroll
          for (int c = 0; c < RP; ++c) {
            yp[c] = a[h][c];
            a[h][c] = make_float2(0.f, 0.f);
          }
        }
      }
      group_barrier<NR>(q);
      if (q == nq && next) {
        if (half == 0 && pq + 1 < NQ) {
          apply(a[0], 0, p);
          owner_first(true);
          factor(a[0], p + 1);
        } else {
          apply(a[1], 1, p);
          owner_first(true);
          factor(a[1], p + 1);
        }
      } else {
        if (!(q == pq && half == 0)) apply(a[0], 0, p);
        if (!(q == pq && half == 1)) apply(a[1], 1, p);
      }
    }
  }
  // X[i][c] = W[row at position i][position of row c], through shared memory
  __syncthreads();
  if (q == 0 && has) rowof[mypos] = r;
  __syncthreads();
#pragma unroll
  for (int h = 0; h < 2; ++h)
#pragma unroll
    for (int c = 0; c < RP; ++c) {
      const int j = (h * NQ + q) * RP + c;
      if (has && j < n) S[mypos * (NR + 1) + rowof[j]] = a[h][c];
    }
  __syncthreads();
  zc* Xo = X.at(u);
  {
    int rr = tid / n, c = tid - rr * n;
#pragma unroll 4
    for (int i = tid; i < n * n; i += NT) {
      Xo[i] = widen(S[rr * (NR + 1) + c]);
      rr += drow;
      c += dcol;
      if (c >= n) { c -= n; ++rr; }
    }
  }
  if (sing && r == 0 && status) status[u] = NEGF_ERR_SINGULAR;   // (a panel's group saw it)
}

template <int NR>
cudaError_t launch_reg(BMat X, BMat M, int n, int units, const int* active, int32_t* status, cudaStream_t s) {
  const int slot = NR == 128 ? INIT_INV128 : NR == 96 ? INIT_INV96 : NR == 64 ? INIT_INV64 : INIT_INV32;
  cudaError_t e = once_per_device(slot, [](int) {
    return cudaFuncSetAttribute(inv_reg_kernel<NR>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)reg_smem<NR>());
  });
  if (e != cudaSuccess) return e;
  return launch_pdl(inv_reg_kernel<NR>, units, NR * (NR / RC), reg_smem<NR>(), s, X, M, n, active, status);
}

}  // namespace

cudaError_t zinv_reg(BMat X, BMat M, int n, int units, const int* active, int32_t* status, cudaStream_t s) {
  if (units <= 0 || n <= 0) return cudaSuccess;
  if (n > 128) return cudaErrorInvalidValue;
  return n <= 32 ? launch_reg<32>(X, M, n, units, active, status, s)
       : n <= 64 ? launch_reg<64>(X, M, n, units, active, status, s)
       : n <= 96 ? launch_reg<96>(X, M, n, units, active, status, s) : launch_reg<128>(X, M, n, units, active, status, s);
}

size_t zinv_tiles_bytes(int n, int units, int single) {
  return (tile_stride(n) * (single ? sizeof(float2) : sizeof(double2)) + 2 * (size_t)n * sizeof(uint16_t)) * units;
}

cudaError_t zinv_tiles(BMat X, BMat M, int n, int units, const int* active, int single, void* scratch, int32_t* status,
                       cudaStream_t s, bool few) {
  if (units <= 0 || n <= 0) return cudaSuccess;
  if (!scratch || n > kMaxN) return cudaErrorInvalidValue;
  return single ? run<float>(X, M, n, units, active, few, scratch, status, s)
                : run<double>(X, M, n, units, active, few, scratch, status, s);
}

}  // namespace negf
