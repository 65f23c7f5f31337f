// Batched FP32 Gauss-Jordan inverse with partial pivoting, spread over several CTAs per
// block: the FP32 stage of the refined inverse (row a7 of the hot path).
//
// The n x n matrix lives in global scratch (L2 resident) as column tiles of kTW columns.
// Launch k applies panel k to every other tile and factors panel k + 1: one CTA per (tile,
// unit) with one thread per matrix row, the row's kTW entries in registers.
//   * In-place Gauss-Jordan leaves in the panel's own columns the matrix C that takes any
//     other column y to its new value: with y_K the panel's pivot rows, row r becomes
//     y_r + C_r y_K, and a pivot row C_r y_K.  So a tile's update is a rank-kTW product
//     with C read row by row (coalesced) and y_K broadcast from shared memory.
//   * The CTA whose tile is the next panel runs that panel's pivot steps on its registers
//     right after its update, while the other CTAs update the rest.
//   * Rows never move: each row keeps the position it would hold after the interchanges
//     (the pivot is the first largest |.|^2 in position order), and the last kernel
//     gathers X[i][c] = W[row at position i][position of row c].
// What bounds it: the n sequential pivot steps, each about 250 instructions of every warp
// of one CTA and one barrier, plus a launch per panel; the updates (FP32 FMAs, W and C from
// L2) run beside them.  Measured (GB300): n = 512, 16 blocks 27.9 -> 1.22 ms; n = 256, 8
// blocks 4.01 -> 0.28 ms; n = 128, 512 blocks 0.91 -> 0.46 ms against one CTA per block.
// kTW = 16: a row's entries fit in 32 registers (two CTAs of 512 threads per SM), and the
// update reads C once for 16 columns.
#include "negf_internal.cuh"

namespace negf {

namespace {

constexpr int kTW = 16;         // columns per tile
constexpr int kTQ = kTW / 2;    // column pairs per tile
constexpr int kMaxN = 512;

// Element (r, j) of a unit's matrix: pairs of columns side by side, rows consecutive (a
// warp's rows of one pair are one 512-byte segment); an odd last column alone.
__device__ __forceinline__ size_t elem(int n, int r, int j) {
  const size_t base = (size_t)(j >> 1) * 2 * n;
  return ((j | 1) < n) ? base + 2 * (size_t)r + (j & 1) : base + r;
}

// elements of one unit's matrix, even so that the column pairs stay 16-byte aligned
__host__ __device__ __forceinline__ size_t tile_stride(int n) { return ((size_t)n * n + 1) & ~(size_t)1; }

__device__ __forceinline__ void cfma(float2& a, float2 b, float2 c) {   // a += b c
  a.x = fmaf(b.x, c.x, fmaf(-b.y, c.y, a.x));
  a.y = fmaf(b.x, c.y, fmaf(b.y, c.x, a.y));
}

__device__ __forceinline__ void load_pair(const float2* W, int n, int r, int j, float2& v0, float2& v1) {
  v0 = v1 = make_float2(0.f, 0.f);
  if (j + 1 < n) {
    const float4 t = *reinterpret_cast<const float4*>(W + elem(n, r, j));
    v0 = make_float2(t.x, t.y);
    v1 = make_float2(t.z, t.w);
  } else if (j < n) {
    v0 = W[elem(n, r, j)];
  }
}

struct TileInv {
  BMat M, X;
  int n, units;
  const int* active;
  float2* W;         // [unit][tile_stride(n)]
  uint16_t* pos;     // [2][unit][n]: positions of the rows, alternating between the panels
  int32_t* status;
};

// panel = -1: take the tiles from M and factor panel 0; else apply that panel and factor
// the next one
template <int NT>
__global__ void __launch_bounds__(NT, 1024 / NT) inv_tile_kernel(TileInv g, int panel) {
  const int t = blockIdx.x, u = blockIdx.y;
  if (t == panel || (g.active && !g.active[u])) return;
  const int n = g.n, r = threadIdx.x, lane = r & 31, warp = r >> 5;
  const bool has = r < n;
  float2* W = g.W + (size_t)u * tile_stride(n);
  const size_t prow_n = (size_t)g.units * n;
  const uint16_t* pos_in = g.pos + (size_t)(panel & 1) * prow_n + (size_t)u * n;
  __shared__ float4 yk[kTW][kTQ];
  __shared__ float4 prow[2][NT / 32][kTQ];
  __shared__ unsigned int s_key[2][NT / 32];
  __shared__ int s_pos[2][NT / 32];

  float2 a[kTW];
  int mypos = r;
  if (panel < 0) {
    const zc* Min = g.M.at(u);
#pragma unroll
    for (int c = 0; c < kTW; ++c) {
      const int j = t * kTW + c;
      a[c] = make_float2(0.f, 0.f);
      if (has && j < n) {
        const zc v = Min[(size_t)r * n + j];
        a[c] = make_float2((float)v.x, (float)v.y);
      }
    }
  } else {
    int pj = -1;   // this row's pivot step within the panel
    if (has) {
      mypos = pos_in[r];
      pj = mypos - panel * kTW;
    }
#pragma unroll
    for (int q = 0; q < kTQ; ++q) {
      a[2 * q] = a[2 * q + 1] = make_float2(0.f, 0.f);
      if (has) load_pair(W, n, r, t * kTW + 2 * q, a[2 * q], a[2 * q + 1]);
    }
    if (pj >= 0 && pj < kTW) {
#pragma unroll
      for (int q = 0; q < kTQ; ++q) {
        yk[pj][q] = make_float4(a[2 * q].x, a[2 * q].y, a[2 * q + 1].x, a[2 * q + 1].y);
        a[2 * q] = a[2 * q + 1] = make_float2(0.f, 0.f);
      }
    }
    if ((panel + 1) * kTW > n) {   // a ragged last panel: no pivot rows past n
      for (int i = n - panel * kTW + r / kTQ; i < kTW; i += NT / kTQ) yk[i][r % kTQ] = make_float4(0.f, 0.f, 0.f, 0.f);
    }
    __syncthreads();
#pragma unroll 2
    for (int q = 0; q < kTQ; ++q) {
      float2 c0 = make_float2(0.f, 0.f), c1 = c0;
      if (has) load_pair(W, n, r, panel * kTW + 2 * q, c0, c1);
#pragma unroll
      for (int x = 0; x < kTQ; ++x) {
        const float4 y0 = yk[2 * q][x];
        cfma(a[2 * x], c0, make_float2(y0.x, y0.y));
        cfma(a[2 * x + 1], c0, make_float2(y0.z, y0.w));
      }
#pragma unroll
      for (int x = 0; x < kTQ; ++x) {
        const float4 y1 = yk[2 * q + 1][x];
        cfma(a[2 * x], c1, make_float2(y1.x, y1.y));
        cfma(a[2 * x + 1], c1, make_float2(y1.z, y1.w));
      }
    }
  }

  if (t == panel + 1) {
    // ---- the pivot steps of this panel
    const int k0 = t * kTW, w = min(kTW, n - k0);
    bool sing = false;
    // a rolled loop (unrolled, its straight-line code is fetched once per launch and the
    // fetch bounds it): the entries rotate by one column per step, so that a[0] is always
    // the pivot column, and are back in place after kTW steps
#pragma unroll 1
    for (int j = 0; j < kTW; ++j) {
      if (j >= w) {   // a ragged last panel: only the rotation
        const float2 z = a[0];
#pragma unroll
        for (int c = 1; c < kTW; ++c) a[c - 1] = a[c];
        a[kTW - 1] = z;
        continue;
      }
      const int k = k0 + j, bf = j & 1;
      // the largest |.|^2 among the rows at positions >= k, first in position order.  Keys:
      // the float's bits + 1 (1 for zero and NaN), 0 for the other rows
      const float v = a[0].x * a[0].x + a[0].y * a[0].y;
      const bool cand = has && mypos >= k;
      const unsigned int key = cand ? (v > 0.f ? __float_as_uint(v) + 1u : 1u) : 0u;
      unsigned int m = __reduce_max_sync(0xffffffffu, key);
      int p = __reduce_min_sync(0xffffffffu, (cand && key == m) ? mypos : kMaxN);
      // every warp publishes its own candidate with its row; one barrier, then all
      // threads pick the winner (the buffers alternate: a warp may be one step ahead)
      if (cand && mypos == p) {
        s_key[bf][warp] = m;
        s_pos[bf][warp] = p;
#pragma unroll
        for (int x = 0; x < kTQ; ++x)
          prow[bf][warp][x] = make_float4(a[2 * x].x, a[2 * x].y, a[2 * x + 1].x, a[2 * x + 1].y);
      } else if (lane == 0 && m == 0u) {
        s_key[bf][warp] = 0u;
        s_pos[bf][warp] = kMaxN;
      }
      __syncthreads();
      const unsigned int wk = (lane < NT / 32) ? s_key[bf][lane] : 0u;
      const int wp = (lane < NT / 32) ? s_pos[bf][lane] : kMaxN;
      m = __reduce_max_sync(0xffffffffu, wk);
      p = __reduce_min_sync(0xffffffffu, wk == m ? wp : kMaxN);
      const int ww = __ffs(__ballot_sync(0xffffffffu, wk == m && wp == p)) - 1;
      const float4* pr = prow[bf][ww];
      const float4 y0 = pr[0];
      const float den = y0.x * y0.x + y0.y * y0.y;
      // 1 / pivot (0: a zero column, where the first row left stands in for the pivot)
      const float2 di = (den > 0.f) ? make_float2(y0.x / den, -y0.y / den) : make_float2(0.f, 0.f);
      if (m <= 1u) sing = true;
      const bool win = has && mypos == p;
      // row r -= f (pivot row / d), with -f / d in place of the pivot column; the pivot
      // row becomes itself / d
      const float2 f = a[0];
      float2 h = make_float2(f.y * di.y - f.x * di.x, -(f.x * di.y + f.y * di.x));
      if (win) {
#pragma unroll
        for (int c = 1; c < kTW; ++c) a[c] = make_float2(0.f, 0.f);
        h = di;
      }
#pragma unroll
      for (int x = 0; x < kTQ; ++x) {
        const float4 y = x ? pr[x] : y0;
        if (x) {
          cfma(a[2 * x], h, make_float2(y.x, y.y));
          a[2 * x - 1] = a[2 * x];
        }
        cfma(a[2 * x + 1], h, make_float2(y.z, y.w));
        a[2 * x] = a[2 * x + 1];
      }
      a[kTW - 1] = h;
      if (mypos == k) mypos = p;   // the row at position k takes the pivot row's place
      if (win) mypos = k;
    }
    if (has) g.pos[(size_t)((panel + 1) & 1) * prow_n + (size_t)u * n + r] = (uint16_t)mypos;
    if (sing && r == 0 && g.status) g.status[u] = NEGF_ERR_SINGULAR;
  }
  if (has) {
#pragma unroll
    for (int q = 0; q < kTQ; ++q) {
      const int j = t * kTW + 2 * q;
      if (j + 1 < n)
        *reinterpret_cast<float4*>(W + elem(n, r, j)) =
            make_float4(a[2 * q].x, a[2 * q].y, a[2 * q + 1].x, a[2 * q + 1].y);
      else if (j < n)
        W[elem(n, r, j)] = a[2 * q];
    }
  }
}

// X[i][c] = W[row at position i][position of row c], in FP64
constexpr int kOutRows = 16;
__global__ void __launch_bounds__(256) inv_gather_kernel(TileInv g, int last_panel) {
  const int u = blockIdx.y;
  if (g.active && !g.active[u]) return;
  const int n = g.n, i0 = blockIdx.x * kOutRows;
  __shared__ int s_pos[kMaxN];
  __shared__ int s_row[kOutRows];
  const uint16_t* pos = g.pos + (size_t)(last_panel & 1) * g.units * n + (size_t)u * n;
  for (int r = threadIdx.x; r < n; r += 256) {
    const int p = pos[r];
    s_pos[r] = p;
    if (p >= i0 && p < i0 + kOutRows) s_row[p - i0] = r;
  }
  __syncthreads();
  const float2* W = g.W + (size_t)u * tile_stride(n);
  zc* X = g.X.at(u);
  const int rows = min(kOutRows, n - i0);
  for (int i = threadIdx.x >> 5; i < rows; i += 8) {
    const int r = s_row[i];
#pragma unroll 4
    for (int c = threadIdx.x & 31; c < n; c += 32) {
      const float2 v = W[elem(n, r, s_pos[c])];
      X[(size_t)(i0 + i) * n + c] = zmake((double)v.x, (double)v.y);
    }
  }
}

template <int NT>
cudaError_t launch_tiles(const TileInv& g, int tiles, cudaStream_t s) {
  for (int panel = -1; panel < tiles; ++panel) {
    if (panel == 0 && tiles == 1) break;   // no other tile to update
    inv_tile_kernel<NT><<<dim3(tiles, g.units), NT, 0, s>>>(g, panel);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

size_t zinv_tiles_bytes(int n, int units) {
  return (tile_stride(n) * sizeof(float2) + 2 * (size_t)n * sizeof(uint16_t)) * units;
}

cudaError_t zinv_tiles(BMat X, BMat M, int n, int units, const int* active, void* scratch, int32_t* status,
                       cudaStream_t s) {
  if (units <= 0 || n <= 0) return cudaSuccess;
  if (!scratch || n > kMaxN) return cudaErrorInvalidValue;
  TileInv g;
  g.M = M; g.X = X; g.n = n; g.units = units; g.active = active;
  g.W = (float2*)scratch;
  g.pos = (uint16_t*)(g.W + tile_stride(n) * units);
  g.status = status;
  const int tiles = (n + kTW - 1) / kTW;
  cudaError_t e = n <= 128 ? launch_tiles<128>(g, tiles, s)
                : n <= 256 ? launch_tiles<256>(g, tiles, s) : launch_tiles<512>(g, tiles, s);
  if (e != cudaSuccess) return e;
  inv_gather_kernel<<<dim3((n + kOutRows - 1) / kOutRows, units), 256, 0, s>>>(g, tiles - 1);
  return cudaGetLastError();
}

}  // namespace negf
