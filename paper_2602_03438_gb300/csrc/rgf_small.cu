// The RGF sweeps of devices with small blocks (b <= 16) as ONE persistent launch: one CTA
// per energy runs the whole forward and backward recursion of G^R and of the Keldysh
// functions G^< (and G^>) (Sec. II, Eqs. (1)-(2); the textbook block recursion), keeping
// the left-connected blocks and the running G blocks in shared memory, in FP64.
//
// At these sizes every block product is below the smallest tensor-core tile, and the
// batched per-step launches (about 16 launches per block index) are bound by launch and
// fill latency rather than by arithmetic: one CTA per energy with two threads per block
// element (one per component, small_block.cuh) does the same FP64 operations with no launch
// between them, bound by the FP64 pipe.  Measured (GB300): 64 energies of 16 blocks of 8,
// G^R and G^<, 0.59 -> 0.35 ms against one thread per element.
//
// Forward, i = 0 .. nb-1 (Y_{i-1} = A_{i,i-1} g_{i-1}):
//   g_i = (A_ii - Y_{i-1} A_{i-1,i})^{-1},
//   g^x_i = g_i (Sigma^x_ii + A_{i,i-1} g^x_{i-1} A_{i,i-1}^H) g_i^H          (x = <, >)
// Backward, i = nb-2 .. 0 (X = g_i A_{i,i+1}):
//   G_{i,i+1} = -X G_{i+1,i+1},  G_ii = g_i - G_{i,i+1} Y_i,  G_{i+1,i} = -G_{i+1,i+1} Y_i,
//   Z = A_{i+1,i} g^x_i,  P = G^x_{i+1,i+1} X^H,  W = G_{i,i+1} Z,
//   G^x_ii = g^x_i + X P - W + W^H,  G^x_{i+1,i} = -G_{i+1,i+1} Z - P.
// The block inverse is Gauss-Jordan with partial pivoting (first row of largest
// modulus), in place, its row interchanges undone as column interchanges.
#include "small_block.cuh"

namespace negf {

namespace {

constexpr int kBufs = 13;

__global__ void __launch_bounds__(small_threads(kSmallB)) rgf_small_kernel(SmallSweep a) {
  pdl_begin();
  const int u = blockIdx.x;
  const int b = a.b, nb = a.nb;
  const long long bb = (long long)b * b;
  const long long step = (long long)a.U * bb;   // stride of the assembled blocks' index
  extern __shared__ __align__(16) unsigned char smem_raw[];
  zc* buf[kBufs];
  for (int q = 0; q < kBufs; ++q) buf[q] = reinterpret_cast<zc*>(smem_raw) + (size_t)q * small_block_elems(b);
  __shared__ int piv[kSmallB];
  const SmallElem t(b);
  bool ok = true;

  // named roles; G, M and the inverse's second block V swap by pointer
  zc *Al = buf[0], *Au = buf[1], *Yb = buf[2], *T1 = buf[3], *T2 = buf[4], *S = buf[5];
  zc *X = buf[6], *Gu = buf[7], *P = buf[8], *G = buf[9], *M = buf[10];
  zc* K[2] = {buf[11], buf[12]};
  const zc* sigx[2] = {a.Sl, a.Sg};
  const SBlk outx[2] = {a.gL, a.gG};
  const SBlk lowx[2] = {a.Ll, a.Gl};
  // the adjacent lane's component of the transposed element, from shared memory
  auto herm = [&](const zc* A) {   // this component of A^H at (r, c)
    const double v = reinterpret_cast<const double*>(A + t.c * t.ld + t.r)[t.comp];
    return t.comp ? -v : v;
  };

  // ---------------- forward sweep
  for (int i = 0; i < nb; ++i) {
    double m = t.get_g(a.Ad + i * step + u * bb);
    if (i > 0) {
      t.put(Al, t.get_g(a.Al + (i - 1) * step + u * bb));
      t.put(Au, t.get_g(a.Au + (i - 1) * step + u * bb));
      __syncthreads();
      const double y = t.mul(Al, G);   // Y_{i-1} = A_{i,i-1} g_{i-1}
      t.put(Yb, y);
      t.put_g(a.Y.at(u, i - 1), y);
      __syncthreads();
      m -= t.mul(Yb, Au);
    }
    t.put(M, m);
    __syncthreads();
    ok = small_inverse(M, T2, t, piv) && ok;   // M <- g_i
    t.put_g(a.gR.at(u, i), t.get(M));
    for (int x = 0; x < a.nk; ++x) {
      double v = t.get_g(sigx[x] + i * step + u * bb);
      if (i > 0) {
        t.put(T1, t.mul(Al, K[x]));               // A_{i,i-1} g^x_{i-1}
        __syncthreads();
        v += t.mul<false, true>(T1, Al);
      }
      t.put(T2, v);
      __syncthreads();
      v = t.mul(M, T2);
      t.put(S, v);
      __syncthreads();
      v = t.mul<false, true>(S, M);               // g^x_i
      t.put(K[x], v);
      t.put_g(outx[x].at(u, i), v);
      __syncthreads();
    }
    zc* sw = G; G = M; M = sw;   // G <- g_i
  }
  // ---------------- backward sweep (G holds G_{i+1,i+1}, K[x] G^x_{i+1,i+1})
  for (int i = nb - 2; i >= 0; --i) {
    __syncthreads();
    t.put(Au, t.get_g(a.Au + i * step + u * bb));
    t.put(Al, t.get_g(a.Al + i * step + u * bb));
    t.put(M, t.get_g(a.gR.at(u, i)));    // g_i
    t.put(Yb, t.get_g(a.Y.at(u, i)));
    __syncthreads();
    t.put(X, t.mul(M, Au));              // X = g_i A_{i,i+1}
    __syncthreads();
    double v = -t.mul(X, G);             // G_{i,i+1} = -X G_{i+1,i+1}
    t.put(Gu, v);
    if (a.Ru.p) t.put_g(a.Ru.at(u, i), v);
    if (a.Rl.p) t.put_g(a.Rl.at(u, i), -t.mul(G, Yb));   // G_{i+1,i} = -G_{i+1,i+1} Y_i
    for (int x = 0; x < a.nk; ++x) {
      const double gx = t.get_g(outx[x].at(u, i));   // g^x_i
      t.put(T2, gx);
      __syncthreads();
      t.put(T1, t.mul(Al, T2));                 // Z = A_{i+1,i} g^x_i
      const double pv = t.mul<false, true>(K[x], X);   // P = G^x_{i+1,i+1} X^H
      t.put(P, pv);
      __syncthreads();
      if (lowx[x].p) t.put_g(lowx[x].at(u, i), -(t.mul(G, T1) + pv));   // G^x_{i+1,i} = -G_{i+1,i+1} Z - P
      const double w = t.mul(Gu, T1);           // W = G_{i,i+1} Z
      t.put(S, w);
      v = gx + t.mul(X, P);
      __syncthreads();
      v = (v - w) + herm(S);                    // G^x_ii = g^x_i + X P - W + W^H
      t.put(K[x], v);
      t.put_g(outx[x].at(u, i), v);
      __syncthreads();
    }
    if (a.nk == 0) __syncthreads();
    v = t.get(M) - t.mul(Gu, Yb);               // G_ii = g_i - G_{i,i+1} Y_i
    __syncthreads();
    t.put(M, v);
    t.put_g(a.gR.at(u, i), v);
    zc* sw = G; G = M; M = sw;   // G <- G_ii
  }
  if (threadIdx.x == 0 && !ok && a.status) a.status[u] = NEGF_ERR_SINGULAR;
}

}  // namespace

// b = 16 reaches the sliced product's smallest tile in NEGF_MIXED, but seven eighths of its
// 128 rows are padding there: a sweep of 256 energies, 8 blocks and both Keldysh kinds
// took 8.5 ms step by step and takes 2.0 ms in one launch
bool rgf_small_supported(int b, int mixed) { return b >= 1 && (b < 16 || (b == 16 && mixed != 2)); }

bool rgf_small_optional(int b, int mixed) { return b == 16 && mixed == 1; }

size_t rgf_small_smem(int b) { return sizeof(zc) * (size_t)kBufs * small_block_elems(b); }

cudaError_t rgf_small_sweep(const SmallSweep& a, cudaStream_t s) {
  if (a.U <= 0) return cudaSuccess;
  if (a.b < 1 || a.b > kSmallB || a.nk < 0 || a.nk > 2) return cudaErrorInvalidValue;
  const size_t smem = rgf_small_smem(a.b);
  cudaError_t e = once_per_device(INIT_SMALL, [](int) {
    return cudaFuncSetAttribute(rgf_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)rgf_small_smem(kSmallB));
  });
  if (e != cudaSuccess) return e;
  launch_pdl(rgf_small_kernel, a.U, small_threads(a.b), smem, s, a);
  return cudaGetLastError();
}

}  // namespace negf
