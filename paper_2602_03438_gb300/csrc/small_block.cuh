// Products and inverses of b x b complex128 blocks (b <= 16) in the shared memory of one
// CTA, for the kernels that run a whole recursion of small blocks in one launch.
//
// GB300's FP64 pipe is narrow: half a lane per clock in each of an SM's four partitions,
// so one FP64 instruction of a warp holds its partition's pipe for 64 clocks and a b x b
// product is bound by 4 b^3 / 2 clocks per SM (1024 at b = 8).  Two threads share an
// element, one per component, so that b = 8 already gives each partition a warp, and
// everything but the arithmetic itself (maxima, pivots, interchanges) stays in integers.
#pragma once

#include "negf_internal.cuh"

namespace negf {

constexpr int kSmallB = 16;

// threads of a CTA for b x b blocks: a component of an element each
__host__ __device__ constexpr int small_threads(int b) { return (2 * b * b + 31) / 32 * 32; }
__host__ __device__ constexpr size_t small_block_elems(int b) { return (size_t)b * (b + 1); }

struct SmallElem {
  int b, ld, r, c, comp;   // element (r, c); comp 0: real part, 1: imaginary part
  bool on;                 // this thread has an element
  __device__ explicit SmallElem(int b_) : b(b_), ld(b_ + 1) {
    const int e = threadIdx.x >> 1;
    comp = threadIdx.x & 1;
    on = e < b * b;
    r = on ? e / b : 0;
    c = on ? e - r * b : 0;
  }
  __device__ double of(zc v) const { return comp ? v.y : v.x; }
  __device__ double get(const zc* A) const { return reinterpret_cast<const double*>(A + r * ld + c)[comp]; }
  __device__ void put(zc* D, double v) const {
    if (on) reinterpret_cast<double*>(D + r * ld + c)[comp] = v;
  }
  __device__ double get_g(const zc* A) const { return reinterpret_cast<const double*>(A + r * b + c)[comp]; }
  __device__ void put_g(zc* D, double v) const {
    if (on) reinterpret_cast<double*>(D + r * b + c)[comp] = v;
  }
  // this thread's component of element (r, c) of op(A) op(B), in the order of zfma over k
  template <bool HA = false, bool HB = false>
  __device__ double mul(const zc* A, const zc* B) const {
    double acc = 0.0;
    const zc* pa = HA ? A + r : A + r * ld;
    const zc* pb = HB ? B + c * ld : B + c;
    const int sa = HA ? ld : 1, sb = HB ? 1 : ld;
    // re: a.x b.x - a.y b.y, im: a.x b.y + a.y b.x, the conjugates flipping the y's: sign
    // flips of a.y and of a.x's factor, by integer XOR (a negation that the compiler cannot
    // fold into an operand is an FP64 instruction)
    const int ma = (comp == 0) != (HA != (HB && comp == 0)) ? (int)0x80000000 : 0;
    const int mb = (HB && comp) ? (int)0x80000000 : 0;
#pragma unroll 4
    for (int k = 0; k < b; ++k) {
      const zc a = pa[k * sa], v = pb[k * sb];
      const double ay = __hiloint2double(__double2hiint(a.y) ^ ma, __double2loint(a.y));
      double w = comp ? v.y : v.x;
      if (HB) w = __hiloint2double(__double2hiint(w) ^ mb, __double2loint(w));
      acc = fma(a.x, w, fma(ay, comp ? v.x : v.y, acc));
    }
    return acc;
  }
};

// The pivot of column k (the first row >= k of largest |.|^2) by one warp, lane = row, n <= 16:
// returns its row and 1 / pivot (~k and 0 when the column is zero) to every lane.  The largest
// comes from integer maxima of the two halves (non-negative doubles order like their bits),
// and every lane starts its own division before it is known who wins.
__device__ __forceinline__ int small_pivot(const zc* W, int ld, int n, int k, zc& dinv) {
  const int lane = threadIdx.x & 31;
  const bool cand = lane >= k && lane < n;
  const zc x = cand ? W[lane * ld + k] : zmake(0.0, 0.0);
  const double v = zabs2(x);
  const double rv = 1.0 / v;
  const bool nan = __double_as_longlong(v) > 0x7FF0000000000000ll;   // never the largest
  const unsigned int hi = (cand && !nan) ? (unsigned int)__double2hiint(v) : 0u;
  const unsigned int mh = __reduce_max_sync(0xffffffffu, hi);
  const bool c2 = cand && !nan && hi == mh;
  const unsigned int lo = c2 ? (unsigned int)__double2loint(v) : 0u;
  const unsigned int ml = __reduce_max_sync(0xffffffffu, lo);
  const unsigned int win = __ballot_sync(0xffffffffu, c2 && lo == ml);
  if (win == 0u || (mh | ml) == 0u) {
    dinv = zmake(0.0, 0.0);
    return ~k;
  }
  const int p = __ffs(win) - 1;
  zc q = zmake(x.x * rv, -x.y * rv);
  if (mh < 0x03000000u) q = zmake(x.x / v, -x.y / v);   // |pivot|^2 below ~1e-290: 1 / v may overflow
  dinv = zmake(__shfl_sync(0xffffffffu, q.x, p), __shfl_sync(0xffffffffu, q.y, p));
  return p;
}

// W <- W^{-1} (Gauss-Jordan, partial pivoting: the first row of largest |.|^2), the
// interchanges undone as column interchanges; V: a second block.  The caller synchronises
// before the call; the result is in W, synchronised.  Returns false to every thread when a
// pivot column is zero.  The steps alternate between the two blocks: one barrier per step.
// With a warp per partition (b <= 8) every warp finds the pivot itself; with more, one warp
// does and publishes it, since the others' divisions would hold the FP64 pipe.
__device__ __forceinline__ bool small_inverse(zc*& W, zc*& V, const SmallElem& t, int* piv) {
  __shared__ zc s_dinv;
  __shared__ int s_p;
  const int n = t.b, ld = t.ld;
  const bool each = blockDim.x <= 128;
  bool ok = true;
  for (int k = 0; k < n; ++k) {
    zc dinv = zmake(0.0, 0.0);
    int p = k;
    if (each || threadIdx.x < 32) p = small_pivot(W, ld, n, k, dinv);
    if (!each) {
      if (threadIdx.x == 0) {
        s_dinv = dinv;
        s_p = p;
      }
      __syncthreads();
      p = s_p;
      dinv = s_dinv;
    }
    if (p < 0) {   // a zero column: the row at position k stays
      ok = false;
      p = k;
    }
    if (threadIdx.x == 0) piv[k] = p;
    // this component of the scaled pivot row at column c, and the other one from the pair
    const zc w = W[p * ld + t.c];
    const double mine = t.comp ? fma(w.x, dinv.y, w.y * dinv.x) : fma(w.x, dinv.x, -w.y * dinv.y);
    const double other = __shfl_xor_sync(0xffffffffu, mine, 1);
    const zc prc = (t.c == k) ? dinv : (t.comp ? zmake(other, mine) : zmake(mine, other));
    double nv = t.of(prc);
    if (t.r != k) {
      const int src = (t.r == p) ? k : t.r;   // row r of the interchanged matrix
      const zc f = W[src * ld + k];
      const double w0 = (t.c == k) ? 0.0 : t.get(W + (src - t.r) * ld);
      nv = t.comp ? fma(-f.x, prc.y, fma(-f.y, prc.x, w0)) : fma(-f.x, prc.x, fma(f.y, prc.y, w0));
    }
    t.put(V, nv);
    __syncthreads();
    zc* s = W; W = V; V = s;
  }
  // column c of the inverse: follow the column interchanges (k = n-1 .. 0) back from c
  int pos = t.c;
  for (int k = 0; k < n; ++k) {
    const int p = piv[k];
    pos = (pos == k) ? p : (pos == p) ? k : pos;
  }
  const double res = reinterpret_cast<const double*>(W + t.r * ld + pos)[t.comp];
  t.put(V, res);
  __syncthreads();
  zc* s = W; W = V; V = s;
  return ok;
}

}  // namespace negf
