// The open boundary (Sec. II "LSE+OBC") of small blocks (b <= 16) as ONE launch: one CTA per
// lead unit (side, energy) runs the Lopez Sancho-Rubio decimation to its own convergence,
// the surface function and its residual, up to three Newton steps on the surface
// fixed-point equation (Smith doubling of the Stein equation) and Sigma, in shared memory
// and FP64.  The steps, their order and the stop rules are those of the batched path
// (negf_obc); a unit stops when it has converged instead of when the batch is polled.
//
// What bounds it: the FP64 pipe (small_block.cuh) along one unit's serial chain of six
// products and an inverse per decimation step and four products per Smith level.
// Measured (GB300, 64 energies of blocks of 8, both leads): 0.48 ms, against 7.06 ms for the
// batched path's 426 launches.  Beyond b = 16 (kObcSmallB) a product's 4 b^3 FP64 FMAs per
// SM pass what the batched path's launches cost.
#include "small_block.cuh"

namespace negf {

namespace {

constexpr int kObcBufs = 10;
constexpr int kMaxWarps = small_threads(kObcSmallB) / 32;

// the sum (MAX: largest) over the CTA of non-negative values, to every thread; red is
// alternated by the caller so that one barrier suffices
template <bool MAX>
__device__ __forceinline__ double cta_reduce(double v, double* red) {
  for (int off = 16; off > 0; off >>= 1) {
    const double o = __shfl_xor_sync(0xffffffffu, v, off);
    if (MAX) v = __double_as_longlong(o) > __double_as_longlong(v) ? o : v;   // order of non-negative doubles
    else v += o;
  }
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = red[0];
  for (int w = 1; w < (int)(blockDim.x >> 5); ++w) {
    const double o = red[w];
    if (MAX) v = __double_as_longlong(o) > __double_as_longlong(v) ? o : v;
    else v += o;
  }
  return v;
}

__global__ void __launch_bounds__(small_threads(kObcSmallB)) obc_small_kernel(ObcSmall a) {
  pdl_begin();
  const int u = blockIdx.x, b = a.b;
  const bool left = u < a.U;
  const int k = left ? u : u - a.U;   // the energy unit
  int e = a.e0 + k;
  if (a.udev) {
    a.dv = a.udev[a.unit_dev[k]].dv;
    e = a.unit_e[k];
  }
  const long long bb = (long long)b * b;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  auto buf = [&](int q) { return reinterpret_cast<zc*>(smem_raw) + (size_t)q * small_block_elems(b); };
  __shared__ double red[4][kMaxWarps];
  __shared__ int piv[kSmallB];
  const SmallElem t(b);
  const zc z = zmake(a.dv.E[e], a.dv.eta);
  const int cd = left ? 0 : a.dv.nb - 1, cu = left ? 0 : a.dv.nb - 2;
  const long long idx = (long long)t.r * b + t.c, cr = (long long)t.c * b + t.r;
  zc *al = buf(0), *be = buf(1), *g = buf(2), *V = buf(3), *T0 = buf(4), *T1 = buf(5);
  zc *S = buf(6), *F = buf(7), *X = buf(8), *Y = buf(9);

  // this thread's component of the lead's A blocks: the onsite block, the coupling alpha away
  // from the surface and beta back (right lead: a01, a10; left lead: swapped)
  auto a01 = [&]() {
    const zc s = a.dv.Su ? a.dv.Su[cu * bb + idx] : zmake(0.0, 0.0);
    return t.of(zsub(zmul(z, s), a.dv.Hu[cu * bb + idx]));
  };
  auto a10 = [&]() {
    const zc s = a.dv.Su ? zconj(a.dv.Su[cu * bb + cr]) : zmake(0.0, 0.0);
    return t.of(zsub(zmul(z, s), zconj(a.dv.Hu[cu * bb + cr])));
  };
  const zc s00 = a.dv.Sd ? a.dv.Sd[cd * bb + idx] : zmake(t.r == t.c ? 1.0 : 0.0, 0.0);
  const double a00 = t.of(zsub(zmul(z, s00), a.dv.Hd[cd * bb + idx]));
  auto load_hops = [&]() {
    t.put(al, left ? a10() : a01());
    t.put(be, left ? a01() : a10());
  };
  // the largest |entry| of the two hops
  int turn = 0;
  auto abs2 = [&](double v) {   // |element|^2 from the two components of the thread pair
    const double o = __shfl_xor_sync(0xffffffffu, v, 1);
    return t.on ? (t.comp ? fma(o, o, v * v) : fma(v, v, o * o)) : 0.0;
  };
  auto or_zero = [](double v) { return __double_as_longlong(v) > 0x7FF0000000000000ll ? 0.0 : v; };   // fmax passes NaN by
  // largest squared moduli (the square roots would cost about as much as a product)
  auto largest = [&](double v) { return cta_reduce<true>(or_zero(abs2(v)), red[turn ^= 1]); };
  auto hop_norm2 = [&]() {
    const double x = or_zero(abs2(t.get(al))), y = or_zero(abs2(t.get(be)));
    return cta_reduce<true>(__double_as_longlong(x) > __double_as_longlong(y) ? x : y, red[turn ^= 1]);
  };
  // K = a00 - al X be (kept in T1), F = K X - I; returns ||F||_F / sqrt(b).  al, be: the
  // lead's own hops; needs X synchronised
  auto residual = [&](const zc* Xm) {
    t.put(T0, t.mul(al, Xm));
    __syncthreads();
    t.put(T1, a00 - t.mul(T0, be));
    __syncthreads();
    double f = t.mul(T1, Xm);
    if (t.r == t.c && t.comp == 0) f -= 1.0;
    t.put(F, f);
    const double sum = cta_reduce<false>(abs2(f) * 0.5, red[2]);   // both threads of a pair hold |f|^2
    return sqrt(sum / b);
  };

  // ---------------- decimation
  load_hops();
  double eps = a00, epss = a00;
  __syncthreads();
  const double ref = fmax(sqrt(hop_norm2()), 1e-300);
  const double lim = a.tol * ref, lim2 = lim * lim;
  int done = 0, iters = 0;
  for (int it = 0; it <= a.max_iter; ++it) {
    const double m2 = hop_norm2();
    const bool fin = isfinite(m2);
    if (!fin || (lim2 > 1e-280 ? m2 < lim2 : sqrt(m2) < lim)) {
      done = fin ? 1 : 2;
      iters = it;
      break;
    }
    if (it == a.max_iter) break;
    t.put(g, eps);
    __syncthreads();
    small_inverse(g, V, t, piv);
    t.put(T0, t.mul(al, g));          // al g
    t.put(T1, t.mul(be, g));          // be g
    __syncthreads();
    const double agb = t.mul(T0, be), bga = t.mul(T1, al);
    const double na = -t.mul(T0, al), nb = -t.mul(T1, be);
    epss -= agb;
    eps = (eps - agb) - bga;
    __syncthreads();
    t.put(al, na);
    t.put(be, nb);
    __syncthreads();
  }
  // ---------------- surface function and its residual
  __syncthreads();
  load_hops();
  t.put(g, epss);
  __syncthreads();
  small_inverse(g, V, t, piv);
  double res = residual(g);
  // ---------------- Newton polishing: D = -K^{-1} F + (K^{-1} al) D (be g)
  int steps = 0;
  bool need = res > a.target;
  while (need && steps < 3) {
    __syncthreads();
    t.put(X, t.get(T1));
    __syncthreads();
    small_inverse(X, V, t, piv);                          // K^{-1}
    const double p0 = t.mul(X, al), q0 = t.mul(be, g), s0 = -t.mul(X, F);
    __syncthreads();
    zc *Pm = X, *Qm = Y;
    t.put(Pm, p0);
    t.put(Qm, q0);
    t.put(S, s0);
    double sv = s0;
    __syncthreads();
    for (int j = 0; j < 96; ++j) {
      t.put(T0, t.mul(Pm, S));                            // P S
      const double pp = t.mul(Pm, Pm), qq = t.mul(Qm, Qm);   // P^2, Q^2 (of a level that may be the last)
      __syncthreads();
      const double inc = t.mul(T0, Qm);                   // P S Q
      sv += inc;
      const double mi = largest(inc), ms = largest(sv);
      if (mi <= 1e-30 * ms || !isfinite(ms)) break;   // |increment| <= 1e-15 |S|
      // balance P^2 against Q^2 by the power of two nearest to the square root of the ratio
      // of their largest entries (from the exponent fields of the squared moduli)
      const int ep = (int)(__double_as_longlong(largest(pp)) >> 52), eq = (int)(__double_as_longlong(largest(qq)) >> 52);
      const int sh = (ep > 0 && eq > 0 && ep < 2047 && eq < 2047) ? (eq - ep) / 4 : 0;
      const double sc = __longlong_as_double((long long)(1023 + sh) << 52);
      const double si = __longlong_as_double((long long)(1023 - sh) << 52);
      t.put(S, sv);
      t.put(Pm, pp * sc);
      t.put(Qm, qq * si);
      __syncthreads();
    }
    const double gv = t.get(g), gn = gv + sv;
    t.put(V, gn);
    __syncthreads();
    const double resn = residual(V);
    ++steps;
    const bool take = resn < res;
    if (take) {
      res = resn;
      t.put(g, gn);
    }
    need = take && res > a.target;
    __syncthreads();
  }
  // ---------------- outputs: g, Sigma = al g be
  const BMat& gs = left ? a.gs_L : a.gs_R;
  const BMat& sg = left ? a.sigma_L : a.sigma_R;
  if (gs.p) t.put_g(gs.at(k), t.get(g));
  t.put(T0, t.mul(al, g));
  __syncthreads();
  t.put_g(sg.at(k), t.mul(T0, be));
  if (threadIdx.x == 0) {
    a.done[u] = done;
    a.iters[u] = iters;
    a.nsteps[u] = steps;
    a.res[u] = res;
  }
}

size_t obc_small_smem(int b) { return sizeof(zc) * (size_t)kObcBufs * small_block_elems(b); }

}  // namespace

cudaError_t obc_small(const ObcSmall& a, cudaStream_t s) {
  if (a.U <= 0) return cudaSuccess;
  if (a.b < 1 || a.b > kObcSmallB) return cudaErrorInvalidValue;
  cudaError_t e = once_per_device(INIT_OBC_SMALL, [](int) {
    return cudaFuncSetAttribute(obc_small_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)obc_small_smem(kObcSmallB));
  });
  if (e != cudaSuccess) return e;
  launch_pdl(obc_small_kernel, 2 * a.U, small_threads(a.b), obc_small_smem(a.b), s, a);
  return cudaGetLastError();
}

}  // namespace negf
