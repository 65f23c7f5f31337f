// The open boundary (Sec. II "LSE+OBC") of small blocks (b <= 16) as ONE launch: one CTA per
// lead unit (side, energy) runs the Lopez Sancho-Rubio decimation to its own convergence,
// the surface function and its residual, up to three Newton steps on the surface
// fixed-point equation (Smith doubling of the Stein equation) and Sigma, in shared memory
// and FP64.  The steps, their order and the stop rules are those of the batched path
// (negf_obc); a unit stops when it has converged instead of when the batch is polled.  (A second
// launch holds the rare units that start again.)
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

// AGAIN: the restarts (restart_widen) of the units that the launch before left open, in a launch of
// its own, which costs the others 1 us (as a loop around the one pass it cost 5 to 17)
template <bool AGAIN>
__global__ void __launch_bounds__(small_threads(kObcSmallB)) obc_small_kernel(ObcSmall a) {
  pdl_begin();
  const int u = blockIdx.x, b = a.b;
  int passes = 1;
  if (AGAIN) {
    if (!a.open[u]) return;
    int open = 0;
    for (int i = 0; i < 2 * a.U; i += blockDim.x) open += __syncthreads_count(i + threadIdx.x < 2 * a.U && a.open[i + threadIdx.x]);
    passes = open <= restart_many(2 * a.U) ? kRestarts : 1;
  }
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
  const int cd = left ? 0 : a.dv.nb - 1, cu = left ? 0 : a.dv.nb - 2;
  const long long idx = (long long)t.r * b + t.c, cr = (long long)t.c * b + t.r;
  zc *al = buf(0), *be = buf(1), *g = buf(2), *V = buf(3), *T0 = buf(4), *T1 = buf(5);
  zc *S = buf(6), *F = buf(7), *X = buf(8), *Y = buf(9);

  // this thread's component of the lead's A blocks at broadening eta: the onsite block, the
  // coupling alpha away from the surface and beta back (right lead: a01, a10; left lead: swapped)
  auto onsite = [&](double eta) {
    const zc s = a.dv.Sd ? a.dv.Sd[cd * bb + idx] : zmake(t.r == t.c ? 1.0 : 0.0, 0.0);
    return t.of(zsub(zmul(zmake(a.dv.E[e], eta), s), a.dv.Hd[cd * bb + idx]));
  };
  auto load_hops = [&](double eta) {
    const zc z = zmake(a.dv.E[e], eta);
    const zc s01 = a.dv.Su ? a.dv.Su[cu * bb + idx] : zmake(0.0, 0.0);
    const zc s10 = a.dv.Su ? zconj(a.dv.Su[cu * bb + cr]) : zmake(0.0, 0.0);
    const double a01 = t.of(zsub(zmul(z, s01), a.dv.Hu[cu * bb + idx]));
    const double a10 = t.of(zsub(zmul(z, s10), zconj(a.dv.Hu[cu * bb + cr])));
    t.put(al, left ? a10 : a01);
    t.put(be, left ? a01 : a10);
  };
  const double a00 = onsite(a.dv.eta);
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

  // the retarded root: every LDL^H pivot of i (g - g^H) is above -1e-12 times its largest
  // diagonal entry (a pivot within that of zero is skipped), as retarded_check_kernel has it
  auto retarded = [&]() {
    const zc x = g[t.r * t.ld + t.c], y = g[t.c * t.ld + t.r];
    double v = t.comp ? x.x - y.x : -(x.y + y.y);
    const double top = cta_reduce<true>(t.on && t.r == t.c && t.comp == 0 ? fmax(v, 0.0) : 0.0, red[turn ^= 1]);
    const double lim = 1e-12 * fmax(top, 1e-300);
    t.put(V, v);
    for (int p = 0; p < b; ++p) {
      __syncthreads();
      const double d = V[p * t.ld + p].x;
      if (d < -lim || !isfinite(d)) return false;   // (the same in every thread)
      if (d > lim && t.r > p && t.c > p) {          // rows and columns up to p are read only
        const zc l = V[t.r * t.ld + p], q = V[p * t.ld + t.c];
        v -= (t.comp ? l.x * q.y + l.y * q.x : l.x * q.x - l.y * q.y) / d;
        t.put(V, v);
      }
    }
    return true;
  };

  int done = 0, iters = 0, steps = 0;
  double res = 0.0;
#pragma unroll 1
  for (int again = 0; again < passes; ++again) {
    const double eta = AGAIN ? restart_widen(again) * a.dv.eta : a.dv.eta;
    done = 0;
    // ---------------- decimation
    __syncthreads();
    load_hops(eta);
    double eps = AGAIN ? onsite(eta) : a00, epss = eps;
    __syncthreads();
    const double ref = fmax(sqrt(hop_norm2()), 1e-300);
    const double lim = a.tol * ref, lim2 = lim * lim;
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
    load_hops(a.dv.eta);
    t.put(g, epss);
    __syncthreads();
    small_inverse(g, V, t, piv);
    res = residual(g);
    // ---------------- Newton polishing: D = -K^{-1} F + (K^{-1} al) D (be g)
    bool need = res > a.target;
    bool diverged = isnan(res);
    for (int step = 0; need && step < (AGAIN ? kRestartSteps : 3); ++step) {
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
      diverged = !(resn <= kDiverged * res);
      need = take && res > a.target;
      __syncthreads();
    }
    if (!AGAIN) {
      if (threadIdx.x == 0) a.open[u] = done == 2 || (done == 1 && !(res <= a.accept) && diverged);
    } else {
      if (done == 1 && res <= a.accept && retarded()) break;
      if (again + 1 == passes) return;   // the first result stands
    }
  }
  __syncthreads();
  // ---------------- outputs: g, Sigma = al g be
  const BMat& gs = left ? a.gs_L : a.gs_R;
  const BMat& sg = left ? a.sigma_L : a.sigma_R;
  if (gs.p) t.put_g(gs.at(k), t.get(g));
  t.put(T0, t.mul(al, g));
  __syncthreads();
  t.put_g(sg.at(k), t.mul(T0, be));
  if (threadIdx.x == 0) {
    a.done[u] = done;
    if (!AGAIN) a.iters[u] = iters;
    a.nsteps[u] = steps + (AGAIN ? a.nsteps[u] : 0);
    a.res[u] = res;
  }
}

size_t obc_small_smem(int b) { return sizeof(zc) * (size_t)kObcBufs * small_block_elems(b); }

}  // namespace

cudaError_t obc_small(const ObcSmall& a, cudaStream_t s) {
  if (a.U <= 0) return cudaSuccess;
  if (a.b < 1 || a.b > kObcSmallB) return cudaErrorInvalidValue;
  cudaError_t e = once_per_device(INIT_OBC_SMALL, [](int) {
    const cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
    const cudaError_t r = cudaFuncSetAttribute(obc_small_kernel<false>, smem, (int)obc_small_smem(kObcSmallB));
    return r != cudaSuccess ? r : cudaFuncSetAttribute(obc_small_kernel<true>, smem, (int)obc_small_smem(kObcSmallB));
  });
  if (e != cudaSuccess) return e;
  e = launch_pdl(obc_small_kernel<false>, 2 * a.U, small_threads(a.b), obc_small_smem(a.b), s, a);
  if (e != cudaSuccess) return e;
  return launch_pdl(obc_small_kernel<true>, 2 * a.U, small_threads(a.b), obc_small_smem(a.b), s, a);
}

}  // namespace negf
