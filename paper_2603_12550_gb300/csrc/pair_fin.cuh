#pragma once
// pair_fin.cuh -- the O(N) epilogues of the pair passes: the partial sums of a
// particle added in a fixed order (FP64), then densities and energies, or
// gradients, velocities, time-step updates and the implicit minimiser's
// direction.  Included by pair_impl.cuh.
//
// One thread per (particle, component) and share of the partial sums: PB
// particles x D x SPL threads per CTA, the particle the fast index, so
// partials (component planes) and the shared arrays are read by consecutive
// lanes.  The FP64 pipe of GB300 is narrow and its latency long: one thread
// per particle, looping over components with the space dimension known only
// at run time, took 29.7 us at N = 1000, D = 9 and 38.7 us at N = 65536.  The
// partials are therefore (sum, compensation) pairs of FP32, added as such
// (two-sum, about 48 bits) and not as FP64 numbers: at N = 65536 the
// symmetric gradient pass leaves 40 per component, and their FP64 sum alone
// took 107 us.

namespace vds_pair {

// Entries of the Rouse matrix's inverse: min(j,k)(nb+1-max(j,k))/(nb+1), 1-based.
template <int NB>
__device__ __forceinline__ double rouse_Ainv(int j, int k) {
  const int lo = (j < k ? j : k) + 1, hi = (j > k ? j : k) + 1;
  return (double)(lo * (NB + 1 - hi)) * (1.0 / (double)(NB + 1));
}

// Particles per CTA and threads per (particle, component).
template <int D>
struct FinCfg {
  static constexpr int PB = 32;
  static constexpr int SPL = D == 2 ? 8 : D <= 4 ? 4 : D <= 9 ? 2 : 1;
  static constexpr int NT = PB * D * SPL;
};

// A sum of partials carried as s + c.
struct Sum2 {
  float s = 0.f, c = 0.f;
  __device__ __forceinline__ void add(float2 v) {  // v.x + v.y
    const float t = s + v.x, b = t - s;
    c += ((s - (t - b)) + (v.x - b)) + v.y;
    s = t;
  }
  __device__ __forceinline__ double value() const { return (double)s + (double)c; }
};

// Deterministic grid reduction of K values per thread: warp, CTA, then the
// last CTA to arrive (ticket) sums the CTAs' partials in a fixed order.  Only
// the first NA threads of a CTA have values, and only warps that hold some
// take part: FP64 sums of 32 warps of zeros took 4 us of a pass at N = 512.
// Returns true in the thread that holds the final value.
template <int K, int NT, int NA>
__device__ __forceinline__ bool grid_reduce(const double (&v)[K], const bool (&is_max)[K], double *red,
                                            unsigned *ticket, double (&out)[K]) {
  constexpr int NW = NT / 32;
  __shared__ double sh[NW][K];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  auto cta = [&](double (&x)[K], int nw) {  // of the first nw warps; result in thread 0
    if (w < nw)
#pragma unroll
      for (int k = 0; k < K; ++k) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
          const double y = __shfl_xor_sync(0xffffffffu, x[k], o);
          x[k] = is_max[k] ? fmax(x[k], y) : x[k] + y;
        }
        if (lane == 0) sh[w][k] = x[k];
      }
    __syncthreads();
    if (threadIdx.x == 0)
#pragma unroll
      for (int k = 0; k < K; ++k) {
        double s = sh[0][k];
        for (int q = 1; q < nw; ++q) s = is_max[k] ? fmax(s, sh[q][k]) : s + sh[q][k];
        x[k] = s;
      }
  };
  double x[K];
#pragma unroll
  for (int k = 0; k < K; ++k) x[k] = v[k];
  cta(x, (NA + 31) / 32);
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < K; ++k) red[(size_t)blockIdx.x * K + k] = x[k];
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
#pragma unroll
  for (int k = 0; k < K; ++k) x[k] = 0.0;  // the maxima are of absolute values
  for (unsigned b = threadIdx.x; b < gridDim.x; b += NT)
#pragma unroll
    for (int k = 0; k < K; ++k) {
      const double y = __ldcg(red + (size_t)b * K + k);
      x[k] = is_max[k] ? fmax(x[k], y) : x[k] + y;
    }
  const int nw = (int)((gridDim.x + 31u) / 32u);
  cta(x, nw < NW ? nw : NW);
  if (threadIdx.x != 0) return false;
#pragma unroll
  for (int k = 0; k < K; ++k) out[k] = x[k];
  *ticket = 0u;
  return true;
}

// Where a pair pass left the partial sums of its particles.
struct PartSrc {
  Sched sc;
  const float2 *i;  // [tile][segment][component][TI], (sum, rest)
  const float2 *j;  // symmetric passes: [tile][component][columns after it]
};

// Partial sum number x (0 <= x < part_count) of component a (of ACC) of particle p.
__device__ __forceinline__ int part_count(const PartSrc &s, int p, int &nseg) {
  const int t = p / s.sc.TI;
  nseg = sched_first_cta(sched_start(t + 1, s.sc) - 1, s.sc) - sched_first_cta(sched_start(t, s.sc), s.sc) + 1;
  return nseg + (s.sc.cpt ? t : 0);
}
template <int ACC>
__device__ __forceinline__ float2 part_get(const PartSrc &s, int p, int a, int x, int nseg) {
  const int t = p / s.sc.TI;
  if (x < nseg) return s.i[(((size_t)t * s.sc.maxseg + x) * ACC + a) * s.sc.TI + (p - t * s.sc.TI)];
  const int r = x - nseg;  // the sums that tile r formed for the particles after it
  return s.j[(size_t)sched_jrow(r, s.sc) * ACC + (size_t)a * sched_jcols(r, s.sc) + (p - (r + 1) * s.sc.TI)];
}

// ------------------------------------------------------------ epilogue maths
// Called by all threads of a CTA of NT >= PB x D; thread p + PB a is component
// a of the CTA's particle p, the threads from PB x D on have none.

template <int D, int PB>
struct FinShared {
  double y[D][PB];  // the point the sums were taken at
  double g[D][PB];
  double d[D][PB];  // displacements
  float o[PB * D];  // rows to be written, particle major
};

// Spring energy and force factor of the bond at y[0..S): grad Psi_k = f q_k.
template <int S>
__device__ __forceinline__ bool bond_eval(const KParams &kp, int k, double n2, double &psi, double &f) {
  if (kp.spring == 0) {
    psi = 0.5 * kp.H[k] * n2;
    f = kp.H[k];
    return true;
  }
  const double x = 1.0 - n2 / kp.b;
  if (!(x > 0.0)) {
    psi = 0.0;
    f = 0.0;
    return false;
  }
  psi = -0.5 * kp.H[k] * kp.b * log(x);
  f = kp.H[k] / x;
  return true;
}

// Arguments of the epilogues that both the finish kernels and the small-cloud
// passes take.
struct FinArgs {
  float *rec;           // records: w is written here (density), or the next step's (explicit)
  float *out;           // rho (density, may be NULL) or the gradient pass's output
  const float *ybase, *ydelta, *qa, *qb;
  float *q_io;
  int want_energy;
  double *red;
  unsigned *ticket;
  double *scal;
  int *err;
  ImpArgs imp;  // imp.st NULL: not a minimiser's pass
};

// The displacements of a pass (a copy of the arguments with the minimiser's in
// their place would put them all in local memory).
struct FinPtrs {
  const float *ydelta, *qa;
};
// Whether the pass is due (a minimiser's may not be), and its displacements.
__device__ __forceinline__ bool imp_take(const FinArgs &A, bool grad, FinPtrs &P) {
  P.ydelta = A.ydelta;
  P.qa = A.qa;
  const ImpState *s = A.imp.st;
  if (!s) return true;
  if (!imp_due(s, grad)) return false;
  P.ydelta = (s->cur != 0) == grad ? A.imp.d[1] : A.imp.d[0];
  if (!grad) P.qa = P.ydelta;
  return true;
}

// The minimiser's next state after the trial's objective J.  One thread, after
// every CTA has raised its flags.
__device__ __forceinline__ void imp_after_trial(ImpState *s, double J, int *err) {
  const int e = *(volatile int *)err;
  const bool start = s->phase == IMP_READY || s->start;
  if (s->phase == IMP_READY) {
    s->it = 0;
    s->cold = s->step == 0;
  }
  if (e != 0 && e != VDS_EDOMAIN) {
    s->phase = IMP_STOP;
    return;
  }
  if (start) {
    if (e == VDS_EDOMAIN) {
      if (s->cold) {
        s->phase = IMP_STOP;  // q* itself is outside
        return;
      }
      *err = 0;
      s->cold = 1;  // the previous correction leads outside: start from q*
      s->start = 1;
      s->alpha = 0.0;
      s->phase = IMP_TRIAL;
      return;
    }
    s->start = 0;
  } else if (e == VDS_EDOMAIN || !(J <= s->J - 1e-4 * s->alpha * s->dec + s->jfloor * (1.0 + fabs(s->J)))) {
    *err = 0;
    s->alpha *= 0.5;
    if (++s->ls > 30) {
      s->status = VDS_ENOCONV;
      s->phase = IMP_STOP;
    }
    return;
  }
  s->J = J;
  s->cur = 1 - s->cur;
  if (s->it >= s->max_iter) {
    s->status = VDS_ENOCONV;
    s->fin_dir = 0;
    s->phase = IMP_FINAL;
  } else {
    s->phase = IMP_GRAD;
  }
}

// ... after a direction: decrease dec, largest entries of the direction and of y.
__device__ __forceinline__ void imp_after_grad(ImpState *s, double dec, double dmax, double ymax, int *err) {
  if (*(volatile int *)err != 0) {
    s->phase = IMP_STOP;
    return;
  }
  ++s->it;
  s->dec = dec;
  if (dmax <= s->tol * (1.0 + ymax)) {
    s->fin_dir = 1;
    s->phase = IMP_FINAL;
  } else {
    s->alpha = 1.0;
    s->ls = 0;
    s->phase = IMP_TRIAL;
  }
}

// y of every particle of the CTA into sh.y (FP32 sum of base and delta), and
// qa - qb (or ydelta) into sh.d where asked; ends with a barrier.
template <int D, int PB>
__device__ __forceinline__ void fin_load(const FinArgs &A, const FinPtrs &P, int base, int N, bool want_d, bool d_is_delta,
                                         FinShared<D, PB> &sh) {
  const int n = min(PB, N - base) * D;
  const int e = threadIdx.x;
  if (e < n) {
    const size_t x = (size_t)base * D + e;
    float v = A.ybase[x];
    if (P.ydelta) v = v + P.ydelta[x];
    sh.y[e % D][e / D] = (double)v;
    if (want_d)
      sh.d[e % D][e / D] = d_is_delta ? (double)P.ydelta[x] : (double)P.qa[x] - (A.qb ? (double)A.qb[x] : 0.0);
  }
  __syncthreads();
}

// Density: rho of the particle in every one of its threads.
template <int D, int S, int PB, int NT>
__device__ __forceinline__ void fin_density(const KParams &kp, const FinArgs &A, const FinPtrs &P, int base, double rho,
                                            FinShared<D, PB> &sh) {
  constexpr int DP = Rec<D>::DP, NB = D / S;
  const int p = threadIdx.x % PB, a = threadIdx.x / PB, i = base + p;
  const bool on = i < kp.N && a < D;
  if (on && a == 0) {
    if (!(rho >= 0.5 && rho <= 1e300)) vds_flag(A.err, VDS_ENAN);
    A.rec[(size_t)i * DP + D] = (float)(1.0 / rho);
    if (A.out) A.out[i] = (float)rho;
  }
  if (!A.want_energy) return;
  fin_load<D, PB>(A, P, base, kp.N, P.qa != nullptr, false, sh);
  double e = 0.0;
  if (on) {
    const int k = a / S, al = a - k * S;
    if (al == 0) {
      double n2 = 0.0, psi, f;
#pragma unroll
      for (int b = 0; b < S; ++b) n2 += sh.y[k * S + b][p] * sh.y[k * S + b][p];
      if (!bond_eval<S>(kp, k, n2, psi, f)) vds_flag(A.err, VDS_EDOMAIN);
      e += psi;
    }
    if (a == 0) e += kp.kBT * (log(rho) + kp.lnorm);
    if (P.qa) {
      double m = 0.0;
#pragma unroll
      for (int kb = 0; kb < NB; ++kb) m += rouse_Ainv<NB>(k, kb) * sh.d[kb * S + al][p];
      e += 0.5 * kp.zeta_dt * sh.d[a][p] * m;
    }
  }
  double v[1] = {e}, out[1];
  const bool mx[1] = {false};
  if (grid_reduce<1, NT, PB * D>(v, mx, A.red, A.ticket, out)) {
    const double E = out[0] / (double)kp.N;
    A.scal[SC_E] = E;
    if (!(fabs(E) <= 1e300)) vds_flag(A.err, VDS_ENAN);
    if (A.imp.st) imp_after_trial(A.imp.st, E, A.err);
  }
}

// Gradient: u_sum is sum_J u dqhat of (particle p, component a).
template <int D, int S, int MODE, int PB, int NT>
__device__ __forceinline__ void fin_grad(const KParams &kp, const FinArgs &A, const FinPtrs &P, int base, double u_sum,
                                         FinShared<D, PB> &sh) {
  constexpr int DP = Rec<D>::DP, NB = D / S;
  const int p = threadIdx.x % PB, a = threadIdx.x / PB, i = base + p;
  const bool on = i < kp.N && a < D;
  const int k = a / S, al = a - k * S;
  const bool want_d = MODE == GM_IMPLICIT_DIR || (MODE == GM_OUT && P.qa != nullptr);
  fin_load<D, PB>(A, P, base, kp.N, want_d, MODE == GM_IMPLICIT_DIR, sh);
  double g = 0.0;
  if (on) {
    double f = kp.H[k];
    if (kp.spring == 1) {
      double n2 = 0.0;
#pragma unroll
      for (int b = 0; b < S; ++b) n2 += sh.y[k * S + b][p] * sh.y[k * S + b][p];
      const double x = 1.0 - n2 / kp.b;
      if (x > 0.0) {
        f = f / x;
      } else {
        f = 0.0;
        vds_flag(A.err, VDS_EDOMAIN);
      }
    }
    g = kp.kBT * (-kp.sfac * u_sum) + f * sh.y[a][p];
    if (MODE == GM_OUT && want_d) {
      double m = 0.0;
#pragma unroll
      for (int kb = 0; kb < NB; ++kb) m += rouse_Ainv<NB>(k, kb) * sh.d[kb * S + al][p];
      g += kp.zeta_dt * m;
    }
  }
  float row = (float)g;  // what this thread contributes to its particle's row
  double dec = 0.0, dmax = 0.0, ymax = 0.0;
  if constexpr (MODE != GM_OUT) {
    if (a < D) sh.g[a][p] = g;
    __syncthreads();
    if (on) {
      // (A g)_k: 2 on the diagonal of the Rouse matrix, -1 beside it
      double m = 2.0 * g;
      if (k > 0) m -= sh.g[a - S][p];
      if (k + 1 < NB) m -= sh.g[a + S][p];
      if constexpr (MODE == GM_IMPLICIT_DIR) {
        double aid = 0.0;
#pragma unroll
        for (int kb = 0; kb < NB; ++kb) aid += rouse_Ainv<NB>(k, kb) * sh.d[kb * S + al][p];
        const double dr = sh.d[a][p] + kp.dt_zeta * m;
        const double G = kp.zeta_dt * aid + g;
        row = (float)dr;
        dec = G * dr;
        dmax = fabs((double)row);
        ymax = fabs(sh.y[a][p]);
      } else {
        double v = 0.0;
#pragma unroll
        for (int be = 0; be < S; ++be) v += kp.kappa[al * S + be] * sh.y[k * S + be][p];
        const double vel = v - m * kp.rzeta;
        row = MODE == GM_VEL ? (float)vel : (float)(sh.y[a][p] + kp.dt * vel);
      }
    }
  }
  if (a < D) sh.o[p * D + a] = row;
  __syncthreads();
  const int np = min(PB, kp.N - base);
  float *dst = MODE == GM_EXPLICIT ? A.q_io : A.out;
  if ((int)threadIdx.x < np * D) dst[(size_t)base * D + threadIdx.x] = sh.o[threadIdx.x];
  if constexpr (MODE == GM_EXPLICIT) {
    if (kp.spring == 1 && on && al == 0) {
      double n2 = 0.0;
#pragma unroll
      for (int b = 0; b < S; ++b) n2 += (double)sh.o[p * D + a + b] * sh.o[p * D + a + b];
      if (!(n2 < kp.b)) vds_flag(A.err, VDS_EDOMAIN);
    }
    for (int x = threadIdx.x; x < np * DP; x += NT) {
      const int pp = x / DP, d = x - pp * DP;
      A.rec[(size_t)base * DP + x] = d < D ? kp.c * sh.o[pp * D + d] : 0.f;
    }
  }
  if constexpr (MODE == GM_IMPLICIT_DIR) {
    double v[3] = {dec, dmax, ymax}, o[3];
    const bool mx[3] = {false, true, true};
    if (grid_reduce<3, NT, PB * D>(v, mx, A.red, A.ticket, o)) {
      if (!(fabs(o[0]) <= 1e300)) vds_flag(A.err, VDS_ENAN);
      if (A.imp.st) imp_after_grad(A.imp.st, o[0] / (double)kp.N, o[1], o[2], A.err);
    }
  }
}

template <int D, int S>
__global__ void __launch_bounds__(FinCfg<D>::NT) k_dens_finish(PartSrc src, KParams kp, FinArgs A) {
  FinPtrs P;
  if (!imp_take(A, false, P)) return;
  using F = FinCfg<D>;
  constexpr int PB = F::PB, SH = D * F::SPL;  // shares of a particle's partial sums
  __shared__ FinShared<D, PB> sh;
  __shared__ float2 ps[SH][PB];
  const int base = blockIdx.x * PB;
  const int p = threadIdx.x % PB, u = threadIdx.x / PB, i = base + p;
  // the particle's threads share its partial sums, and the shares are added in order
  Sum2 s;
  if (i < kp.N) {
    int nseg;
    const int n = part_count(src, i, nseg);
    for (int x = u; x < n; x += SH) s.add(part_get<1>(src, i, 0, x, nseg));
  }
  ps[u][p] = make_float2(s.s, s.c);
  __syncthreads();
  Sum2 t;
#pragma unroll
  for (int b = 0; b < SH; ++b) t.add(ps[b][p]);
  fin_density<D, S, PB, F::NT>(kp, A, P, base, t.value(), sh);
}

template <int D, int S, int MODE>
__global__ void __launch_bounds__(FinCfg<D>::NT) k_grad_finish(PartSrc src, KParams kp, FinArgs A) {
  FinPtrs P;
  if (!imp_take(A, true, P)) return;
  using F = FinCfg<D>;
  constexpr int PB = F::PB, SPL = F::SPL;
  __shared__ FinShared<D, PB> sh;
  __shared__ float2 ps[SPL][D][PB];
  const int base = blockIdx.x * PB;
  const int p = threadIdx.x % PB, u = threadIdx.x / PB, i = base + p;
  const int a = u % D, share = u / D;
  Sum2 s[4];
  if (i < kp.N) {
    int nseg;
    const int n = part_count(src, i, nseg);
    for (int x = share; x < n; x += 4 * SPL)
#pragma unroll
      for (int v = 0; v < 4; ++v)
        if (x + v * SPL < n) s[v].add(part_get<D>(src, i, a, x + v * SPL, nseg));
#pragma unroll
    for (int v = 1; v < 4; ++v) s[0].add(make_float2(s[v].s, s[v].c));
  }
  double sum = 0.0;
  if constexpr (SPL > 1) {
    ps[share][a][p] = make_float2(s[0].s, s[0].c);
    __syncthreads();
    if (share == 0)
#pragma unroll
      for (int v = 1; v < SPL; ++v) s[0].add(ps[v][a][p]);
  }
  sum = s[0].value();
  fin_grad<D, S, MODE, PB, F::NT>(kp, A, P, base, sum, sh);
}

}  // namespace vds_pair
