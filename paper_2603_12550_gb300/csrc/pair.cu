// pair.cu -- dispatch of the pair passes over the supported D = nb*s and the
// parameters they take; the kernels themselves are in pair_impl.cuh,
// instantiated once per D in pair_d<D>.cu.
#include <math.h>

#include "pair.cuh"
#include "pair_impl.cuh"

namespace {
// End of an implicit step: q = q* + d, d = d[cur] (- dir) kept for the next
// step's start; the last CTA closes the step.
__global__ void __launch_bounds__(256)
    k_imp_end(int n, ImpArgs imp, const float *__restrict__ qs, const float *__restrict__ dir, float *__restrict__ q,
              int *__restrict__ iters, unsigned *ticket) {
  ImpState *s = imp.st;
  if (s->phase != IMP_FINAL) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) {
    const float *dcur = s->cur ? imp.d[1] : imp.d[0];
    float *doth = s->cur ? imp.d[0] : imp.d[1];
    float d = dcur[i];
    if (s->fin_dir) d = d - 1.f * dir[i];
    doth[i] = d;
    q[i] = qs[i] + d;
  }
  __syncthreads();
  if (threadIdx.x != 0) return;
  __threadfence();
  if (atomicAdd(ticket, 1u) != gridDim.x - 1) return;
  *ticket = 0u;
  iters[s->step] = s->it;
  s->cur = 1 - s->cur;
  ++s->step;
  s->phase = s->status ? IMP_STOP : IMP_READY;
}

}  // namespace

// Supported D = nb * s with s in {2,3}, nb <= 8, D <= 16.
#define VDS_DISPATCH_D(D, CALL)                          \
  switch (D) {                                           \
    case 2: return CALL(2);                              \
    case 3: return CALL(3);                              \
    case 4: return CALL(4);                              \
    case 6: return CALL(6);                              \
    case 8: return CALL(8);                              \
    case 9: return CALL(9);                              \
    case 10: return CALL(10);                            \
    case 12: return CALL(12);                            \
    case 14: return CALL(14);                            \
    case 15: return CALL(15);                            \
    case 16: return CALL(16);                            \
    default: return VDS_EARG;                            \
  }

int vds_prep_2(vds_ctx *, const KParams &, const float *);
int vds_density_2(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_2(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_2(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_2(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_2(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_2(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_3(vds_ctx *, const KParams &, const float *);
int vds_density_3(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_3(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_3(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_3(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_3(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_3(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_4(vds_ctx *, const KParams &, const float *);
int vds_density_4(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_4(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_4(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_4(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_4(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_4(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_6(vds_ctx *, const KParams &, const float *);
int vds_density_6(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_6(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_6(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_6(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_6(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_6(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_8(vds_ctx *, const KParams &, const float *);
int vds_density_8(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_8(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_8(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_8(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_8(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_8(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_9(vds_ctx *, const KParams &, const float *);
int vds_density_9(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_9(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_9(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_9(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_9(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_9(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_10(vds_ctx *, const KParams &, const float *);
int vds_density_10(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_10(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_10(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_10(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_10(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_10(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_12(vds_ctx *, const KParams &, const float *);
int vds_density_12(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_12(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_12(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_12(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_12(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_12(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_14(vds_ctx *, const KParams &, const float *);
int vds_density_14(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_14(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_14(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_14(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_14(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_14(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_15(vds_ctx *, const KParams &, const float *);
int vds_density_15(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_15(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_15(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_15(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_15(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_15(vds_ctx *, const KParams &, const float *, const float *, int, float *);
int vds_prep_16(vds_ctx *, const KParams &, const float *);
int vds_density_16(vds_ctx *, const KParams &, float *, bool, const float *, const float *, const float *, const float *, const ImpArgs *);
int vds_grad_16(vds_ctx *, const KParams &, int, float *, const float *, const float *, const float *, const float *, float *, const ImpArgs *);
int vds_stress_16(vds_ctx *, const KParams &, const float *, double *, double *);
int vds_impbegin_16(vds_ctx *, const KParams &, const ImpArgs &, const float *, float *);
int vds_imptrial_16(vds_ctx *, const KParams &, const ImpArgs &, const float *, const float *);
int vds_query_16(vds_ctx *, const KParams &, const float *, const float *, int, float *);

int vds_rowsdens_2(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_2(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_3(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_3(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_4(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_4(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_6(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_6(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_8(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_8(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_9(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_9(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_10(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_10(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_12(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_12(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_14(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_14(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_15(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_15(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);
int vds_rowsdens_16(vds_ctx *, const KParams &, const float *, int, int, float *);
int vds_rowsgrad_16(vds_ctx *, const KParams &, const float *, const float *, int, int, int, float *);

KParams make_kparams(const vds_params *p, int N, int D) {
  KParams k;
  k.N = N;
  k.D = D;
  k.nb = p->nb;
  k.s = p->s;
  k.spring = p->spring;
  k.h = p->h;
  k.kBT = p->kBT;
  k.zeta = p->zeta;
  k.dt = p->dt;
  k.b = p->b;
  for (int j = 0; j < 8; ++j) k.H[j] = p->H[j];
  for (int j = 0; j < 9; ++j) k.kappa[j] = p->kappa[j];
  const double c = sqrt(1.4426950408889634 / (2.0 * p->h * p->h));  // log2(e)/(2h^2)
  k.c = (float)c;
  k.sfac = 1.0 / (p->h * p->h * (double)k.c);
  k.rzeta = 1.0 / p->zeta;
  k.zeta_dt = p->dt != 0.0 ? p->zeta / p->dt : 0.0;
  k.dt_zeta = p->dt / p->zeta;
  k.lnorm = -log((double)N) - 0.5 * D * log(2.0 * 3.14159265358979323846 * p->h * p->h);
  return k;
}

int pass_npad(int N) { return (N + vds_pair::TJ - 1) / vds_pair::TJ * vds_pair::TJ; }

int pass_prep(vds_ctx *c, const KParams &kp, const float *y) {
#define CALL(DD) vds_prep_##DD(c, kp, y)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int pass_density(vds_ctx *c, const KParams &kp, float *rho_out, bool want_energy,
                 const float *ybase, const float *ydelta, const float *qa, const float *qb,
                 const ImpArgs *imp) {
#define CALL(DD) vds_density_##DD(c, kp, rho_out, want_energy, ybase, ydelta, qa, qb, imp)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int pass_grad(vds_ctx *c, const KParams &kp, int mode, float *out, const float *ybase,
              const float *ydelta, const float *qa, const float *qb, float *q_io, const ImpArgs *imp) {
#define CALL(DD) vds_grad_##DD(c, kp, mode, out, ybase, ydelta, qa, qb, q_io, imp)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int pass_stress(vds_ctx *c, const KParams &kp, const float *q, double *tau, double *qq) {
#define CALL(DD) vds_stress_##DD(c, kp, q, tau, qq)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int imp_begin(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *q, float *qs) {
#define CALL(DD) vds_impbegin_##DD(c, kp, imp, q, qs)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int imp_trial(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *qs, const float *dir) {
#define CALL(DD) vds_imptrial_##DD(c, kp, imp, qs, dir)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int imp_end(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *qs, const float *dir, float *q,
            int *iters) {
  const int n = kp.N * kp.D;
  k_imp_end<<<(n + 255) / 256, 256, 0, c->stream>>>(n, imp, qs, dir, q, iters, c->ticket + TK_MISC);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

int pass_density_at(vds_ctx *c, const KParams &kp, const float *q, const float *y, int M, float *f_out) {
#define CALL(DD) vds_query_##DD(c, kp, q, y, M, f_out)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int pass_density_rows(vds_ctx *c, const KParams &kp, const float *q, int row0, int nrows, float *rho) {
#define CALL(DD) vds_rowsdens_##DD(c, kp, q, row0, nrows, rho)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}

int pass_grad_rows(vds_ctx *c, const KParams &kp, const float *q, const float *rho, int row0, int nrows,
                   int mode, float *out) {
#define CALL(DD) vds_rowsgrad_##DD(c, kp, q, rho, row0, nrows, mode, out)
  VDS_DISPATCH_D(kp.D, CALL)
#undef CALL
}
