// pair.cuh -- host-side interface of the O(N^2) Gaussian-kernel pair passes
// and their fused epilogues (pair.cu).
#pragma once
#include "vds_internal.cuh"

// Stream-K schedule of a pair pass: the (i-tile, j-chunk) items of the N x N
// pair square, flattened i-tile major, are split into G contiguous equal
// ranges, one per CTA of a grid sized to the resident capacity of the GPU.
// A CTA accumulates in registers while its i-tile is unchanged and writes one
// partial (an FP32 sum and its compensation) per (i-tile, segment, component);
// an epilogue sums the segments of each i-tile in a fixed order, so results do
// not depend on timing.
// With cpt > 0 (the symmetric passes) i-tile t takes the j-chunks from its
// own first one on, cpt per tile: the upper triangle of the square.
struct Sched {
  long long items;  // sched_start(n_itiles)
  int G;            // CTAs
  int nchunk;       // j-chunks
  int cpt;          // j-chunks per i-tile left out below the diagonal (0: none)
  int n_itiles;
  int maxseg;       // max segments per i-tile
  int TI;           // particles per i-tile
  int Npad;         // N rounded up to a multiple of TJ (j records)
  int Nipad;        // rows of the i-record array (= Npad unless the i points
                    // are other points than the particles, as for queries)
};

__host__ __device__ __forceinline__ int sched_first_cta(long long x, const Sched &s) {
  return (int)(((x + 1) * (long long)s.G + s.items - 1) / s.items - 1);
}

// First item of i-tile t (t <= n_itiles).
__host__ __device__ __forceinline__ long long sched_start(int t, const Sched &s) {
  return (long long)t * s.nchunk - (long long)s.cpt * ((long long)t * (t - 1) / 2);
}

// Symmetric passes: partials of the j side, one row of sums per i-tile t
// and component over the particles of the tiles after it, [t][component][j -
// (t + 1) TI].  Columns of row t, and the row's first element per component.
__host__ __device__ __forceinline__ long long sched_jcols(int t, const Sched &s) {
  return (long long)(s.nchunk - (t + 1) * s.cpt) * (s.TI / s.cpt);
}
__host__ __device__ __forceinline__ long long sched_jrow(int t, const Sched &s) {
  return ((long long)t * s.nchunk - (long long)s.cpt * ((long long)t * (t + 1) / 2)) * (s.TI / s.cpt);
}

// The implicit step's minimiser as the device runs it (vds_capi.cu): which
// evaluation comes next, and the line search's state.  Kernels launched for an
// evaluation that is not due return at once.
enum ImpPhase {
  IMP_READY = 0,  // between steps (begun by k_imp_begin while step < nsteps)
  IMP_TRIAL = 1,  // density at the trial point
  IMP_GRAD = 2,   // gradient and direction at the accepted point
  IMP_FINAL = 3,  // the step's update of q
  IMP_STOP = 4    // failed
};
struct ImpState {
  double J, alpha, dec;
  double tol, jfloor;
  int phase, it, ls, cur, fin_dir, status;
  int start;   // the trial is the step's first point
  int cold;    // ... without the previous step's correction
  int step, nsteps, max_iter, pad;
};
__device__ __forceinline__ bool imp_due(const ImpState *s, bool grad) {
  const int ph = s->phase;
  return grad ? ph == IMP_GRAD : (ph == IMP_TRIAL || (ph == IMP_READY && s->step < s->nsteps));
}
// What a minimiser's passes take: its state and the two displacement buffers
// (the accepted one is d[cur], the trial's d[1 - cur]).
struct ImpArgs {
  ImpState *st = nullptr;
  float *d[2] = {nullptr, nullptr};
};

// Physical parameters as the kernels see them.
struct KParams {
  int N, D, nb, s, spring;
  float c;          // coordinate scale: qhat = c q, khat = exp2(-|dqhat|^2)
  double h, kBT, zeta, dt, b;
  double H[8];
  double kappa[9];
  double lnorm;     // -ln N - (D/2) ln(2 pi h^2)
  double sfac;      // S = -sfac * sum u dqhat, sfac = 1/(h^2 c)
  // ratios the epilogues use, so that no FP64 division is on their chain
  double rzeta, zeta_dt, dt_zeta;  // 1/zeta, zeta/dt and dt/zeta (0 where dt = 0)
};

KParams make_kparams(const vds_params *p, int N, int D);

// Rows of the record array written by pass_prep for N particles: N rounded
// up to the pair passes' j-tile.
int pass_npad(int N);
// Records of y scaled by c, with w = 0, in ctx->rec; the rows beyond N far away
// (kernel value 0).
int pass_prep(vds_ctx *c, const KParams &kp, const float *y);

// Density pass: rho_I over all J, then the epilogue: w_I = 1/rho_I into the
// records, optional rho output, and when want_energy, the FP64 energy
//   (1/N) sum_I [kBT (ln rho_I + lnorm) + Psi(y_I)]
//   + (zeta/2dt)(1/N) sum_I dI^T (A^-1 (x) I) dI,   dI = qa_I - qb_I
// (the quadratic term only when qa != NULL; qb may be NULL) into scal[SC_E].
// y_I = ybase_I + ydelta_I (ydelta may be NULL).  imp (pass_grad too): the
// pass of a device-run minimiser, with its displacements in place of ydelta
// and qa, and its next state set by the epilogue.
int pass_density(vds_ctx *c, const KParams &kp, float *rho_out, bool want_energy,
                 const float *ybase, const float *ydelta, const float *qa, const float *qb,
                 const ImpArgs *imp = nullptr);

// The same density without the energy, with the pair dot products on the
// tensor cores (dens_tc.cu: 3xTF32; 1e-5 relative for the median particle of
// an equilibrium cloud, 1e-4 at its outermost, more on stretched clouds): w_I = 1/rho_I
// into the records (which must come from pass_prep), optional rho output.
// D = 6 and 9 only; VDS_EARG otherwise, and the caller takes pass_density.
int pass_density_tc(vds_ctx *c, const KParams &kp, float *rho_out);
// The operand images of that density (a_I rows and b_J rows, TF32 hi/lo
// split, 128 bytes per row, rows [0, pass_npad(N)) in 8-row groups of 1024
// bytes) from the records in ctx->rec, into the context's workspace: for the
// refresh, which forms its kernel values from the same dot products.  D = 6
// and 9 only (VDS_EARG otherwise).
int pass_density_tc_images(vds_ctx *c, int N, int D, const uint8_t **aimg, const uint8_t **bimg);

// Gradient pass (records must hold w from pass_density) and its epilogues.
enum GradMode { GM_OUT = 0, GM_EXPLICIT = 1, GM_IMPLICIT_DIR = 2, GM_VEL = 3 };
// GM_OUT: g = kBT S + grad Psi(y) (+ (zeta/dt)(A^-1 (x) I)(qa - qb) if qa).
// GM_EXPLICIT: q_io += dt [kappa q - (1/zeta)(A (x) I) g]; rebuild records.
// GM_VEL: out = kappa y - (1/zeta)(A (x) I) g (the particle velocity).
// GM_IMPLICIT_DIR: dir = d + (dt/zeta)(A (x) I) g with d the minimiser's accepted
//   displacement; its state takes (1/N) sum <G, dir>, G = (zeta/dt)(A^-1 (x) I) d
//   + g, max|dir| and max|y|.
int pass_grad(vds_ctx *c, const KParams &kp, int mode, float *out,
              const float *ybase, const float *ydelta, const float *qa,
              const float *qb, float *q_io, const ImpArgs *imp = nullptr);

// Stress and second moments (FP64) into host arrays.
int pass_stress(vds_ctx *c, const KParams &kp, const float *q, double *tau, double *qq);

// Kernel density estimate at M query points y (M x D):
//   f_out[J] = (1/N)(2 pi h^2)^(-D/2) sum_I exp(-|y_J - q_I|^2 / (2 h^2)),
// the particles' records built from q, the queries' in their own buffer.
int pass_density_at(vds_ctx *c, const KParams &kp, const float *q, const float *y, int M, float *f_out);

// The minimiser's own kernels (an implicit step is begin, then passes and
// trial points by turns, then end; each returns at once where it is not due):
// imp_begin: q* = q + dt kappa q into qs, the start displacement into the
//   trial buffer, its records;
// imp_trial: trial displacement d[cur] - alpha dir, its records;
// imp_end: q = q* + d[cur] (- dir), which also becomes the next start.
int imp_begin(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *q, float *qs);
int imp_trial(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *qs, const float *dir);
int imp_end(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *qs, const float *dir, float *q,
            int *iters);

// Row-range passes (rows row0 .. row0 + nrows - 1 against all N columns):
// rho of the rows; and, given rho of all N particles, g of the rows (mode 0)
// or their explicit Euler update (mode 1) into out (nrows x D).
int pass_density_rows(vds_ctx *c, const KParams &kp, const float *q, int row0, int nrows, float *rho);
int pass_grad_rows(vds_ctx *c, const KParams &kp, const float *q, const float *rho, int row0, int nrows,
                   int mode, float *out);
