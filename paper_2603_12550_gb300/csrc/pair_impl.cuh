#pragma once
// pair_impl.cuh -- the O(N^2) Gaussian-kernel pair passes of the VDS hot path and
// their fused O(N) epilogues, for GB300 (sm_103a).
//
// k_pair is the ordered form (rows of any points against all particles): the
// queries, the row ranges and the allocation-free evaluation; a cloud against
// itself takes the symmetric form of pair_sym.cuh from sym_min_n() particles on.
//
// Density pass (Eq. model_DeteParAppr, denominators of Eq. model_DymRepPar):
//   rho_I = sum_J exp2(-|qhat_I - qhat_J|^2),  qhat = c q,  c^2 = log2(e)/(2h^2)
// Gradient pass (Eq. model_DymRepPar with grad K = -(x/h^2) K):
//   S_I = -(1/(h^2 c)) sum_J khat_IJ (w_I + w_J)(qhat_I - qhat_J),  w = 1/rho.
//
// Each CTA owns a contiguous range of (i-tile, j-chunk) items (stream-K),
// keeps RI particles per thread in registers and streams j-tiles of particle
// records through a ring of shared-memory stages filled by TMA bulk copies
// (cp.async.bulk + mbarrier transaction counts) issued by one thread.  All
// threads read the same record at a time (shared-memory broadcast).  Inside a
// j-tile sums are plain FP32; across tiles they are Kahan-compensated; across
// CTAs they are left as FP32 (sum, rest) pairs, which the epilogue adds by
// two-sums in a fixed order.
#include <math.h>

#include "pair.cuh"
#include "pair_fin.cuh"
#include "pair_small.cuh"
#include "pair_sym.cuh"

namespace vds_pair {

// Tile shape (overridable at build time for tuning sweeps).
#ifndef VDS_PAIR_TJ
#define VDS_PAIR_TJ 256
#endif
#ifndef VDS_PAIR_NSTAGE
#define VDS_PAIR_NSTAGE 3
#endif
constexpr int TJ = VDS_PAIR_TJ;          // records per j-tile (= j-chunk)
constexpr int NSTAGE = VDS_PAIR_NSTAGE;  // shared-memory ring depth

// Threads per CTA and particles per thread of each pass.  D = 9 takes the
// fastest shapes of a sweep on GB300 at N = 65536 (density 512 x 4, gradient
// 384 x 3: 2.46 + 3.86 ms against 2.51 + 3.99 ms for 256 x 4 in both); other
// D keep 256 threads, 4 particles per thread, 2 for the gradient above D = 9
// (255 registers).
template <int D>
struct PairCfg {
  static constexpr int NT_DENS = (D == 9) ? 512 : 256;
  static constexpr int RI_DENS = 4;
  static constexpr int NT_GRAD = (D == 9) ? 384 : 256;
  static constexpr int RI_GRAD = (D <= 6) ? 4 : (D == 9 ? 3 : (D <= 9 ? 4 : 2));
};

// Small clouds (the paper's P = 1000 workloads, the 2D dumbbell): with the
// shapes above the (i-tile, j-chunk) items would cover fewer than half the
// SMs (N = 1000 gives 4 items), so such passes take 128 threads of one
// particle and 64-record j-tiles instead (N = 1000: 128 items).  Explicit
// step on GB300: N = 1000, D = 9 131 -> 50 us; N = 512, D = 2 40 -> 23 us;
// N = 4096, D = 9 142 -> 102 us.
constexpr int NT_SMALL = 128, RI_SMALL = 1, TJ_SMALL = 64;

// ------------------------------------------------------------- pair kernel

// Records with a norm slot (D + 1): the squared norm of qhat, for the passes
// that form their dot products on the tensor cores.
template <int D>
struct HasNorm {
  static constexpr bool value = Rec<D>::DP >= D + 2;
};

template <int D, int RI, int NT, bool GRAD, int TJK = TJ>
__global__ void __launch_bounds__(NT)
    k_pair(const float *__restrict__ rec, const float *__restrict__ reci, Sched sc,
           float2 *__restrict__ part, int *__restrict__ err, const ImpState *imp = nullptr) {
  static_assert(TJ % TJK == 0, "j-tiles divide the record padding");
  constexpr int DP = Rec<D>::DP;
  constexpr int ACC = GRAD ? D : 1;
  constexpr uint32_t TILE_FLOATS = TJK * DP;
  constexpr uint32_t TILE_BYTES = TILE_FLOATS * 4;
  extern __shared__ __align__(128) float tiles[];  // NSTAGE * TILE_FLOATS
  __shared__ __align__(8) uint64_t full[NSTAGE];

  const int tid = threadIdx.x;
  const long long it0 = (long long)blockIdx.x * sc.items / sc.G;
  const long long it1 = (long long)(blockIdx.x + 1) * sc.items / sc.G;
  if (it0 >= it1 || (imp && !imp_due(imp, GRAD))) return;  // uniform over the CTA

  if (tid == 0) {
#pragma unroll
    for (int s = 0; s < NSTAGE; ++s) mbar_init(&full[s], 1);
    fence_mbar_init();
  }
  __syncthreads();
  if (tid == 0) {
    for (int s = 0; s < NSTAGE && it0 + s < it1; ++s) {
      const int ch = (int)((it0 + s) % sc.nchunk);
      mbar_arrive_expect_tx(&full[s], TILE_BYTES);
      bulk_g2s(tiles + s * TILE_FLOATS, rec + (size_t)ch * TILE_FLOATS, TILE_BYTES, &full[s]);
    }
  }

  float xi[RI][D];
  float wi[RI];
  float sum[RI][ACC], cmp[RI][ACC];
  int cur = -1, seg = 0;
  long long it_fail = -1;

  auto flush = [&]() {
#pragma unroll
    for (int k = 0; k < RI; ++k) {
      const int il = tid + k * NT;
#pragma unroll
      for (int a = 0; a < ACC; ++a)
        part[(((size_t)cur * sc.maxseg + seg) * ACC + a) * sc.TI + il] =
            make_float2(sum[k][a], -cmp[k][a]);
    }
  };

  for (long long it = it0; it < it1; ++it) {
    const int t = (int)(it / sc.nchunk);
    if (t != cur) {
      if (cur >= 0) flush();
      cur = t;
      seg = (int)blockIdx.x - sched_first_cta((long long)t * sc.nchunk, sc);
#pragma unroll
      for (int k = 0; k < RI; ++k) {
        int i = t * sc.TI + tid + k * NT;
        i = i < sc.Nipad ? i : sc.Nipad - 1;
        const float *r = reci + (size_t)i * DP;
#pragma unroll
        for (int d = 0; d < D; ++d) xi[k][d] = r[d];
        wi[k] = GRAD ? r[D] : 0.f;
#pragma unroll
        for (int a = 0; a < ACC; ++a) sum[k][a] = cmp[k][a] = 0.f;
      }
    }
    const int stage = (int)((it - it0) % NSTAGE);
    const uint32_t parity = (uint32_t)(((it - it0) / NSTAGE) & 1);
    const bool got = mbar_wait_bounded(&full[stage], parity, VDS_WAIT_LIMIT_NS);
    if (__syncthreads_or(!got)) {
      it_fail = it;
      break;
    }

    const float *tj = tiles + stage * TILE_FLOATS;
    float acc[RI][ACC];
#pragma unroll
    for (int k = 0; k < RI; ++k)
#pragma unroll
      for (int a = 0; a < ACC; ++a) acc[k][a] = 0.f;

#pragma unroll 2
    for (int j = 0; j < TJK; ++j) {
      float xj[DP];
      const float4 *pj = reinterpret_cast<const float4 *>(tj + j * DP);
#pragma unroll
      for (int v = 0; v < DP / 4; ++v) {
        const float4 f = pj[v];
        xj[4 * v + 0] = f.x;
        xj[4 * v + 1] = f.y;
        xj[4 * v + 2] = f.z;
        xj[4 * v + 3] = f.w;
      }
#pragma unroll
      for (int k = 0; k < RI; ++k) {
        float dd[D];
        dd[0] = xi[k][0] - xj[0];
        float r2 = dd[0] * dd[0];
#pragma unroll
        for (int d = 1; d < D; ++d) {
          dd[d] = xi[k][d] - xj[d];
          r2 = fmaf(dd[d], dd[d], r2);
        }
        const float e = ex2_approx(-r2);
        if constexpr (!GRAD) {
          acc[k][0] += e;
        } else {
          const float u = e * (wi[k] + xj[D]);
#pragma unroll
          for (int d = 0; d < D; ++d) acc[k][d] = fmaf(u, dd[d], acc[k][d]);
        }
      }
    }
    // Kahan-compensated accumulation of the tile sums
#pragma unroll
    for (int k = 0; k < RI; ++k)
#pragma unroll
      for (int a = 0; a < ACC; ++a) {
        const float y = acc[k][a] - cmp[k][a];
        const float tt = sum[k][a] + y;
        cmp[k][a] = (tt - sum[k][a]) - y;
        sum[k][a] = tt;
      }
    __syncthreads();  // stage fully consumed
    if (tid == 0 && it + NSTAGE < it1) {
      fence_proxy_async_smem();
      const int ch = (int)((it + NSTAGE) % sc.nchunk);
      mbar_arrive_expect_tx(&full[stage], TILE_BYTES);
      bulk_g2s(tiles + stage * TILE_FLOATS, rec + (size_t)ch * TILE_FLOATS, TILE_BYTES,
               &full[stage]);
    }
  }
  if (it_fail >= 0) {
    if (tid == 0) {
      vds_flag(err, VDS_ETIMEOUT);
      // copies for items it_fail .. it_fail+NSTAGE-1 may still be in flight:
      // give each a bounded chance to land before shared memory is released
      for (long long k = it_fail; k < it_fail + NSTAGE && k < it1; ++k)
        mbar_wait_bounded(&full[(k - it0) % NSTAGE], (uint32_t)(((k - it0) / NSTAGE) & 1),
                          VDS_WAIT_LIMIT_NS / 8);
    }
    return;
  }
  if (cur >= 0) flush();
}

// --------------------------------------------------------------- prep kernel

// Records of the N x D points y, and far ones up to Npad.
template <int D>
__global__ void k_prep(int N, int Npad, float c, const float *__restrict__ y, float *__restrict__ rec) {
  constexpr int DP = Rec<D>::DP;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Npad) return;
  float o[DP];
  if (i < N) {
#pragma unroll
    for (int d = 0; d < D; ++d) o[d] = c * y[(size_t)i * D + d];
  } else {
#pragma unroll
    for (int d = 0; d < D; ++d) o[d] = VDS_PAD_COORD;
  }
#pragma unroll
  for (int d = D; d < DP; ++d) o[d] = 0.f;
  if constexpr (HasNorm<D>::value) {
    // the squared norm, rounded as the tensor-core passes subtract it
    float nrm = o[0] * o[0];
#pragma unroll
    for (int d = 1; d < D; ++d) nrm = fmaf(o[d], o[d], nrm);
    o[D + 1] = nrm;
  }
  float4 *dst = reinterpret_cast<float4 *>(rec + (size_t)i * DP);
#pragma unroll
  for (int v = 0; v < DP / 4; ++v) dst[v] = make_float4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
}

// ------------------------------------------------------------ stress kernel

constexpr int STRESS_BP = 128;  // particles staged per block iteration

template <int D>
__global__ void __launch_bounds__(256)
    k_stress(KParams kp, const float *__restrict__ q, double *red, unsigned *ticket, double *scal,
             int *err) {
  __shared__ float ys[STRESS_BP][D];
  const int s = kp.s, ne_tau = s * s, ne = ne_tau + D * D;
  double acc[2] = {0.0, 0.0};  // entries tid and tid+256
  for (int base = blockIdx.x * STRESS_BP; base < kp.N; base += gridDim.x * STRESS_BP) {
    __syncthreads();
    for (int x = threadIdx.x; x < STRESS_BP * D; x += blockDim.x) {
      const int p = x / D, d = x - p * D;
      ys[p][d] = (base + p < kp.N) ? q[(size_t)(base + p) * D + d] : 0.f;
    }
    __syncthreads();
    if (kp.spring == 1 && threadIdx.x < STRESS_BP && base + threadIdx.x < kp.N) {
      const int p = threadIdx.x;
      for (int k = 0; k < kp.nb; ++k) {
        double n2 = 0.0;
        for (int a = 0; a < s; ++a) n2 += (double)ys[p][s * k + a] * ys[p][s * k + a];
        if (!(n2 < kp.b)) vds_flag(err, VDS_EDOMAIN);
      }
    }
    const int np = min(STRESS_BP, kp.N - base);
    for (int r = 0; r < 2; ++r) {
      const int e = threadIdx.x + r * 256;
      if (e >= ne) continue;
      double a = 0.0;
      if (e < ne_tau) {
        const int al = e / s, be = e - al * s;
        for (int p = 0; p < np; ++p) {
          for (int k = 0; k < kp.nb; ++k) {
            double f = kp.H[k];
            if (kp.spring == 1) {
              double n2 = 0.0;
              for (int c = 0; c < s; ++c) n2 += (double)ys[p][s * k + c] * ys[p][s * k + c];
              f = kp.H[k] / (1.0 - n2 / kp.b);
            }
            a += (double)ys[p][s * k + al] * f * (double)ys[p][s * k + be];
          }
        }
      } else {
        const int x = e - ne_tau, ra = x / D, rb = x - ra * D;
        for (int p = 0; p < np; ++p) a += (double)ys[p][ra] * (double)ys[p][rb];
      }
      acc[r] += a;
    }
  }
  // block partials of all entries, then ticketed final sum in block order
  __shared__ bool last;
  for (int r = 0; r < 2; ++r) {
    const int e = threadIdx.x + r * 256;
    if (e < ne) red[(size_t)blockIdx.x * ne + e] = acc[r];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int e = threadIdx.x; e < ne; e += blockDim.x) {
    double x = 0.0;
    for (unsigned b = 0; b < gridDim.x; ++b) x += __ldcg(red + (size_t)b * ne + e);
    scal[SC_AUX + e] = x / (double)kp.N;
  }
  __syncthreads();
  if (threadIdx.x == 0) *ticket = 0u;
}

// Record of y (scaled by c, everything behind it zero), or of a padding row.
template <int D>
__device__ __forceinline__ void put_record(float *rec, int i, float c, const float (&y)[D], bool pad) {
  constexpr int DP = Rec<D>::DP;
  float o[DP];
#pragma unroll
  for (int d = 0; d < DP; ++d) o[d] = 0.f;
#pragma unroll
  for (int d = 0; d < D; ++d) o[d] = pad ? VDS_PAD_COORD : c * y[d];
  float4 *dst = reinterpret_cast<float4 *>(rec + (size_t)i * DP);
#pragma unroll
  for (int v = 0; v < DP / 4; ++v) dst[v] = make_float4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
}

// Start of an implicit step: q* = q + dt kappa q, and the first trial y = q* +
// d with the previous step's correction d (none in a call's first step).
template <int D>
__global__ void k_imp_begin(KParams kp, ImpArgs imp, int Npad, const float *__restrict__ q, float *__restrict__ qs,
                            float *__restrict__ rec) {
  const ImpState *s = imp.st;
  if (s->phase != IMP_READY || s->step >= s->nsteps) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Npad) return;
  const bool on = i < kp.N;
  const float *dcur = s->cur ? imp.d[1] : imp.d[0];
  float *doth = s->cur ? imp.d[0] : imp.d[1];
  const bool cold = s->step == 0;
  float y[D];
  if (on) {
#pragma unroll
    for (int a = 0; a < D; ++a) y[a] = q[(size_t)i * D + a];
    float f[D];
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const int k = a / kp.s, al = a - k * kp.s;
      double v = 0.0;
#pragma unroll
      for (int b = 0; b < D; ++b)
        if (b / kp.s == k) v += kp.kappa[al * kp.s + (b - k * kp.s)] * (double)y[b];
      f[a] = (float)((double)y[a] + kp.dt * v);
    }
#pragma unroll
    for (int a = 0; a < D; ++a) {
      const float d = cold ? 0.f : dcur[(size_t)i * D + a];
      qs[(size_t)i * D + a] = f[a];
      doth[(size_t)i * D + a] = d;
      y[a] = f[a] + d;
    }
  }
  put_record<D>(rec, i, kp.c, y, !on);
}

// The next trial point: d[cur] - alpha dir (zero where the step starts cold).
template <int D>
__global__ void k_imp_trial(KParams kp, ImpArgs imp, const float *__restrict__ qs, const float *__restrict__ dir,
                            float *__restrict__ rec) {
  const ImpState *s = imp.st;
  if (s->phase != IMP_TRIAL) return;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= kp.N) return;
  const float *dcur = s->cur ? imp.d[1] : imp.d[0];
  float *doth = s->cur ? imp.d[0] : imp.d[1];
  const float al = (float)s->alpha;
  const bool zero = s->start != 0;
  float y[D];
#pragma unroll
  for (int a = 0; a < D; ++a) {
    const float d = zero ? 0.f : dcur[(size_t)i * D + a] - al * dir[(size_t)i * D + a];
    doth[(size_t)i * D + a] = d;
    y[a] = qs[(size_t)i * D + a] + d;
  }
  put_record<D>(rec, i, kp.c, y, false);
}

// ------------------------------------------------------------ host plumbing

// Most CTAs that share one i-tile.
inline int sched_maxseg(const Sched &sc) {
  int m = 1;
  for (int t = 0; t < sc.n_itiles; ++t) {
    const int f = sched_first_cta(sched_start(t, sc), sc);
    const int l = sched_first_cta(sched_start(t + 1, sc) - 1, sc);
    if (l - f + 1 > m) m = l - f + 1;
  }
  return m;
}

// i points: the Ni records at reci (the particles themselves unless a query
// pass); j points: the N particle records in c->rec.
template <int D, int RI, int NT, bool GRAD, int TJK = TJ>
int launch_pair(vds_ctx *c, int N, Sched &sc, int Ni, const float *reci, const ImpState *imp) {
  constexpr int DP = Rec<D>::DP;
  constexpr int ACC = GRAD ? D : 1;
  constexpr int TI = NT * RI;
  const size_t smem = (size_t)NSTAGE * TJK * DP * sizeof(float);
  // per device: the attribute is a property of the function on that device
  static int occ_dev[VDS_MAX_DEVICES] = {};
  int &occ = occ_dev[c->device < VDS_MAX_DEVICES ? c->device : 0];
  if (occ <= 0 || c->device >= VDS_MAX_DEVICES) {
    // large D needs more than the default 48 KB of dynamic shared memory
    VDS_CUDA_TRY(cudaFuncSetAttribute(k_pair<D, RI, NT, GRAD, TJK>,
                                      cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int o = 0;
    VDS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, k_pair<D, RI, NT, GRAD, TJK>, NT, smem));
    occ = o > 0 ? o : 1;
  }
  sc.TI = TI;
  sc.Npad = (N + TJ - 1) / TJ * TJ;
  sc.Nipad = (Ni + TJ - 1) / TJ * TJ;
  sc.nchunk = sc.Npad / TJK;
  sc.cpt = 0;
  sc.n_itiles = (Ni + TI - 1) / TI;
  sc.items = (long long)sc.n_itiles * sc.nchunk;
  const long long cap = (long long)c->num_sms * occ;
  sc.G = (int)(sc.items < cap ? sc.items : cap);
  sc.maxseg = sched_maxseg(sc);
  VDS_TRY(vds_ensure(c, c->part, (size_t)sc.n_itiles * sc.maxseg * TI * ACC * sizeof(float2)));
  const int pk = GRAD ? PK_GRADIENT : PK_DENSITY;
  VDS_TRY(vds_time_begin(c, pk));
  k_pair<D, RI, NT, GRAD, TJK><<<sc.G, NT, smem, c->stream>>>((const float *)c->rec.ptr, reci, sc,
                                                                     (float2 *)c->part.ptr, c->err, imp);
  VDS_CUDA_TRY(cudaGetLastError());
  VDS_TRY(vds_time_end(c, pk));
  ++c->launches;
  return VDS_OK;
}

template <int D>
int prep_impl(vds_ctx *c, const KParams &kp, const float *y) {
  const int Npad = (kp.N + TJ - 1) / TJ * TJ;
  VDS_TRY(vds_ensure(c, c->rec, (size_t)Npad * Rec<D>::DP * sizeof(float)));
  k_prep<D><<<(Npad + 255) / 256, 256, 0, c->stream>>>(kp.N, Npad, kp.c, y, (float *)c->rec.ptr);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

// One pair pass with the pass's shape, or the small-cloud shape when the
// former's items would cover fewer than half the SMs.  Between the two
// (fewer than 8 items per SM), the pass's shape takes 64-record j-chunks:
// four times the items, so that the last round of the stream-K split is
// not a large fraction of the pass (N = 10000 at D = 9: 200 and 360 items
// per pass at 256 records).
template <int D, bool GRAD>
int launch_pass(vds_ctx *c, int N, Sched &sc, int Ni, const float *reci, const ImpState *imp = nullptr) {
  constexpr int RI = GRAD ? PairCfg<D>::RI_GRAD : PairCfg<D>::RI_DENS;
  constexpr int NT = GRAD ? PairCfg<D>::NT_GRAD : PairCfg<D>::NT_DENS;
  const long long items = (long long)((Ni + NT * RI - 1) / (NT * RI)) * ((N + TJ - 1) / TJ);
  if (2 * items < c->num_sms) return launch_pair<D, RI_SMALL, NT_SMALL, GRAD, TJ_SMALL>(c, N, sc, Ni, reci, imp);
  if (items < 8LL * c->num_sms) return launch_pair<D, RI, NT, GRAD, TJ_SMALL>(c, N, sc, Ni, reci, imp);
  return launch_pair<D, RI, NT, GRAD>(c, N, sc, Ni, reci, imp);
}

// Shapes of the symmetric passes, from sweeps of particles per lane (RI),
// CTAs of 128 threads per SM (MINB: the register budget) and threads per CTA
// on GB300: the most particles per lane whose warps still fill the schedulers.
// Gradient, N = 65536, D = 9: RI = 6 at three CTAs 2.81 ms, 5 at three 2.95,
// 4 at four 3.18, 8 at two 3.20 (k_pair 3.86; with the folds of sym_run every
// 128 records, every 64 the first takes 2.93 in the bench).  D = 6: 8 at three 2.10, 6 at
// four 2.12.  Density, D = 9: 10 at three 1.36, 8 at four 1.49, 12 at two 1.42
// (k_pair 2.46).
template <int D, bool GRAD>
struct SymCfg {
  static constexpr int RI = GRAD ? (D == 2 ? 12 : D <= 6 ? 8 : D <= 9 ? 6 : D == 12 ? 5 : 4)
                                 : (D <= 4 ? 12 : D == 9 ? 10 : D <= 12 ? 8 : 4);
  static constexpr int MINB128 = GRAD ? (D <= 4 ? 4 : D <= 10 ? 3 : 2) : (D == 9 || D == 12 ? 3 : 4);
  static constexpr int NT_LARGE = MINB128 * 128;  // one CTA per SM
};

// The j sums of a symmetric pass may take this much workspace, and a quarter of
// the free memory; beyond either the pass takes the ordered form.
constexpr size_t SYM_MAX_PARTJ = (size_t)4 << 30;
// Smaller clouds take k_small.  Explicit step, k_small / symmetric passes:
// N = 4096, D = 2 25 / 29 us, D = 9 49 / 63, D = 16 72 / 75; N = 6144, D = 3
// 45 / 53, D = 6 76 / 81, D = 9 108 / 83.
template <int D>
constexpr int sym_min_n() { return D <= 6 ? 6145 : 4865; }
// From here on the gradient pass takes one CTA per SM: a third of the i-tiles
// and of the j sums written and read (N = 65536, D = 9: 65 instead of 199 MB).
constexpr int SYM_LARGE_N = 49152;
// j-chunks of 64 records in the density pass from here on; 32 below, where the
// items per CTA are few.
constexpr int SYM_CHUNK_N = 32768;

// The symmetric pass over the N records at c->rec; done = false (and nothing
// launched) where its workspace is over the limit or cannot be had.
template <int D, bool GRAD, int NT, int TJS>
int launch_sym(vds_ctx *c, int N, Sched &sc, const ImpState *imp, bool &done) {
  using C = SymCfg<D, GRAD>;
  constexpr int RI = C::RI, TI = NT * RI, ACC = GRAD ? D : 1, MINB = C::MINB128 * 128 / NT;
  constexpr size_t smem = SymSmem<D, RI, NT, GRAD, TJS>::BYTES;
  auto kern = k_sym<D, RI, NT, MINB, GRAD, TJS>;
  done = false;
  // per device: the attribute is a property of the function on that device
  static int occ_dev[VDS_MAX_DEVICES] = {};
  int &occ = occ_dev[c->device < VDS_MAX_DEVICES ? c->device : 0];
  if (occ <= 0 || c->device >= VDS_MAX_DEVICES) {
    VDS_CUDA_TRY(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    int o = 0;
    VDS_CUDA_TRY(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, kern, NT, smem));
    occ = o > 0 ? o : 1;
  }
  sc.TI = TI;
  sc.Npad = sc.Nipad = (N + TJ - 1) / TJ * TJ;  // rows of the record array
  sc.nchunk = (N + TJS - 1) / TJS;
  sc.cpt = TI / TJS;
  sc.n_itiles = (N + TI - 1) / TI;
  sc.items = sched_start(sc.n_itiles, sc);
  // CTAs per SM: all that fit, or the fewer of them whose largest share of an
  // SM's items is smaller by more than 3 % (N = 10007, D = 6, 64-thread CTAs:
  // 41.3 items per SM, which eight CTAs take as 8 x 6 and seven as 7 x 6)
  auto cost = [&](int o) {
    const long long g = (long long)c->num_sms * o;
    return o * ((sc.items + g - 1) / g);
  };
  int per = occ;
  for (int o = occ - 1; 2 * o >= occ; --o)
    if (100 * cost(o) < 97 * cost(per)) per = o;
  const long long cap = (long long)c->num_sms * per;
  sc.G = (int)(sc.items < cap ? sc.items : cap);
  sc.maxseg = sched_maxseg(sc);
  const size_t jbytes = (size_t)sched_jrow(sc.n_itiles - 1, sc) * ACC * sizeof(float2);
  if (jbytes > SYM_MAX_PARTJ) return VDS_OK;
  int st = jbytes ? vds_ensure_spare(c, c->partj, jbytes) : VDS_OK;
  if (st == VDS_OK) st = vds_ensure(c, c->part, (size_t)sc.n_itiles * sc.maxseg * TI * ACC * sizeof(float2));
  if (st == VDS_ENOMEM) {
    (void)cudaGetLastError();
    return VDS_OK;
  }
  VDS_TRY(st);
  const int pk = GRAD ? PK_GRADIENT : PK_DENSITY;
  VDS_TRY(vds_time_begin(c, pk));
  kern<<<sc.G, NT, smem, c->stream>>>((const float *)c->rec.ptr, sc, N, (float2 *)c->part.ptr,
                                      (float2 *)c->partj.ptr, imp);
  VDS_CUDA_TRY(cudaGetLastError());
  VDS_TRY(vds_time_end(c, pk));
  ++c->launches;
  done = true;
  return VDS_OK;
}

// The pass of the N particles at c->rec against themselves.
template <int D, bool GRAD>
int launch_self(vds_ctx *c, int N, PartSrc &src, const ImpState *imp) {
  bool done = false;
  if constexpr (GRAD) {
    if (N >= SYM_LARGE_N) VDS_TRY((launch_sym<D, true, SymCfg<D, true>::NT_LARGE, 32>(c, N, src.sc, imp, done)));
    else VDS_TRY((launch_sym<D, true, 128, 32>(c, N, src.sc, imp, done)));
  } else {
    if (N >= SYM_CHUNK_N) VDS_TRY((launch_sym<D, false, 128, 64>(c, N, src.sc, imp, done)));
    else VDS_TRY((launch_sym<D, false, 128, 32>(c, N, src.sc, imp, done)));
  }
  if (!done) VDS_TRY((launch_pass<D, GRAD>(c, N, src.sc, N, (const float *)c->rec.ptr, imp)));
  src.i = (const float2 *)c->part.ptr;
  src.j = (const float2 *)c->partj.ptr;
  return VDS_OK;
}

// Epilogue launches, by the space dimension S of D = nb S.
template <int D>
int launch_dens_finish(cudaStream_t st, const PartSrc &src, const KParams &kp, const FinArgs &A) {
  using F = FinCfg<D>;
  const int nb = (kp.N + F::PB - 1) / F::PB;
  if constexpr (D % 2 == 0)
    if (kp.s == 2) k_dens_finish<D, 2><<<nb, F::NT, 0, st>>>(src, kp, A);
  if constexpr (D % 3 == 0)
    if (kp.s == 3) k_dens_finish<D, 3><<<nb, F::NT, 0, st>>>(src, kp, A);
  VDS_CUDA_TRY(cudaGetLastError());
  return VDS_OK;
}

template <int D, int MODE>
int launch_grad_finish(cudaStream_t st, const PartSrc &src, const KParams &kp, const FinArgs &A) {
  using F = FinCfg<D>;
  const int nb = (kp.N + F::PB - 1) / F::PB;
  if constexpr (D % 2 == 0)
    if (kp.s == 2) k_grad_finish<D, 2, MODE><<<nb, F::NT, 0, st>>>(src, kp, A);
  if constexpr (D % 3 == 0)
    if (kp.s == 3) k_grad_finish<D, 3, MODE><<<nb, F::NT, 0, st>>>(src, kp, A);
  VDS_CUDA_TRY(cudaGetLastError());
  return VDS_OK;
}

// CTAs of an epilogue, each of which leaves up to three FP64 partials.
template <int D>
size_t fin_red_bytes(int N) {
  return (size_t)((N + FinCfg<D>::PB - 1) / FinCfg<D>::PB) * 3 * sizeof(double);
}

// Small clouds: pass and epilogue in one launch.
template <int D, int MODE, int RI, int NT>
int launch_small_shape(vds_ctx *c, const KParams &kp, const FinArgs &A) {
  const int nb = (kp.N + 8 * RI - 1) / (8 * RI);
  const float *rec = (const float *)c->rec.ptr;
  VDS_TRY(vds_ensure(c, c->red, (size_t)nb * 3 * sizeof(double)));
  FinArgs B = A;
  B.red = (double *)c->red.ptr;
  const int pk = MODE == SM_DENS ? PK_DENSITY : PK_GRADIENT;
  VDS_TRY(vds_time_begin(c, pk));
  if constexpr (D % 2 == 0)
    if (kp.s == 2) k_small<D, 2, RI, NT, MODE><<<nb, NT, 0, c->stream>>>(rec, kp, B);
  if constexpr (D % 3 == 0)
    if (kp.s == 3) k_small<D, 3, RI, NT, MODE><<<nb, NT, 0, c->stream>>>(rec, kp, B);
  VDS_CUDA_TRY(cudaGetLastError());
  VDS_TRY(vds_time_end(c, pk));
  ++c->launches;
  return VDS_OK;
}

// Particles per lane: one while that leaves at most two CTAs per SM; two or,
// where the registers of D = 8 to 10 make the most of it, four above (N = 4096:
// D = 3 34 / 33 / 31 us a step with 1 / 2 / 4, D = 6 57 / 36 / 41, D = 9
// 70 / 58 / 49, D = 16 136 / 72 / 108).
// 1024 threads per CTA where an SM has one CTA (or D leaves the registers for
// two), 512 otherwise: N = 1000, D = 9 11.7 / 14.3 / 19.0 us with 1024 / 512 /
// 256; N = 1536, D = 9 19.7 / 18.8.
template <int D, int MODE>
int launch_small(vds_ctx *c, const KParams &kp, const FinArgs &A) {
  constexpr int RI2 = D >= 8 && D <= 10 ? 4 : 2;
  if (kp.N > (D <= 10 ? 16 : 8) * c->num_sms) return launch_small_shape<D, MODE, RI2, 512>(c, kp, A);
  if (D <= 3 || kp.N <= 8 * c->num_sms) return launch_small_shape<D, MODE, 1, 1024>(c, kp, A);
  return launch_small_shape<D, MODE, 1, 512>(c, kp, A);
}

template <int D>
int density_impl(vds_ctx *c, const KParams &kp, float *rho_out, bool want_energy,
                 const float *ybase, const float *ydelta, const float *qa, const float *qb, const ImpArgs *imp) {
  FinArgs A{(float *)c->rec.ptr, rho_out, ybase, ydelta, qa, qb, nullptr, want_energy ? 1 : 0,
            nullptr, c->ticket + TK_DENS, c->scal, c->err, imp ? *imp : ImpArgs{}};
  if (kp.N < sym_min_n<D>()) return launch_small<D, SM_DENS>(c, kp, A);
  PartSrc src;
  VDS_TRY((launch_self<D, false>(c, kp.N, src, A.imp.st)));
  VDS_TRY(vds_ensure(c, c->red, fin_red_bytes<D>(kp.N)));
  A.red = (double *)c->red.ptr;
  VDS_TRY((launch_dens_finish<D>(c->stream, src, kp, A)));
  ++c->launches;
  return VDS_OK;
}

template <int D>
int grad_impl(vds_ctx *c, const KParams &kp, int mode, float *out, const float *ybase,
              const float *ydelta, const float *qa, const float *qb, float *q_io, const ImpArgs *imp) {
  FinArgs A{(float *)c->rec.ptr, out, ybase, ydelta, qa, qb, q_io, 0, nullptr, c->ticket + TK_GRAD, c->scal, c->err,
            imp ? *imp : ImpArgs{}};
  if (kp.N < sym_min_n<D>()) {
    if (mode == GM_OUT) return launch_small<D, GM_OUT>(c, kp, A);
    if (mode == GM_VEL) return launch_small<D, GM_VEL>(c, kp, A);
    if (mode == GM_IMPLICIT_DIR) return launch_small<D, GM_IMPLICIT_DIR>(c, kp, A);
    // the records of the next step go to the other array: CTAs that are still
    // summing read this one
    VDS_TRY(vds_ensure(c, c->rec2, (size_t)pass_npad(kp.N) * Rec<D>::DP * sizeof(float)));
    A.rec = (float *)c->rec2.ptr;
    VDS_TRY((launch_small<D, GM_EXPLICIT>(c, kp, A)));
    const DevBuf t = c->rec;
    c->rec = c->rec2;
    c->rec2 = t;
    return VDS_OK;
  }
  PartSrc src;
  VDS_TRY((launch_self<D, true>(c, kp.N, src, A.imp.st)));
  VDS_TRY(vds_ensure(c, c->red, fin_red_bytes<D>(kp.N)));
  A.red = (double *)c->red.ptr;
  if (mode == GM_OUT) VDS_TRY((launch_grad_finish<D, GM_OUT>(c->stream, src, kp, A)));
  else if (mode == GM_EXPLICIT) VDS_TRY((launch_grad_finish<D, GM_EXPLICIT>(c->stream, src, kp, A)));
  else if (mode == GM_VEL) VDS_TRY((launch_grad_finish<D, GM_VEL>(c->stream, src, kp, A)));
  else VDS_TRY((launch_grad_finish<D, GM_IMPLICIT_DIR>(c->stream, src, kp, A)));
  ++c->launches;
  return VDS_OK;
}

// f at the query points: the segment partials of each query summed in a
// fixed order, times (1/N)(2 pi h^2)^(-D/2).
constexpr int NT_FIN = 256;

template <int D>
__global__ void __launch_bounds__(NT_FIN)
    k_query_finish(PartSrc src, int M, double scale, float *__restrict__ f_out,
                   int *err) {
  const int i = blockIdx.x * NT_FIN + threadIdx.x;
  if (i >= M) return;
  int nseg;
  const int n = part_count(src, i, nseg);
  Sum2 t;
  for (int x = 0; x < n; ++x) t.add(part_get<1>(src, i, 0, x, nseg));
  const double s = t.value();
  if (!(s >= 0.0 && s <= 1e300)) vds_flag(err, VDS_ENAN);
  f_out[i] = (float)(s * scale);
}

template <int D>
int query_impl(vds_ctx *c, const KParams &kp, const float *q, const float *y, int M, float *f_out) {
  VDS_TRY(prep_impl<D>(c, kp, q));
  const int Mpad = (M + TJ - 1) / TJ * TJ;
  VDS_TRY(vds_ensure(c, c->recq, (size_t)Mpad * Rec<D>::DP * sizeof(float)));
  k_prep<D><<<(Mpad + 255) / 256, 256, 0, c->stream>>>(M, Mpad, kp.c, y, (float *)c->recq.ptr);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  PartSrc src;
  VDS_TRY((launch_pass<D, false>(c, kp.N, src.sc, M, (const float *)c->recq.ptr)));
  src.i = (const float2 *)c->part.ptr;
  src.j = nullptr;
  k_query_finish<D><<<(M + NT_FIN - 1) / NT_FIN, NT_FIN, 0, c->stream>>>(src, M,
                                                                         exp(kp.lnorm), f_out, c->err);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

// ------------------------------------------------- row-range passes
//
// The pair passes restricted to the particles row0 .. row0 + nrows - 1 as
// the rows I (all N particles as the columns J): the pieces of one
// evaluation split over ranks by rows (each rank holds all of q, and all of
// rho before its gradient pass).

// w = 1/rho of every particle into its record, from a gathered rho array.
template <int D>
__global__ void k_set_w(int N, const float *__restrict__ rho, float *__restrict__ rec, int *err) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const float r = rho[i];
  if (!(r >= 0.5f && r <= 3.0e38f)) vds_flag(err, VDS_ENAN);
  rec[(size_t)i * Rec<D>::DP + D] = (float)(1.0 / (double)r);
}

// The records of nrows consecutive particles (src already offset to row0)
// copied into their own array padded to Mpad rows, so a pass reads its i
// records from a buffer whose padding rows are far away (kernel value 0).
template <int D>
__global__ void k_copy_rows(int nrows, int Mpad, const float *__restrict__ src, float *__restrict__ dst) {
  constexpr int DP = Rec<D>::DP;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= Mpad) return;
  float4 *d = reinterpret_cast<float4 *>(dst + (size_t)i * DP);
  if (i < nrows) {
    const float4 *s = reinterpret_cast<const float4 *>(src + (size_t)i * DP);
#pragma unroll
    for (int v = 0; v < DP / 4; ++v) d[v] = s[v];
  } else {
    float o[DP];
#pragma unroll
    for (int a = 0; a < D; ++a) o[a] = VDS_PAD_COORD;
#pragma unroll
    for (int a = D; a < DP; ++a) o[a] = 0.f;
#pragma unroll
    for (int v = 0; v < DP / 4; ++v) d[v] = make_float4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
  }
}

template <int D>
int rows_records(vds_ctx *c, int row0, int nrows) {
  const int Mpad = (nrows + TJ - 1) / TJ * TJ;
  VDS_TRY(vds_ensure(c, c->recq, (size_t)Mpad * Rec<D>::DP * sizeof(float)));
  k_copy_rows<D><<<(Mpad + 255) / 256, 256, 0, c->stream>>>(nrows, Mpad, (const float *)c->rec.ptr +
                                                                             (size_t)row0 * Rec<D>::DP,
                                                           (float *)c->recq.ptr);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

// rho of the rows (FP32) from the density pass over all N columns.
template <int D>
int rows_density_impl(vds_ctx *c, const KParams &kp, const float *q, int row0, int nrows, float *rho_rows) {
  VDS_TRY(prep_impl<D>(c, kp, q));
  VDS_TRY(rows_records<D>(c, row0, nrows));
  PartSrc src;
  VDS_TRY((launch_pass<D, false>(c, kp.N, src.sc, nrows, (const float *)c->recq.ptr)));
  src.i = (const float2 *)c->part.ptr;
  src.j = nullptr;
  k_query_finish<D><<<(nrows + NT_FIN - 1) / NT_FIN, NT_FIN, 0, c->stream>>>(src, nrows, 1.0, rho_rows, c->err);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

// With rho of all N particles: the gradient pass for the rows, then either
// g = kBT S + grad Psi of the rows (mode 0) or their explicit Euler update
// (mode 1) into out (nrows x D).
template <int D>
int rows_grad_impl(vds_ctx *c, const KParams &kp, const float *q, const float *rho, int row0, int nrows,
                   int mode, float *out) {
  VDS_TRY(prep_impl<D>(c, kp, q));
  k_set_w<D><<<(kp.N + 255) / 256, 256, 0, c->stream>>>(kp.N, rho, (float *)c->rec.ptr, c->err);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  VDS_TRY(rows_records<D>(c, row0, nrows));
  PartSrc src;
  VDS_TRY((launch_pass<D, true>(c, kp.N, src.sc, nrows, (const float *)c->recq.ptr)));
  src.i = (const float2 *)c->part.ptr;
  src.j = nullptr;
  KParams kl = kp;
  kl.N = nrows;
  const FinArgs A{(float *)c->recq.ptr, mode == 0 ? out : nullptr, q + (size_t)row0 * D, nullptr, nullptr, nullptr,
                  mode == 0 ? nullptr : out, 0, nullptr, nullptr, c->scal, c->err, ImpArgs{}};
  if (mode == 0) VDS_TRY((launch_grad_finish<D, GM_OUT>(c->stream, src, kl, A)));
  else VDS_TRY((launch_grad_finish<D, GM_EXPLICIT>(c->stream, src, kl, A)));
  ++c->launches;
  return VDS_OK;
}

template <int D>
int stress_impl(vds_ctx *c, const KParams &kp, const float *q, double *tau, double *qq) {
  const int ne = kp.s * kp.s + D * D;
  int nblk = (kp.N + STRESS_BP - 1) / STRESS_BP;
  if (nblk > 2 * c->num_sms) nblk = 2 * c->num_sms;
  VDS_TRY(vds_ensure(c, c->red, (size_t)nblk * ne * sizeof(double)));
  k_stress<D><<<nblk, 256, 0, c->stream>>>(kp, q, (double *)c->red.ptr, c->ticket + TK_STRESS, c->scal,
                                          c->err);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  VDS_CUDA_TRY(cudaMemcpyAsync(c->h_scal, c->scal, SC_COUNT * sizeof(double), cudaMemcpyDeviceToHost,
                               c->stream));
  VDS_TRY(vds_sync_status(c));
  for (int e = 0; e < kp.s * kp.s; ++e) tau[e] = c->h_scal[SC_AUX + e];
  if (qq)
    for (int e = 0; e < D * D; ++e) qq[e] = c->h_scal[SC_AUX + kp.s * kp.s + e];
  return VDS_OK;
}

template <int D>
int imp_begin_impl(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *q, float *qs) {
  const int Npad = (kp.N + TJ - 1) / TJ * TJ;
  VDS_TRY(vds_ensure(c, c->rec, (size_t)Npad * Rec<D>::DP * sizeof(float)));
  k_imp_begin<D><<<(Npad + 127) / 128, 128, 0, c->stream>>>(kp, imp, Npad, q, qs, (float *)c->rec.ptr);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

template <int D>
int imp_trial_impl(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *qs, const float *dir) {
  k_imp_trial<D><<<(kp.N + 127) / 128, 128, 0, c->stream>>>(kp, imp, qs, dir, (float *)c->rec.ptr);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  return VDS_OK;
}

}  // namespace vds_pair

// One translation unit per supported D (pair_d<D>.cu) instantiates the passes
// through this macro, so the library builds in parallel.
#define VDS_PAIR_INSTANTIATE(DD)                                                              \
  int vds_prep_##DD(vds_ctx *c, const KParams &kp, const float *y) {                          \
    return vds_pair::prep_impl<DD>(c, kp, y);                                                 \
  }                                                                                           \
  int vds_density_##DD(vds_ctx *c, const KParams &kp, float *rho_out, bool want_energy,       \
                       const float *ybase, const float *ydelta, const float *qa,              \
                       const float *qb, const ImpArgs *imp) {                                 \
    return vds_pair::density_impl<DD>(c, kp, rho_out, want_energy, ybase, ydelta, qa, qb, imp); \
  }                                                                                           \
  int vds_grad_##DD(vds_ctx *c, const KParams &kp, int mode, float *out, const float *ybase,  \
                    const float *ydelta, const float *qa, const float *qb, float *q_io,       \
                    const ImpArgs *imp) {                                                     \
    return vds_pair::grad_impl<DD>(c, kp, mode, out, ybase, ydelta, qa, qb, q_io, imp);       \
  }                                                                                           \
  int vds_stress_##DD(vds_ctx *c, const KParams &kp, const float *q, double *tau, double *qq) { \
    return vds_pair::stress_impl<DD>(c, kp, q, tau, qq);                                      \
  }                                                                                           \
  int vds_impbegin_##DD(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *q, float *qs) { \
    return vds_pair::imp_begin_impl<DD>(c, kp, imp, q, qs);                                   \
  }                                                                                           \
  int vds_imptrial_##DD(vds_ctx *c, const KParams &kp, const ImpArgs &imp, const float *qs,    \
                        const float *dir) {                                                   \
    return vds_pair::imp_trial_impl<DD>(c, kp, imp, qs, dir);                                 \
  }                                                                                           \
  int vds_query_##DD(vds_ctx *c, const KParams &kp, const float *q, const float *y, int M,     \
                     float *f) {                                                              \
    return vds_pair::query_impl<DD>(c, kp, q, y, M, f);                                       \
  }                                                                                           \
  int vds_rowsdens_##DD(vds_ctx *c, const KParams &kp, const float *q, int row0, int nrows,    \
                        float *rho) {                                                         \
    return vds_pair::rows_density_impl<DD>(c, kp, q, row0, nrows, rho);                       \
  }                                                                                           \
  int vds_rowsgrad_##DD(vds_ctx *c, const KParams &kp, const float *q, const float *rho,       \
                        int row0, int nrows, int mode, float *out) {                          \
    return vds_pair::rows_grad_impl<DD>(c, kp, q, rho, row0, nrows, mode, out);               \
  }
