#pragma once
// pair_sym.cuh -- the O(N^2) pair passes over unordered pairs, for GB300
// (sm_103a).  Included by pair_impl.cuh.
//
// khat_IJ = khat_JI, so one kernel value serves both particles of a pair:
//   density   rho_I += khat, rho_J += khat:   2D + 2 FP32 lane-ops and one ex2
//             per unordered pair (2 (2D + 1) and two ex2 as ordered pairs);
//   gradient  u = khat (w_I + w_J), S_I += u dq, S_J -= u dq:   4D + 2 and one
//             ex2 (2 (3D + 2) and two ex2).
// The FP32 pipe bounds both passes, as it bounds the ordered form (k_pair).
// N = 65536, D = 9: density 2.46 -> 1.36 ms, gradient 3.86 -> 2.93 ms (ordered
// form -> this one); N = 16384, D = 3: 78 -> 51 and 128 -> 88 us.
//
// i-tiles of TI = NT x RI particles, j-chunks of TJS; tile t takes the chunks
// from its own first one on (Sched::cpt), the ones inside the tile as ordered
// pairs (i side only).  RI particles per lane stay in registers.  A lane must
// not share its j with the rest of its warp, or the j sums would need a
// reduction over lanes for every pair: so at step t of 32 lane l takes record
// (l + t) mod 32 of the chunk's slice and adds its RI values to that j's sums
// in a shared-memory slot array of the warp's own, conflict-free (float4
// planes, consecutive lanes on consecutive slots).  RI is the lever: the
// shared-memory traffic of a step (records, and the D sums in and out) is paid
// once per RI pairs of a lane.
//
// Sums: the i side in FP32 over 64 records,
// Kahan-compensated in shared memory across them; the j side in FP32 over the
// RI particles of a step, then over the 32 steps of a warp (one chain of 32 RI
// terms would save D of its 4D RI operations a step, 3 % of a pass, and double
// the gradient's error), Kahan-compensated over the CTA's warps.  Both leave (sum, compensation)
// pairs, which the epilogues add in a fixed order, so results do not depend on
// the schedule.

namespace vds_pair {

// The ACC sums of one j as float4 / float2 / float planes of TJS slots.
template <int ACC, int TJS>
struct JSlots {
  static constexpr int F4 = ACC / 4, F2 = (ACC % 4) / 2, F1 = ACC % 2;
  static constexpr int FLOATS = ACC * TJS;
  __device__ static __forceinline__ void load(const float *s, int j, float (&v)[ACC]) {
#pragma unroll
    for (int p = 0; p < F4; ++p) {
      const float4 f = reinterpret_cast<const float4 *>(s)[p * TJS + j];
      v[4 * p] = f.x;
      v[4 * p + 1] = f.y;
      v[4 * p + 2] = f.z;
      v[4 * p + 3] = f.w;
    }
    if constexpr (F2) {
      const float2 f = reinterpret_cast<const float2 *>(s + F4 * 4 * TJS)[j];
      v[4 * F4] = f.x;
      v[4 * F4 + 1] = f.y;
    }
    if constexpr (F1) v[ACC - 1] = s[(ACC - 1) * TJS + j];
  }
  __device__ static __forceinline__ void store(float *s, int j, const float (&v)[ACC]) {
#pragma unroll
    for (int p = 0; p < F4; ++p)
      reinterpret_cast<float4 *>(s)[p * TJS + j] = make_float4(v[4 * p], v[4 * p + 1], v[4 * p + 2], v[4 * p + 3]);
    if constexpr (F2) reinterpret_cast<float2 *>(s + F4 * 4 * TJS)[j] = make_float2(v[4 * F4], v[4 * F4 + 1]);
    if constexpr (F1) s[(ACC - 1) * TJS + j] = v[ACC - 1];
  }
  // float index of component a of slot j
  __device__ static __forceinline__ int at(int a, int j) {
    if (a < 4 * F4) return ((a >> 2) * TJS + j) * 4 + (a & 3);
    if (a < 4 * F4 + 2 * F2) return F4 * 4 * TJS + j * 2 + (a - 4 * F4);
    return (ACC - 1) * TJS + j;
  }
};

template <int D, int RI, int NT, bool GRAD, int TJS>
struct SymSmem {
  static constexpr int ACC = GRAD ? D : 1;
  // record planes read: coordinates, and the weight in the gradient pass
  static constexpr int V = (D + (GRAD ? 1 : 0) + 3) / 4;
  static constexpr size_t TILE = (size_t)2 * V * TJS * 16;
  static constexpr size_t JS = (size_t)2 * (NT / 32) * ACC * TJS * 4;
  static constexpr size_t KAHAN = (size_t)2 * RI * ACC * NT * 4;
  static constexpr size_t BYTES = TILE + JS + KAHAN;
};

// The pairs of i-tile t (TI particles) with the chunks [ca, cb), from the
// tile's own first chunk on, of the N records at rec: the i side's sums into
// ipart ([component][TI]), the j side's into jrow ([component][ncol], column 0
// the first record after the tile).  All threads of the CTA; sm_raw holds
// SymSmem::BYTES.  What it writes depends on nothing but the records, t, ca
// and cb.
template <int D, int RI, int NT, bool GRAD, int TJS>
__device__ __forceinline__ void sym_run(const float *__restrict__ rec, int N, int t, int ca, int cb,
                                        unsigned char *sm_raw, float2 *__restrict__ ipart, float2 *__restrict__ jrow,
                                        long long ncol) {
  using L = SymSmem<D, RI, NT, GRAD, TJS>;
  constexpr int DP = Rec<D>::DP, VG = DP / 4, V = L::V, ACC = L::ACC, W = NT / 32, TI = NT * RI;
  constexpr int CPT = TI / TJS;
  // records between two Kahan folds of the i side: at 128 the large gradient
  // tiles are 1.2 % faster, but their error at N = 50000, D = 9 is 1.27e-7
  // against 1.13e-7 (and k_pair's 1.13e-7)
  constexpr int FOLD = 64 / TJS;
  using JS = JSlots<ACC, TJS>;
  static_assert(TI % TJS == 0 && TJS % 32 == 0 && 64 % TJS == 0, "tile shapes");
  float4 *tile = reinterpret_cast<float4 *>(sm_raw);                   // [2][V][TJS]
  float *js = reinterpret_cast<float *>(sm_raw + L::TILE);             // [2][W][ACC x TJS]
  float *ks = reinterpret_cast<float *>(sm_raw + L::TILE + L::JS);     // [RI x ACC][NT] sums
  float *kc = ks + (size_t)RI * ACC * NT;                              // ... and compensations

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  auto stage = [&](int chunk, int buf) {
    const float4 *src = reinterpret_cast<const float4 *>(rec) + (size_t)chunk * TJS * VG;
    float4 *dst = tile + buf * V * TJS;
    const int n = N - chunk * TJS;
#pragma unroll
    for (int x0 = 0; x0 < V * TJS; x0 += NT) {
      const int x = x0 + tid;
      if (V * TJS % NT == 0 || x < V * TJS) {
        const int j = x / V, v = x - j * V;
        if (j < n) {
          cp_async16(dst + v * TJS + j, src + (size_t)j * VG + v);
        } else {  // past the last particle: no kernel value, no weight
          float o[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) o[k] = 4 * v + k < D ? VDS_PAD_COORD : 0.f;
          dst[v * TJS + j] = make_float4(o[0], o[1], o[2], o[3]);
        }
      }
    }
  };

  stage(ca, 0);

  float xi[RI][D], wi[RI], acc[RI][ACC];
  int nf = 0;
  const int i0 = warp * 32 * RI + lane;  // this lane's particles of the tile: i0 + 32 k
#pragma unroll
  for (int k = 0; k < RI; ++k) {
    const int i = t * TI + i0 + 32 * k;
    const float *r = rec + (size_t)(i < N ? i : 0) * DP;
#pragma unroll
    for (int d = 0; d < D; ++d) xi[k][d] = i < N ? r[d] : VDS_PAD_COORD;
    wi[k] = GRAD && i < N ? r[D] : 0.f;
#pragma unroll
    for (int a = 0; a < ACC; ++a) {
      acc[k][a] = 0.f;
      ks[(k * ACC + a) * NT + tid] = 0.f;
      kc[(k * ACC + a) * NT + tid] = 0.f;
    }
  }
  auto fold = [&]() {
#pragma unroll
    for (int k = 0; k < RI; ++k)
#pragma unroll
      for (int a = 0; a < ACC; ++a) {
        const int o = (k * ACC + a) * NT + tid;
        const float s = ks[o];
        const float y = acc[k][a] - kc[o];
        const float tt = s + y;
        kc[o] = (tt - s) - y;
        ks[o] = tt;
        acc[k][a] = 0.f;
      }
    nf = 0;
  };
  cp_async_wait_all();
  __syncthreads();
  for (int c = ca; c < cb; ++c) {
    const int b = (c - ca) & 1;
    // the next chunk's records arrive while this one is computed; its buffer
    // was read last before the barrier that ended the previous chunk
    if (c + 1 < cb) stage(c + 1, b ^ 1);

    const float4 *tl = tile + b * V * TJS;
    float *mj = js + (size_t)(b * W + warp) * JS::FLOATS;
    const bool diag = c < (t + 1) * CPT;
    if (diag) {
#pragma unroll 1
      for (int j = 0; j < TJS; ++j) {
        float xj[4 * V];
#pragma unroll
        for (int v = 0; v < V; ++v) {
          const float4 f = tl[v * TJS + j];
          xj[4 * v] = f.x;
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
    } else {
#pragma unroll 1
      for (int s0 = 0; s0 < TJS; s0 += 32) {
        float aj[ACC];
#pragma unroll
        for (int a = 0; a < ACC; ++a) aj[a] = 0.f;
        JS::store(mj, s0 + lane, aj);
        __syncwarp();
#pragma unroll 1
        for (int tt = 0; tt < 32; ++tt) {
          const int j = s0 + ((lane + tt) & 31);
          float xj[4 * V];
#pragma unroll
          for (int v = 0; v < V; ++v) {
            const float4 f = tl[v * TJS + j];
            xj[4 * v] = f.x;
            xj[4 * v + 1] = f.y;
            xj[4 * v + 2] = f.z;
            xj[4 * v + 3] = f.w;
          }
          JS::load(mj, j, aj);
          float ej[RI], tj[ACC];
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
              ej[k] = e;
            } else {
              const float u = e * (wi[k] + xj[D]);
#pragma unroll
              for (int d = 0; d < D; ++d) {
                acc[k][d] = fmaf(u, dd[d], acc[k][d]);
                tj[d] = k == 0 ? -u * dd[d] : fmaf(-u, dd[d], tj[d]);
              }
            }
          }
          if constexpr (GRAD) {
#pragma unroll
            for (int d = 0; d < D; ++d) aj[d] += tj[d];
          } else {
#pragma unroll
            for (int n = 1; n < RI; n *= 2)
#pragma unroll
              for (int k = 0; k + n < RI; k += 2 * n) ej[k] += ej[k + n];
            aj[0] += ej[0];
          }
          JS::store(mj, j, aj);
          __syncwarp();
        }
      }
    }
    if (++nf == FOLD) fold();
    cp_async_wait_all();
    __syncthreads();
    // the chunk's j sums over the warps, in order; this slot buffer is written
    // again only after the next chunk's barrier
    if (!diag) {
      float2 *row = jrow + (size_t)(c - (t + 1) * CPT) * TJS;
      const float *sb = js + (size_t)b * W * JS::FLOATS;
#pragma unroll 1
      for (int x = tid; x < TJS * ACC; x += NT) {
        const int a = x / TJS, j = x - a * TJS;
        const float *p = sb + JS::at(a, j);
        float s = 0.f, cm = 0.f;
#pragma unroll
        for (int w = 0; w < W; ++w) {
          const float y = p[w * JS::FLOATS] - cm;
          const float tt = s + y;
          cm = (tt - s) - y;
          s = tt;
        }
        row[(size_t)a * ncol + j] = make_float2(s, -cm);
      }
    }
  }
  fold();
#pragma unroll
  for (int k = 0; k < RI; ++k)
#pragma unroll
    for (int a = 0; a < ACC; ++a) {
      const int o = (k * ACC + a) * NT + tid;
      ipart[(size_t)a * TI + i0 + 32 * k] = make_float2(ks[o], -kc[o]);
    }
}

template <int D, int RI, int NT, int MINB, bool GRAD, int TJS>
__global__ void __launch_bounds__(NT, MINB)
    k_sym(const float *__restrict__ rec, Sched sc, int N, float2 *__restrict__ part, float2 *__restrict__ partj,
          const ImpState *imp) {
  constexpr int ACC = GRAD ? D : 1, TI = NT * RI, CPT = TI / TJS;
  extern __shared__ __align__(128) unsigned char sm_raw[];
  const long long it0 = (long long)blockIdx.x * sc.items / sc.G;
  const long long it1 = (long long)(blockIdx.x + 1) * sc.items / sc.G;
  if (it0 >= it1 || (imp && !imp_due(imp, GRAD))) return;  // uniform over the CTA
  // i-tile of the first item
  int t = 0, hi = sc.n_itiles;
  while (hi - t > 1) {
    const int m = (t + hi) >> 1;
    if (sched_start(m, sc) <= it0) t = m;
    else hi = m;
  }
  for (long long it = it0; it < it1; ++t) {
    const long long s = sched_start(t, sc), e = sched_start(t + 1, sc);
    const int ca = t * CPT + (int)(it - s), cb = t * CPT + (int)((e < it1 ? e : it1) - s);
    const int seg = (int)blockIdx.x - sched_first_cta(s, sc);
    sym_run<D, RI, NT, GRAD, TJS>(rec, N, t, ca, cb, sm_raw, part + ((size_t)t * sc.maxseg + seg) * ACC * TI,
                                  partj + (size_t)sched_jrow(t, sc) * ACC, sched_jcols(t, sc));
    it = e;
    __syncthreads();  // the next tile's first chunk reuses the buffers
  }
}

}  // namespace vds_pair
