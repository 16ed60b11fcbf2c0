#pragma once
// pair_small.cuh -- the pair passes of small clouds, each one launch with its
// epilogue.  Included by pair_impl.cuh.
//
// A small cloud's passes are bound by launches and latency, not arithmetic: at
// N = 1000, D = 9 a pass is 1 us of FP32 work, and pass + epilogue took four
// launches and 23 us a step.  Here a CTA owns PB = 8 RI particles and sums
// over all others, so it can go on to the epilogue at once (no partial sums in
// global memory, no second launch).  A warp's lanes are 8 particles x 4
// records: a record is read once per CTA (from L2) by one group of 8 lanes,
// the sums of a particle need two shuffles and one sum over the warps.
// Ordered pairs: the two-fold work of k_sym's is the lesser price here.
// N = 1000, D = 9: 23.3 -> 11.7 us a step (the L2 latency of the records and
// the FP64 chain of the epilogue); programmatic dependent launches gave nothing.
//
// Sums: FP32 over a lane's records (48 at most: more are cut in two chains) and
// its 4 lanes, two-sum over the warps in order.

namespace vds_pair {

constexpr int SM_DENS = -1;  // MODE of the density pass; a GradMode otherwise
// Least CTAs per SM (0: the compiler's own register budget), by what was faster
// for a dimension: with two chains N = 4800, D = 2 28.0 -> 22.8 us a step, D = 9
// 57 -> 51, D = 10 69 -> 58; N = 6000, D = 4 58 -> 52 (one chain: 22.9, 52, 67, 46);
// five implicit steps of N = 512, D = 2 687 -> 645 us (32 registers by itself).
constexpr int sm_minb(int D, int RI, int NT, bool dens, bool imp) {
  if (RI == 1) return imp && NT == 1024 && D <= 9 ? 1 : 0;
  if (D == 2 || (D == 3 && !imp) || (D >= 8 && D <= 10)) return 1;
  return D == 4 && !dens ? 3 : D == 16 && dens ? 2 : 0;
}
// From here on (16 warps: 48 records a lane) a lane's records go in two chains,
// each two-summed over the warps.  Relative error of the gradient at N = 6000,
// D = 3, mean of 12 clouds: one chain of 94 1.90e-7, two of 47 1.73e-7 (the
// ordered passes' chains of 64 and Kahan sums 1.72e-7).
constexpr int SM_TWO_N = 3073;

template <int D, int S, int RI, int NT, int MODE>
__global__ void __launch_bounds__(NT, sm_minb(D, RI, NT, MODE == SM_DENS, MODE == GM_IMPLICIT_DIR)) k_small(const float *rec, KParams kp, FinArgs A) {
  constexpr bool GRAD = MODE != SM_DENS;
  constexpr int DP = Rec<D>::DP, ACC = GRAD ? D : 1, PB = 8 * RI, W = NT / 32;
  constexpr int V = (D + (GRAD ? 1 : 0) + 3) / 4;
  static_assert(NT >= PB * D, "the epilogue's threads");
  __shared__ FinShared<D, PB> sh;
  __shared__ float red[W][ACC][PB];
  const int tid = threadIdx.x, w = tid >> 5, li = tid & 7, lj = (tid >> 3) & 3;
  const int base = blockIdx.x * PB, N = kp.N;
  FinPtrs P;
  if (!imp_take(A, GRAD, P)) return;
  float xi[RI][D], wi[RI], acc[RI][ACC];
#pragma unroll
  for (int k = 0; k < RI; ++k) {
    const int i = min(base + li + 8 * k, N - 1);
    const float *r = rec + (size_t)i * DP;
#pragma unroll
    for (int d = 0; d < D; ++d) xi[k][d] = r[d];
    wi[k] = GRAD ? r[D] : 0.f;
#pragma unroll
    for (int a = 0; a < ACC; ++a) acc[k][a] = 0.f;
  }
  auto chain = [&](int j0, int j1) {  // the records [j0, j1) into acc
#pragma unroll 4
    for (int j = j0 + w * 4 + lj; j < j1; j += W * 4) {
      float xj[4 * V];
#pragma unroll
      for (int v = 0; v < V; ++v) {
        const float4 f = reinterpret_cast<const float4 *>(rec + (size_t)j * DP)[v];
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
  };
  const int p = tid % PB, a = tid / PB;
  Sum2 s;
  auto gather = [&]() {  // the lanes' sums of acc added to s, warp after warp
#pragma unroll
    for (int k = 0; k < RI; ++k)
#pragma unroll
      for (int b = 0; b < ACC; ++b) {
        float v = acc[k][b];
        v += __shfl_xor_sync(0xffffffffu, v, 8);
        v += __shfl_xor_sync(0xffffffffu, v, 16);
        if (lj == 0) red[w][b][li + 8 * k] = v;
      }
    __syncthreads();
    if (a < D)
#pragma unroll
      for (int x = 0; x < W; ++x) s.add(make_float2(red[x][GRAD ? a : 0][p], 0.f));
  };
  const bool two = RI > 1 && N >= SM_TWO_N;  // RI = 1 has 2432 records at most
  const int mid = two ? N / 2 : N;
  chain(0, mid);
  if (two) {
    gather();
#pragma unroll
    for (int k = 0; k < RI; ++k)
#pragma unroll
      for (int b = 0; b < ACC; ++b) acc[k][b] = 0.f;
    chain(mid, N);
    __syncthreads();  // red has been read
  }
  gather();
  if constexpr (GRAD) fin_grad<D, S, MODE, PB, NT>(kp, A, P, base, s.value(), sh);
  else fin_density<D, S, PB, NT>(kp, A, P, base, s.value(), sh);
}

}  // namespace vds_pair
