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
// Sums: FP32 over a lane's N / (4 warps) records and its 4 lanes, two-sum
// over the warps in order.

namespace vds_pair {

constexpr int SM_DENS = -1;  // MODE of the density pass; a GradMode otherwise

template <int D, int S, int RI, int NT, int MODE>
__global__ void __launch_bounds__(NT) k_small(const float *rec, KParams kp, FinArgs A) {
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
#pragma unroll 4
  for (int j = w * 4 + lj; j < N; j += W * 4) {
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
#pragma unroll
  for (int k = 0; k < RI; ++k)
#pragma unroll
    for (int a = 0; a < ACC; ++a) {
      float v = acc[k][a];
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      if (lj == 0) red[w][a][li + 8 * k] = v;
    }
  __syncthreads();
  const int p = tid % PB, a = tid / PB;
  Sum2 s;
  if (a < D)
#pragma unroll
    for (int x = 0; x < W; ++x) s.add(make_float2(red[x][GRAD ? a : 0][p], 0.f));
  if constexpr (GRAD) fin_grad<D, S, MODE, PB, NT>(kp, A, P, base, s.value(), sh);
  else fin_density<D, S, PB, NT>(kp, A, P, base, s.value(), sh);
}

}  // namespace vds_pair
