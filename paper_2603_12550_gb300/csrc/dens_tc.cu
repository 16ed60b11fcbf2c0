// dens_tc.cu -- the density pass rho_I = sum_J exp2(-|qh_I - qh_J|^2)
// (Sec. 2.2's kernel density, qh the connectors scaled by sqrt(log2 e / 2h^2))
// with the pair dot products on the 5th-generation tensor cores, for passes
// held to 1e-4 rather than the full-order path's 1e-5: the density at the
// lifted state of the frozen reduced step's refresh, and the density of all
// particles that the surrogate's subset check needs.
//
// -|qh_I - qh_J|^2 = a_I . b_J - |qh_I|^2 with a_I = (qh_I, 1, 0...) and
// b_J = (2 qh_J, -|qh_J|^2, 0...), K = 16 columns.  One tcgen05.mma of kind
// tf32 (M = 128 rows I, N = 256 columns J, K = 8) takes TF32 operands, so each
// value is split into hi = tf32(x) and lo = tf32(x - hi) and the product is
// formed as hi.hi + hi.lo + lo.hi (six MMAs per 128 x 256 tile).  The tensor
// cores accumulate in FP32 rounding toward zero, so the large terms of the
// expansion (|qh|^2 of tens to hundreds) leave an error of a few FP32 ulps of
// them in the exponent: 1e-5 relative for the median particle of an
// equilibrium cloud, 3e-4 at the worst particle of a cloud stretched
// five-fold.  The products land in tensor memory; the epilogue warps read them
// (tcgen05.ld), subtract |qh_I|^2, take ex2 and sum, so the CUDA cores do two
// FP32 operations and one ex2 per pair instead of D + 2 operations and one
// ex2.  Two 256-column accumulators alternate, so the MMAs of one tile run
// while the epilogue reads the previous one.
//
// Operand images (one per 8-row group, 1024 bytes: the hi values in bytes
// 0..511 as K-major core matrices of 8 rows x 4 values, the lo values in
// bytes 512..1023 the same way), written by k_dt_prep from the pass records:
// element (r, k) of the hi part at (r/8)*1024 + (k/4)*128 + (r%8)*16 +
// (k%4)*4.  So one descriptor layout (core matrices 128 bytes apart along K,
// 8-row groups 1024 bytes apart) serves hi and lo, 512 bytes apart.  Rows
// past N: a_I = 0 (their sums are discarded), b_J with -1e30 in column D
// (exp2 of it is 0).
//
// The kernel matrix is symmetric, so only the tiles on and above the diagonal
// are formed: column tile c (256 particles) against the row tiles (128) before
// it, each exponential added to its row's sum and to its column's, and against
// its own two row tiles, whose columns' sums hold both orders.  N = 65536,
// D = 9: 0.75 -> 0.54 ms with the images and the finish (one ex2 per ordered
// pair before); N = 262144 10.5 -> 8.3 ms.  The epilogue warps' issue bounds it
// now (66 % of the slots, six instructions per pair of which four are the
// arithmetic; ex2 44 %, tensor 32 %).  Measured without effect: the three adds
// of a pair packed as f32x2 or not, 16 columns per tensor-memory load under
// one wait (slower: 0.66 ms), the side warps' sleep.
//
// Roles per CTA (one per SM; a contiguous range of the (column tile, row
// tile) list, column tile major): one thread bulk-copies the B image of a
// column tile (two slots) and the A images of the row tiles through a
// DT_NS-stage ring; one thread issues the MMAs; 16 warps read the accumulators
// (warp w: rows 32 (w % 4) + lane, columns 64 (w / 4) ..).  A thread keeps its
// 64 columns' sums in registers over the row tiles; every DT_FOLD tiles, and at
// the end of a column tile, the warp adds them over its lanes (31 exchanges per
// 32 columns) into Kahan-compensated sums, two columns a lane.  Row sums leave
// per tile: the four column groups' through shared memory to one more warp,
// which adds them and writes one FP32 sum per (row, column tile).
// Every wait is bounded; a wait that runs out sets the abort flag and the
// error status, and every role leaves its loop.  k_dt_finish adds a particle's
// row sums and column sums in a fixed order, so the result does not depend on
// the schedule.  The row sums of one launch take up to DT_ROW_BYTES (N^2 / 128
// bytes for a whole cloud: 0.54 GB at N = 262144); larger clouds go in several
// launches, a range of column tiles each.
#include "pair_impl.cuh"
#include "tcgen05.cuh"

namespace {

constexpr int DT_M = 128;                  // rows I per CTA (tensor-memory lanes)
constexpr int DT_N = 256;                  // columns J per MMA tile
constexpr int DT_K = 16;                   // padded dot-product length
constexpr int DT_NS = 6;                   // A ring stages
constexpr int DT_EW = 16;                  // epilogue warps (4 per tensor-memory lane quarter)
constexpr int DT_HC = DT_EW / 4;           // column groups
constexpr int DT_CW = DT_N / DT_HC;        // accumulator columns per epilogue warp
constexpr int DT_NT = (DT_EW + 3) * 32;    // + copy, MMA and row-sum warps
constexpr int DT_RB = 128;                 // image bytes per row (hi 64 + lo 64, interleaved by row group)
constexpr int DT_AB = DT_M * DT_RB;        // 16 KB
constexpr int DT_BB = DT_N * DT_RB;        // 32 KB
constexpr int DT_RS = 4;                   // row-sum buffers
constexpr int DT_FOLD = 64;                // row tiles between two folds of the column sums
constexpr size_t DT_SMEM = (size_t)DT_NS * DT_AB + 2 * (size_t)DT_BB;
constexpr size_t DT_ROW_BYTES = (size_t)1 << 30;  // row sums of one launch ...
constexpr size_t DT_ROW_LEAST = (size_t)1 << 23;  // ... or down to this many where memory is short

// Tiles (column tile c, row tile r <= 2 c + 1), c in [c0, c1), column tile
// major: first one of column tile c.  G CTAs take equal contiguous ranges.  The
// tiles of a launch are at most DT_ROW_BYTES / 512 and those of one column tile,
// times G below 2^32: 64-bit divisions took a microsecond of a small cloud's pass.
struct DtSched {
  int c0, c1, G, maxseg;
  unsigned items;
};
__host__ __device__ __forceinline__ unsigned dt_start(int c, const DtSched &s) {
  return (unsigned)((long long)c * (c + 1) - (long long)s.c0 * (s.c0 + 1));
}
// First row sum of column tile c (its rows are the 256 c before it).
__host__ __device__ __forceinline__ size_t dt_row(int c, const DtSched &s) {
  return (size_t)(DT_N / 2) * ((size_t)c * (c - 1) - (size_t)s.c0 * (s.c0 - 1));
}
__host__ __device__ __forceinline__ int dt_cta_of(unsigned x, const DtSched &s) {
  return (int)(((x + 1) * s.G + s.items - 1) / s.items - 1);
}

__device__ __forceinline__ uint32_t dt_off(int r, int k) {
  return (uint32_t)((r >> 3) * 1024 + (k >> 2) * 128 + (r & 7) * 16 + (k & 3) * 4);
}

// A and B images of rows [0, Npad) from the pass records (qh in slots 0..D-1,
// |qh|^2 in slot D + 1), one thread per (row, column k).
template <int D>
__global__ void k_dt_prep(const float *__restrict__ rec, int N, int Npad, uint8_t *__restrict__ aimg,
                          uint8_t *__restrict__ bimg) {
  constexpr int DP = Rec<D>::DP;
  const long e = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= (long)Npad * DT_K) return;
  const int r = (int)(e / DT_K), k = (int)(e % DT_K);
  float a = 0.f, b = 0.f;
  if (r < N) {
    const float *x = rec + (size_t)r * DP;
    if (k < D) {
      a = x[k];
      b = 2.f * x[k];
    } else if (k == D) {
      a = 1.f;
      b = -x[D + 1];
    }
  } else if (k == D) {
    b = -1e30f;
  }
  const float ah = to_tf32(a), bh = to_tf32(b);
  const size_t o = (size_t)dt_off(r, k);
  *reinterpret_cast<float *>(aimg + o) = ah;
  *reinterpret_cast<float *>(aimg + o + 512) = to_tf32(a - ah);
  *reinterpret_cast<float *>(bimg + o) = bh;
  *reinterpret_cast<float *>(bimg + o + 512) = to_tf32(b - bh);
}

// rho_I: the row sums that the column tiles of this launch left for particle
// I, and its column tile's sums, added in order to what earlier launches left
// (run, unless first); the last launch writes 1/rho into the pass records'
// weight slot (what the gradient passes read) and rho_out.  32 particles x 8
// shares per CTA.
__global__ void __launch_bounds__(256)
    k_dt_finish(DtSched sc, const float *__restrict__ rowp, const float2 *__restrict__ colp, int N, int DP, int wslot,
                int first, int last, float2 *__restrict__ run, float *__restrict__ rec, float *__restrict__ rho_out,
                int *err) {
  __shared__ float2 ps[8][32];
  const int p = threadIdx.x & 31, u = threadIdx.x >> 5, i = blockIdx.x * 32 + p;
  const int ci = i / DT_N;
  vds_pair::Sum2 s;
  if (i < N) {
    for (int c = max(ci + 1, sc.c0) + u; c < sc.c1; c += 8) s.add(make_float2(rowp[dt_row(c, sc) + i], 0.f));
    if (ci >= sc.c0 && ci < sc.c1) {  // four quarters of each CTA's part of the column tile: 72 at N = 4097
      const int f = dt_cta_of(dt_start(ci, sc), sc), l = dt_cta_of(dt_start(ci + 1, sc) - 1, sc);
      const float2 *col = colp + (size_t)(ci - sc.c0) * sc.maxseg * 4 * DT_N + (i - ci * DT_N);
#pragma unroll 4
      for (int g = u; g < 4 * (l - f + 1); g += 8) s.add(col[(size_t)g * DT_N]);
    }
  }
  ps[u][p] = make_float2(s.s, s.c);
  __syncthreads();
  if (u || i >= N) return;
  vds_pair::Sum2 t;
  if (!first) t.add(run[i]);
  for (int v = 0; v < 8; ++v) t.add(ps[v][p]);
  if (!last) {
    run[i] = make_float2(t.s, t.c);
    return;
  }
  const double rho = t.value();
  if (!(rho >= 0.5 && rho <= 1e300)) vds_flag(err, VDS_ENAN);
  rec[(size_t)i * DP + wslot] = (float)(1.0 / rho);
  if (rho_out) rho_out[i] = (float)rho;
}

// Wait for a barrier phase, giving up when another role has aborted or after
// the library's wait limit (then setting the abort flag).
__device__ __forceinline__ bool dt_wait(uint64_t *bar, uint32_t parity, volatile int *abort) {
  if (mbar_try_wait(bar, parity)) return true;
  const uint64_t t0 = global_timer_ns();
  for (uint32_t n = 0;; ++n) {
    if (mbar_try_wait_sleep(bar, parity)) return true;
    if ((n & 15u) == 15u) {
      if (*abort) return false;
      if (global_timer_ns() - t0 > VDS_WAIT_LIMIT_NS) {
        *abort = 1;
        return false;
      }
    }
  }
}

// Sums over the warp's lanes of 32 values per lane: lane l returns the sum of value l.
__device__ __forceinline__ float lane_sums(float (&x)[32], int lane) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float send = up ? x[i] : x[i + o], keep = up ? x[i + o] : x[i];
      x[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return x[0];
}

__device__ __forceinline__ void kahan(float v, float &s, float &c) {
  const float y = v - c, t = s + y;
  c = (t - s) - y;
  s = t;
}

// rowp[dt_row(c) + row] = sum over column tile c of exp2(a_row . b_J -
// |qh_row|^2) for the rows before the tile; colp[c - c0][segment][quarter]
// [column] = sum over a quarter (32 of 128 rows) of the segment's row tiles
// (those of the column tile itself included).
__global__ void __launch_bounds__(DT_NT, 1)
    k_dens_tc(const uint8_t *__restrict__ aimg, const uint8_t *__restrict__ bimg, const float *__restrict__ rec,
              int DP, int nslot, int N, DtSched sc, float *__restrict__ rowp, float2 *__restrict__ colp, int *err) {
  extern __shared__ __align__(1024) uint8_t dsm[];
  __shared__ __align__(8) uint64_t afull[DT_NS], aempty[DT_NS], bfull[2], bempty[2], accfull[2], accfree[2],
      rowfull[DT_RS], rowfree[DT_RS], fin;
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort;
  __shared__ float s_row[DT_RS][DT_HC][DT_M];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const unsigned g0 = blockIdx.x * sc.items / sc.G, g1 = (blockIdx.x + 1) * sc.items / sc.G;
  const int nt = (int)(g1 - g0);
  // the range's first column and row tile
  int cb = sc.c0, re = sc.c1;
  while (re - cb > 1) {
    const int m = (cb + re) >> 1;
    if (dt_start(m, sc) <= g0) cb = m;
    else re = m;
  }
  const int rb = (int)(g0 - dt_start(cb, sc));
  uint8_t *ring = dsm, *sb = dsm + (size_t)DT_NS * DT_AB;
  volatile int *abort = &s_abort;
  if (warp == 0) tc_alloc(&s_tmem, 512);
  if (tid == 0) {
    for (int k = 0; k < DT_NS; ++k) {
      mbar_init(&afull[k], 1);
      mbar_init(&aempty[k], 1);
    }
    for (int k = 0; k < 2; ++k) {
      mbar_init(&bfull[k], 1);
      mbar_init(&bempty[k], 1);
      mbar_init(&accfull[k], 1);
      mbar_init(&accfree[k], DT_EW);  // one arrival per epilogue warp
    }
    for (int k = 0; k < DT_RS; ++k) {
      mbar_init(&rowfull[k], DT_EW);
      mbar_init(&rowfree[k], 1);
    }
    mbar_init(&fin, 1);
    s_abort = 0;
    fence_mbar_init();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s_tmem;

  if (warp == DT_EW) {
    // ------------------------------------------------ bulk copies
    if (lane == 0) {
      int c = cb, r = rb, nc = 0, g = 0;  // nc: column tiles begun
      bool ok = true;
      for (; g < nt; ++g) {
        if (g == 0 || r == 0) {
          const int sl = nc & 1;
          if (nc >= 2 && !dt_wait(&bempty[sl], (uint32_t)(((nc >> 1) - 1) & 1), abort)) {
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&bfull[sl], DT_BB);
          bulk_g2s(sb + (size_t)sl * DT_BB, bimg + (size_t)c * DT_BB, DT_BB, &bfull[sl]);
          ++nc;
        }
        const int st = g % DT_NS;
        if (g >= DT_NS && !dt_wait(&aempty[st], (uint32_t)(((g / DT_NS) - 1) & 1), abort)) {
          ok = false;
          break;
        }
        mbar_arrive_expect_tx(&afull[st], DT_AB);
        bulk_g2s(ring + (size_t)st * DT_AB, aimg + (size_t)r * DT_AB, DT_AB, &afull[st]);
        if (++r == 2 * c + 2) {
          r = 0;
          ++c;
        }
      }
      if (!ok) vds_flag(err, VDS_ETIMEOUT);
      // the copies still in flight land before the CTA may exit
      for (int k = g > DT_NS ? g - DT_NS : 0; k < g; ++k)
        mbar_wait_bounded(&afull[k % DT_NS], (uint32_t)((k / DT_NS) & 1), VDS_WAIT_LIMIT_NS);
      for (int k = nc > 2 ? nc - 2 : 0; k < nc; ++k)
        mbar_wait_bounded(&bfull[k & 1], (uint32_t)((k >> 1) & 1), VDS_WAIT_LIMIT_NS);
    }
  } else if (warp == DT_EW + 1) {
    // ------------------------------------------------ MMA issue
    if (lane == 0) {
      const uint32_t idesc = tc_idesc(TC_FMT_TF32, DT_M, DT_N);
      const uint32_t ab = smem_u32(ring), bb = smem_u32(sb);
      int c = cb, r = rb, nc = 0;
      bool ok = true;
      for (int g = 0; g < nt && ok; ++g) {
        if (g == 0 || r == 0) {
          ok = dt_wait(&bfull[nc & 1], (uint32_t)((nc >> 1) & 1), abort);
          if (!ok) break;
          ++nc;
        }
        const int st = g % DT_NS, b = g & 1, sl = (nc - 1) & 1;
        if (!dt_wait(&afull[st], (uint32_t)((g / DT_NS) & 1), abort)) {
          ok = false;
          break;
        }
        // the epilogue has read this accumulator's previous tile
        if (g >= 2 && !dt_wait(&accfree[b], (uint32_t)(((g >> 1) - 1) & 1), abort)) {
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t d = tmem + (uint32_t)(b * DT_N);
        const uint32_t a0 = ab + (uint32_t)(st * DT_AB), b0 = bb + (uint32_t)(sl * DT_BB);
#pragma unroll
        for (int kk = 0; kk < 2; ++kk) {
          const uint32_t o = (uint32_t)(kk * 256);  // 8 TF32 of K = two core matrices
          tc_mma_tf32(d, tc_sdesc(a0 + o), tc_sdesc(b0 + o), idesc, kk > 0 ? 1 : 0);   // hi . hi
          tc_mma_tf32(d, tc_sdesc(a0 + o), tc_sdesc(b0 + 512 + o), idesc, 1);         // hi . lo
          tc_mma_tf32(d, tc_sdesc(a0 + 512 + o), tc_sdesc(b0 + o), idesc, 1);         // lo . hi
        }
        tc_commit(&aempty[st]);
        tc_commit(&accfull[b]);
        if (++r == 2 * c + 2) {
          tc_commit(&bempty[sl]);
          r = 0;
          ++c;
        }
      }
      if (!ok) vds_flag(err, VDS_ETIMEOUT);
    }
  } else if (warp == DT_EW + 2) {
    // ------------------------------------------------ row sums
    int c = cb, r = rb, nr = 0;  // nr: tiles off the diagonal so far
    bool ok = true;
    for (int g = 0; g < nt && ok; ++g) {
      if (r < 2 * c) {
        const int k = nr % DT_RS;
        ok = __all_sync(0xffffffffu, dt_wait(&rowfull[k], (uint32_t)((nr / DT_RS) & 1), abort));
        if (!ok) break;
        float *dst = rowp + dt_row(c, sc) + (size_t)r * DT_M;
#pragma unroll
        for (int x = 0; x < DT_M / 32; ++x) {
          const int rl = x * 32 + lane;
          dst[rl] = (s_row[k][0][rl] + s_row[k][1][rl]) + (s_row[k][2][rl] + s_row[k][3][rl]);
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowfree[k]);
        ++nr;
      }
      if (++r == 2 * c + 2) {
        r = 0;
        ++c;
      }
    }
    if (!ok && lane == 0) vds_flag(err, VDS_ETIMEOUT);
  } else {
    // ------------------------------------------------ epilogue warps
    const int q = warp & 3, hc = warp >> 2;
    const int rl = q * 32 + lane;
    auto norm = [&](int r) {  // of this lane's row of row tile r; past N no kernel value is left
      const int row = r * DT_M + rl;
      return row < N ? rec[(size_t)row * DP + nslot] : 1e30f;
    };
    unsigned long long col[DT_CW / 2];
#pragma unroll
    for (int k = 0; k < DT_CW / 2; ++k) col[k] = 0ull;
    float t0 = 0.f, c0 = 0.f, t1 = 0.f, c1 = 0.f;  // columns lane and lane + 32, compensated
    int c = cb, r = rb, nr = 0, nf = 0;
    bool ok = true;
    float nI = norm(rb);
    for (int g = 0; g < nt && ok; ++g) {
      const int b = g & 1;
      int cn = c, rn = r + 1;
      if (rn == 2 * c + 2) {
        rn = 0;
        ++cn;
      }
      const float nnext = g + 1 < nt ? norm(rn) : 0.f;
      ok = __all_sync(0xffffffffu, dt_wait(&accfull[b], (uint32_t)((g >> 1) & 1), abort));
      if (!ok) break;
      tc_fence_after();
      const uint32_t ta = tmem + ((uint32_t)(q * 32) << 16) + (uint32_t)(b * DT_N + hc * DT_CW);
      unsigned long long rs = 0ull;
      uint32_t v[2][8];  // the next eight columns are on their way while these are used
      tc_ld8_start(ta, v[0]);
#pragma unroll
      for (int h = 0; h < DT_CW / 8; ++h) {
        uint32_t(&w)[8] = v[h & 1];
        tc_wait_ld(w);
        if (h + 1 < DT_CW / 8) tc_ld8_start(ta + (uint32_t)(h * 8 + 8), v[(h + 1) & 1]);
#pragma unroll
        for (int j = 0; j < 8; j += 2) {
          const unsigned long long e = f2_pack(ex2_approx(__uint_as_float(w[j]) - nI),
                                               ex2_approx(__uint_as_float(w[j + 1]) - nI));
          rs = f2_add(rs, e);
          col[h * 4 + j / 2] = f2_add(col[h * 4 + j / 2], e);
        }
      }
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&accfree[b]);
      if (r < 2 * c) {
        const int k = nr % DT_RS;
        if (nr >= DT_RS)
          ok = __all_sync(0xffffffffu, dt_wait(&rowfree[k], (uint32_t)(((nr / DT_RS) - 1) & 1), abort));
        if (!ok) break;
        float x, y;
        f2_unpack(rs, x, y);
        s_row[k][hc][rl] = x + y;
        __syncwarp();
        if (lane == 0) mbar_arrive(&rowfull[k]);
        ++nr;
      }
      const bool end = cn != c || g + 1 == nt;  // the column tile, or the range, ends here
      if (++nf == DT_FOLD || end) {
        nf = 0;
        float x[32];
#pragma unroll
        for (int k = 0; k < 16; ++k) f2_unpack(col[k], x[2 * k], x[2 * k + 1]);
        kahan(lane_sums(x, lane), t0, c0);
#pragma unroll
        for (int k = 0; k < 16; ++k) f2_unpack(col[16 + k], x[2 * k], x[2 * k + 1]);
        kahan(lane_sums(x, lane), t1, c1);
#pragma unroll
        for (int k = 0; k < DT_CW / 2; ++k) col[k] = 0ull;
      }
      if (end) {
        const int seg = (int)blockIdx.x - dt_cta_of(dt_start(c, sc), sc);
        float2 *dst = colp + (((size_t)(c - sc.c0) * sc.maxseg + seg) * 4 + q) * DT_N + hc * DT_CW + lane;
        dst[0] = make_float2(t0, -c0);
        dst[32] = make_float2(t1, -c1);
        t0 = c0 = t1 = c1 = 0.f;
      }
      nI = nnext;
      c = cn;
      r = rn;
    }
    if (!ok && lane == 0) vds_flag(err, VDS_ETIMEOUT);
  }
  // every role has left its loop; the MMAs issued are complete before the
  // tensor memory is released
  tc_fence_before();
  __syncthreads();
  if (warp == DT_EW + 1 && lane == 0) {
    tc_commit(&fin);
    mbar_wait_bounded(&fin, 0, VDS_WAIT_LIMIT_NS);
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  if (warp == 0) tc_dealloc(tmem, 512);
}

}  // namespace

// ------------------------------------------------------------------ host

namespace {

template <int D>
int dens_tc_impl(vds_ctx *c, int N, float *rho_out) {
  constexpr int DP = Rec<D>::DP;
  const int Npad = (N + DT_N - 1) / DT_N * DT_N;
  const int ntc = Npad / DT_N;
  const size_t img = (size_t)Npad * DT_RB;
  // a launch's column tiles from c0 on: as many as `limit` bytes of row sums hold
  size_t limit = DT_ROW_BYTES;
  auto sched = [&](int c0) {
    DtSched sc;
    sc.c0 = c0;
    sc.c1 = c0 + 1;
    while (sc.c1 < ntc && dt_row(sc.c1 + 1, sc) * sizeof(float) <= limit) ++sc.c1;
    sc.items = dt_start(sc.c1, sc);
    sc.G = sc.items < (unsigned)c->num_sms ? (int)sc.items : c->num_sms;
    sc.maxseg = 1;
    for (int t = sc.c0; t < sc.c1; ++t) {
      const int n = dt_cta_of(dt_start(t + 1, sc) - 1, sc) - dt_cta_of(dt_start(t, sc), sc) + 1;
      if (n > sc.maxseg) sc.maxseg = n;
    }
    return sc;
  };
  size_t rowb, colb;
  for (;;) {
    rowb = colb = 0;
    for (int c0 = 0; c0 < ntc;) {
      const DtSched sc = sched(c0);
      const size_t r = dt_row(sc.c1, sc) * sizeof(float);
      const size_t l = (size_t)(sc.c1 - sc.c0) * sc.maxseg * 4 * DT_N * sizeof(float2);
      if (r > rowb) rowb = r;
      if (l > colb) colb = l;
      c0 = sc.c1;
    }
    const int st = vds_ensure(c, c->dtbuf, 2 * img + colb + (size_t)N * sizeof(float2) + rowb);
    if (st == VDS_OK) break;
    if (st != VDS_ENOMEM || limit <= DT_ROW_LEAST) return st;
    (void)cudaGetLastError();
    limit = (rowb < limit ? rowb : limit) / 4;  // more launches of fewer column tiles
  }
  uint8_t *aimg = (uint8_t *)c->dtbuf.ptr, *bimg = aimg + img;
  float2 *colp = (float2 *)(bimg + img), *run = (float2 *)((uint8_t *)colp + colb);
  float *rowp = (float *)(run + N);
  const float *rec = (const float *)c->rec.ptr;
  const long ne = (long)Npad * DT_K;
  k_dt_prep<D><<<(unsigned)((ne + 255) / 256), 256, 0, c->stream>>>(rec, N, Npad, aimg, bimg);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  static bool attr[VDS_MAX_DEVICES] = {};
  if (c->device >= VDS_MAX_DEVICES || !attr[c->device]) {
    VDS_CUDA_TRY(cudaFuncSetAttribute(k_dens_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)DT_SMEM));
    if (c->device < VDS_MAX_DEVICES) attr[c->device] = true;
  }
  for (int c0 = 0; c0 < ntc;) {
    const DtSched sc = sched(c0);
    k_dens_tc<<<sc.G, DT_NT, DT_SMEM, c->stream>>>(aimg, bimg, rec, DP, D + 1, N, sc, rowp, colp, c->err);
    VDS_CUDA_TRY(cudaGetLastError());
    k_dt_finish<<<(unsigned)((N + 31) / 32), 256, 0, c->stream>>>(sc, rowp, colp, N, DP, D, c0 == 0, sc.c1 == ntc, run,
                                                                 (float *)c->rec.ptr, rho_out, c->err);
    VDS_CUDA_TRY(cudaGetLastError());
    c->launches += 2;
    c0 = sc.c1;
  }
  return VDS_OK;
}

}  // namespace

int pass_density_tc(vds_ctx *c, const KParams &kp, float *rho_out) {
  if (kp.N < 1) return VDS_EARG;
  switch (kp.D) {
    case 6: return dens_tc_impl<6>(c, kp.N, rho_out);
    case 9: return dens_tc_impl<9>(c, kp.N, rho_out);
    default: return VDS_EARG;  // no norm slot in the records, or D + 1 > 16
  }
}

int pass_density_tc_images(vds_ctx *c, int N, int D, const uint8_t **aimg, const uint8_t **bimg) {
  if (N < 1 || (D != 6 && D != 9)) return VDS_EARG;
  const int Npad = (N + DT_N - 1) / DT_N * DT_N;
  const size_t img = (size_t)Npad * DT_RB;
  VDS_TRY(vds_ensure(c, c->dtbuf, 2 * img));
  uint8_t *a = (uint8_t *)c->dtbuf.ptr, *b = a + img;
  const long ne = (long)Npad * DT_K;
  if (D == 6)
    k_dt_prep<6><<<(unsigned)((ne + 255) / 256), 256, 0, c->stream>>>((const float *)c->rec.ptr, N, Npad, a, b);
  else
    k_dt_prep<9><<<(unsigned)((ne + 255) / 256), 256, 0, c->stream>>>((const float *)c->rec.ptr, N, Npad, a, b);
  VDS_CUDA_TRY(cudaGetLastError());
  ++c->launches;
  *aimg = a;
  *bimg = b;
  return VDS_OK;
}
