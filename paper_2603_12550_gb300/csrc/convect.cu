// convect.cu -- the convection term of the micro-macro model: transport of a
// field held at the nodes of a structured macroscopic grid by the flow, the
// u . grad_x q term of Eq. model_DymRepPar (and u . grad_x p of Eq.
// model_DymReduced for reduced coordinates), which the homogeneous-flow
// experiments of Sec. 3 drop and a grid of ensembles needs (include/
// vds_batch.h, vds_convect).
//
// One first-order upwind step per call:
//   Q_out[g] = Q[g] - dt sum_b ( max(u_b,0) (Q[g] - Q[g - e_b])
//                               + min(u_b,0) (Q[g + e_b] - Q[g]) ) / dx_b
// in FP32 (the field is FP32; each output is a handful of operations on
// values of the same magnitude).  The field is M values per node, node-major.
//
// HBM sees one read and one write of the field, the bound (59 us for 512 nodes
// x 98304 values); in between, every value is read up to four times, once for
// its own node and once for each neighbour downwind.  k_convect_tile takes a
// block of up to 64 neighbouring nodes and 128 values per CTA (32 KB), so that
// most of those reads hit in L1, 16 bytes per lane: 95 -> 72 us.
// k_convect, one node per CTA with the neighbours' values from L2 (whose
// bandwidth bound it: four reads of the field in 95 us), is left for values per
// node that are not a multiple of four and for unaligned arrays: the node is
// the fastest grid index, so the CTAs resident at one time cover one or two
// value ranges of every node, which are still in L2 when the neighbours need
// them.
#include "vds_internal.cuh"

#include "vds_batch.h"

namespace {

constexpr int CV_NT = 256;
constexpr int CV_PER = 8;  // values per thread

__global__ void __launch_bounds__(CV_NT)
    k_convect(const float *__restrict__ q, float *__restrict__ out, int nx, int ny, int nz, long M,
              const float *__restrict__ u, float cx, float cy, float cz, int bc) {
  const int g = blockIdx.x;
  const int G = nx * ny * nz;
  if (g >= G) return;
  const int ix = g % nx, iy = (g / nx) % ny, iz = g / (nx * ny);
  // neighbour nodes below and above along each axis (periodic or clamped)
  auto nb = [&](int i, int n, int d) -> int {
    int j = i + d;
    if (j < 0) j = bc == 0 ? n - 1 : 0;
    if (j >= n) j = bc == 0 ? 0 : n - 1;
    return j;
  };
  const int gxm = nb(ix, nx, -1) + nx * (iy + ny * iz), gxp = nb(ix, nx, 1) + nx * (iy + ny * iz);
  const int gym = ix + nx * (nb(iy, ny, -1) + ny * iz), gyp = ix + nx * (nb(iy, ny, 1) + ny * iz);
  const int gzm = ix + nx * (iy + ny * nb(iz, nz, -1)), gzp = ix + nx * (iy + ny * nb(iz, nz, 1));
  // Courant factors dt u_b / dx_b; the upwind neighbour of each axis (the
  // sign of u_b is the same for the whole CTA, so each value reads the node
  // itself and at most three neighbours)
  const float ux = nx > 1 ? u[(size_t)g * 3] * cx : 0.f;
  const float uy = ny > 1 ? u[(size_t)g * 3 + 1] * cy : 0.f;
  const float uz = nz > 1 ? u[(size_t)g * 3 + 2] * cz : 0.f;
  const float *qx = ux > 0.f ? q + (size_t)gxm * M : ux < 0.f ? q + (size_t)gxp * M : nullptr;
  const float *qy = uy > 0.f ? q + (size_t)gym * M : uy < 0.f ? q + (size_t)gyp * M : nullptr;
  const float *qz = uz > 0.f ? q + (size_t)gzm * M : uz < 0.f ? q + (size_t)gzp * M : nullptr;
  const float *qg = q + (size_t)g * M;
  const long chunk = (long)blockIdx.y + (long)gridDim.y * blockIdx.z;
  const long m0 = chunk * CV_NT * CV_PER + threadIdx.x;
  if (m0 >= M) return;
  float *og = out + (size_t)g * M;
  // u_b > 0: u_b (Q[g] - Q[g - e_b]); u_b < 0: u_b (Q[g + e_b] - Q[g])
  auto upd = [](float d, float ub, float c, float v) { return d + (ub > 0.f ? ub * (c - v) : ub * (v - c)); };
  if (m0 + (long)(CV_PER - 1) * CV_NT < M) {
    // a full chunk: every load is issued before the arithmetic (memory-level
    // parallelism is what bounds this kernel)
    float c[CV_PER], vx[CV_PER], vy[CV_PER], vz[CV_PER];
#pragma unroll
    for (int k = 0; k < CV_PER; ++k) {
      const long m = m0 + (long)k * CV_NT;
      c[k] = qg[m];
      vx[k] = qx ? qx[m] : 0.f;
      vy[k] = qy ? qy[m] : 0.f;
      vz[k] = qz ? qz[m] : 0.f;
    }
#pragma unroll
    for (int k = 0; k < CV_PER; ++k) {
      float d = 0.f;
      if (qx) d = upd(d, ux, c[k], vx[k]);
      if (qy) d = upd(d, uy, c[k], vy[k]);
      if (qz) d = upd(d, uz, c[k], vz[k]);
      og[m0 + (long)k * CV_NT] = c[k] - d;
    }
    return;
  }
  for (int k = 0; k < CV_PER; ++k) {
    const long m = m0 + (long)k * CV_NT;
    if (m >= M) break;
    const float ck = qg[m];
    float d = 0.f;
    if (qx) d = upd(d, ux, ck, qx[m]);
    if (qy) d = upd(d, uy, ck, qy[m]);
    if (qz) d = upd(d, uz, ck, qz[m]);
    og[m] = ck - d;
  }
}

constexpr int CT_NODES = 64, CT_NT = 256, CT_COLS = 32;  // nodes, threads, float4 columns per CTA

// A CTA's block of nodes (at most CT_NODES; the last ones of an axis may be
// cut) and of columns.
struct CvTile {
  int x, y, z;     // nodes per axis
  int bx, by, bz;  // blocks per axis
  int lg, cols;    // log2 of the nodes, rounded up; groups of CT_COLS columns
};

__global__ void __launch_bounds__(CT_NT)
    k_convect_tile(const float4 *__restrict__ q, float4 *__restrict__ out, int nx, int ny, int nz, long M4, CvTile T,
                   const float *__restrict__ u, float cx, float cy, float cz, int bc) {
  __shared__ int s_g[CT_NODES], s_nb[3][CT_NODES];  // node, upwind neighbours; -1: none
  __shared__ float s_u[3][CT_NODES];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nodes = 1 << T.lg;
  if (tid < nodes) {
    const int b = blockIdx.x;
    const int ix = (b % T.bx) * T.x + tid % T.x;
    const int iy = ((b / T.bx) % T.by) * T.y + (tid / T.x) % T.y;
    const int iz = (b / (T.bx * T.by)) * T.z + tid / (T.x * T.y);
    int g = -1;
    if (tid < T.x * T.y * T.z && ix < nx && iy < ny && iz < nz) {
      g = ix + nx * (iy + ny * iz);
      // the neighbour that the flow comes from along an axis (periodic or clamped)
      auto up = [&](float v, int i, int n, int stride) -> int {
        if (!(v > 0.f) && !(v < 0.f)) return -1;
        int j = v > 0.f ? i - 1 : i + 1;
        if (j < 0) j = bc == 0 ? n - 1 : 0;
        if (j >= n) j = bc == 0 ? 0 : n - 1;
        return g + (j - i) * stride;
      };
      const float ux = nx > 1 ? u[(size_t)g * 3] * cx : 0.f, uy = ny > 1 ? u[(size_t)g * 3 + 1] * cy : 0.f,
                  uz = nz > 1 ? u[(size_t)g * 3 + 2] * cz : 0.f;
      s_u[0][tid] = ux;
      s_u[1][tid] = uy;
      s_u[2][tid] = uz;
      s_nb[0][tid] = up(ux, ix, nx, 1);
      s_nb[1][tid] = up(uy, iy, ny, nx);
      s_nb[2][tid] = up(uz, iz, nz, nx * ny);
    }
    s_g[tid] = g;
  }
  __syncthreads();
  const long m0 = ((long)blockIdx.y + (long)gridDim.y * blockIdx.z) * T.cols * CT_COLS + lane;
  auto upd = [](float d, float ub, float c, float v) { return d + (ub > 0.f ? ub * (c - v) : ub * (v - c)); };
  for (int x = warp; x < nodes * T.cols; x += CT_NT / 32) {
    const int n = x & (nodes - 1), g = s_g[n];
    const long m = m0 + (long)(x >> T.lg) * CT_COLS;
    if (g < 0 || m >= M4) continue;
    const float4 c = q[(size_t)g * M4 + m];
    float4 v[3], d = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (s_nb[a][n] >= 0) v[a] = q[(size_t)s_nb[a][n] * M4 + m];
#pragma unroll
    for (int a = 0; a < 3; ++a)
      if (s_nb[a][n] >= 0) {
        const float ub = s_u[a][n];
        d.x = upd(d.x, ub, c.x, v[a].x);
        d.y = upd(d.y, ub, c.y, v[a].y);
        d.z = upd(d.z, ub, c.z, v[a].z);
        d.w = upd(d.w, ub, c.w, v[a].w);
      }
    __stcs(out + (size_t)g * M4 + m, make_float4(c.x - d.x, c.y - d.y, c.z - d.z, c.w - d.w));
  }
}

}  // namespace

extern "C" int vds_convect(vds_ctx *c, const float *q_in, float *q_out, int nx, int ny, int nz, long M,
                           const float *u, const double *dx, double dt, int bc) {
  if (!c || !q_in || !q_out || !u || !dx || nx < 1 || ny < 1 || nz < 1 || M < 1) return VDS_EARG;
  if (!(dt > 0.0) || (bc != 0 && bc != 1)) return VDS_EARG;
  for (int b = 0; b < 3; ++b)
    if (!(dx[b] > 0.0)) return VDS_EARG;
  const long long G = (long long)nx * ny * nz;
  if (G > (1ll << 30)) return VDS_EARG;
  const size_t bytes = (size_t)G * (size_t)M * sizeof(float);
  const char *a0 = (const char *)q_in, *b0 = (const char *)q_out;
  if (a0 < b0 + bytes && b0 < a0 + bytes) return VDS_EARG;  // in place is not supported
  int prev = -1;
  if (cudaGetDevice(&prev) != cudaSuccess) return VDS_ECUDA;
  if (prev != c->device && cudaSetDevice(c->device) != cudaSuccess) return VDS_ECUDA;
  const bool wide = M % 4 == 0 && ((size_t)q_in | (size_t)q_out) % 16 == 0;
  CvTile T = {1, 1, 1, 1, 1, 1, 0, 1};
  const int per = wide ? 4 * CT_COLS : CV_NT * CV_PER;
  long chunks = (M + per - 1) / per;
  if (wide) {
    // block of nodes: double the shortest axis that has nodes left; small
    // fields take smaller blocks (a node per warp at least) to use every SM
    int most = CT_NODES, len[3] = {1, 1, 1};
    const int n[3] = {nx, ny, nz};
    while (most > CT_NT / 32 && G / most * chunks < 2 * c->num_sms) most /= 2;
    for (;;) {
      int best = -1;
      for (int a = 0; a < 3; ++a)
        if (len[a] < n[a] && (best < 0 || len[a] < len[best])) best = a;
      if (best < 0 || 2 * len[0] * len[1] * len[2] > most) break;
      len[best] *= 2;
    }
    // blocks of an axis equally long: 9 nodes are 5 and 4, not 8 and 1 (9 x 9
    // nodes x 98304 values 16.7 -> 12.7 us)
    int blk[3];
    for (int a = 0; a < 3; ++a) {
      blk[a] = (n[a] + len[a] - 1) / len[a];
      len[a] = (n[a] + blk[a] - 1) / blk[a];
    }
    T = CvTile{len[0], len[1], len[2], blk[0], blk[1], blk[2], 0, 1};
    while (1 << T.lg < T.x * T.y * T.z) ++T.lg;
    // a block of few nodes takes more columns, so that a CTA still has CT_NODES
    // rows of 32 columns to move, while eight CTAs per SM remain (values per
    // node 8 Mi; k_convect / 32 columns always / this: one node 17 / 107 / 10.5
    // us, 12 in a row 173 / 308 / 136, 5 x 5 360 / 710 / 315)
    const long blocks = (long)blk[0] * blk[1] * blk[2];
    while ((T.cols << T.lg) < CT_NODES && blocks * chunks >= 16L * c->num_sms) {
      T.cols *= 2;
      chunks = (chunks + 1) / 2;
    }
  }
  const unsigned gy = (unsigned)(chunks < 65535 ? chunks : 65535);
  const long gz = (chunks + gy - 1) / gy;
  int st = VDS_OK;
  if (gz > 65535) {
    st = VDS_EARG;
  } else {
    const float cx = (float)(dt / dx[0]), cy = (float)(dt / dx[1]), cz = (float)(dt / dx[2]);
    if (wide) {
      k_convect_tile<<<dim3((unsigned)T.bx * T.by * T.bz, gy, (unsigned)gz), CT_NT, 0, c->stream>>>(
          (const float4 *)q_in, (float4 *)q_out, nx, ny, nz, M / 4, T, u, cx, cy, cz, bc);
    } else {
      k_convect<<<dim3((unsigned)G, gy, (unsigned)gz), CV_NT, 0, c->stream>>>(q_in, q_out, nx, ny, nz, M, u, cx, cy, cz,
                                                                             bc);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) {
      vds_last_cuda_error(e);
      st = VDS_ECUDA;
    } else {
      ++c->launches;
    }
  }
  if (prev >= 0 && prev != c->device) cudaSetDevice(prev);
  return st;
}
